// Launchers of the fused x inverse / cell / x forward kernel (mm_plane_step.cuh).
#include "mm_plane_launch.cuh"
#include "mm_plane_step.cuh"

namespace mm {
namespace {

template <bool STAGE>
int launch_px_cell(mm_ctx* ctx, const float* m_in, float* H, const RkStage<float>& g) {
    const PlanePlan& p = ctx->plane;
    const float2* tw = (const float2*)p.tw;
    const float scale = (float)(1.0 / ((double)p.L * p.P * ctx->Pz));
    Params<float> par = make_params<float>(ctx);
    const bool folded = !par.Ms_cell && !par.A_cell && par.Ms != 0.f;
    if (folded) {
        const float inv = 1.f / par.Ms;
        par.cx = par.A * par.cx * inv;
        par.cy = par.A * par.cy * inv;
        par.cz = par.A * par.cz * inv;
        par.A = 1.f;
    }
    const int nrows = ctx->ny * ctx->nz;
    // four rows a block read and write whole 32-byte sectors of the planes;
    // fewer where that leaves SMs idle
    const int lgB = nrows >= 4 * 152 ? 2 : nrows >= 2 * 152 ? 1 : 0;
    int rc = MM_OK;
    KernelTimer kt(ctx, STAGE ? MM_K_STAGE : MM_K_REDUCE);
    if (!with_length(p.L, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value;
            if constexpr (L1 * L2 <= 512) {
                const int lines = 3 << lgB, width = lines * (L1 > L2 ? L1 : L2);
                const int nt = width > 256 ? (width + 31) / 32 * 32 : 256;
                const size_t smem = (size_t)lines * (plane_pitch(L1, L2) + 4) * sizeof(float2);
                auto fn = k_px_cell<float, L1, L2, STAGE>;
                if ((rc = smem_opt_in(ctx, (const void*)fn, smem))) return;
                dep(fn, (unsigned)((nrows + (1 << lgB) - 1) >> lgB), nt, smem, ctx->stream)(
                    (float2*)p.buf, p.R, par, folded, lgB, scale, tw + p.off_x4, tw + p.off_p, m_in, H, g, ctx->ctl);
            }
        }))
        rc = fail(ctx, MM_ERR_INVALID_ARG, "x length %d", p.L);
    if (rc) return rc;
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

}  // namespace

// Small meshes: four kernels of a stage cost more in gaps, ramps and tails than
// the fused kernel's lower occupancy in the cell part.  One RK4 stage, four
// kernels -> two (uniform Ms / Ms per cell): 100x25x1 13.3 -> 9.2 / 16.0 -> 9.4
// us, 64x64x4 14.0 -> 9.4 / 16.4 -> 10.0, 256x256x1 (66 k cells) 18.2 -> 14.9 /
// 22.5 -> 15.7; 300x300x2 (180 k) 27.3 -> 27.8 / 31.8 -> 29.4, 256x256x4 (262 k)
// 25.7 -> 29.4 / 32.2 -> 32.0.  The effective field alone: 11.5 -> 10.2, 12.0 ->
// 9.9, 16.5 -> 15.0; 25.2 -> 26.3, 23.9 -> 27.6.
constexpr long kFusedCells = 120000;

bool plane_fused(const mm_ctx* ctx) {
    return ctx->prec == MM_F32 && ctx->plane.on && ctx->fft_mode == 0 && ctx->N <= kFusedCells;
}

int plane_stage(mm_ctx* ctx, int method, int s, const void* m_in, const void* m0, void* m_out, void* hd, bool forward) {
    RkStage<float> g = {};
    g.s = s;
    g.last = s == rk_stages(method) - 1;
    g.adaptive = method == MM_RKF45;
    g.forward = forward;
    for (int j = 0; j < s; ++j) {
        g.a[j] = (float)(g.last ? rk_b(method, j) : rk_a(method, s + 1, j));
        g.e[j] = (float)(g.last ? rk_e(method, j) : 0.0);
    }
    g.cs = (float)(g.last ? rk_b(method, s) : rk_a(method, s + 1, s));
    g.es = (float)(g.last ? rk_e(method, s) : 0.0);
    g.m0 = (const float*)m0;
    g.out = (float*)m_out;
    g.hd = (float*)hd;
    g.kb = slopes<float>(ctx);
    return launch_px_cell<true>(ctx, (const float*)m_in, nullptr, g);
}

int plane_field(mm_ctx* ctx, const void* m, void* H) {
    int rc = plane_xfwd(ctx, m);
    if (rc || (rc = plane_yzy(ctx))) return rc;
    return launch_px_cell<false>(ctx, (const float*)m, (float*)H, RkStage<float>{});
}

}  // namespace mm
