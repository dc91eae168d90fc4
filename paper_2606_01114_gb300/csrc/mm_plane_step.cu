// Launchers of the fused x inverse / cell / x forward kernel (mm_plane_step.cuh).
#include "mm_plane_launch.cuh"
#include "mm_plane_step.cuh"

namespace mm {
namespace {

// four rows a block read and write whole 32-byte sectors of the planes; fewer
// where that leaves SMs idle
struct CellGrid {
    int lgB;
    long blocks;
};
CellGrid cell_grid(const mm_ctx* ctx) {
    const long nrows = (long)ctx->ny * ctx->nz;
    const int lgB = nrows >= 4 * kSMs ? 2 : nrows >= 2 * kSMs ? 1 : 0;
    return {lgB, (nrows + (1 << lgB) - 1) >> lgB};
}
constexpr int cell_threads(int L1, int L2, CellGrid c) {
    const int width = (3 << c.lgB) * (L1 > L2 ? L1 : L2);
    return width > 256 ? (width + 31) / 32 * 32 : 256;
}
constexpr size_t cell_smem(int L1, int L2, CellGrid c) {
    return (size_t)(3 << c.lgB) * (plane_pitch(L1, L2) + 4) * sizeof(float2);
}

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
    const CellGrid c = cell_grid(ctx);
    int rc = MM_OK;
    KernelTimer kt(ctx, STAGE ? MM_K_STAGE : MM_K_REDUCE);
    if (!with_length(p.L, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value;
            if constexpr (L1 * L2 <= 512) {
                const size_t smem = cell_smem(L1, L2, c);
                auto fn = k_px_cell<float, L1, L2, STAGE, STAGE ? 512 : 384>;
                // the longest rows lose 3 % to the bound while each block has an SM to itself
                if constexpr (STAGE && L1 * L2 == 512) {
                    if (c.blocks <= kSMs) fn = k_px_cell<float, L1, L2, STAGE, 384>;
                }
                if ((rc = smem_opt_in(ctx, (const void*)fn, smem))) return;
                dep(fn, (unsigned)c.blocks, cell_threads(L1, L2, c), smem, ctx->stream)(
                    (float2*)p.buf, p.R, par, folded, c.lgB, scale, tw + p.off_x4, tw + p.off_p, m_in, H, g, ctx->ctl);
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
// kernels -> two: 100x25x1 13.0 -> 9.2 us, 64x64x4 13.1 -> 8.4, 256x256x1 (66 k
// cells) 17.4 -> 13.5, 300x300x1 18.3 -> 15.4, 512x175x1 18.9 -> 17.8, 350x350x1
// (123 k) 20.1 -> 19.4, 200x200x4 (160 k) 22.6 -> 25.0; with Ms per cell 13.2 ->
// 8.7, 17.7 -> 13.7, 18.7 -> 15.6, 19.5 -> 18.1, 20.7 -> 19.7, 23.9 -> 25.8.
// An SM holds two blocks; a second wave of them pays on short rows only:
// 64x351x4 (351 blocks) 19.3 -> 19.0, but 80x371x4 19.7 -> 21.7.
// The effective field alone has one kernel fewer to save: 64x351x4 18.8 -> 17.0,
// 96x309x4 19.0 -> 18.4, 160x140x4 (90 k) 18.2 -> 17.1, 128x468x1 14.7 -> 14.4, but
// 256x351x1 (90 k) 16.7 -> 18.1, 160x185x4 (118 k) 20.3 -> 21.1, and no mesh of x
// length 320 and more gains (300x100x1 16.1 -> 16.4, 512x29x1 15.1 -> 16.9).
constexpr long kFusedCells = 120000;

bool plane_fused(const mm_ctx* ctx, bool field) {
    const PlanePlan& p = ctx->plane;
    if (ctx->prec != MM_F32 || !p.on || ctx->fft_mode != 0 || ctx->N > kFusedCells) return false;
    if (field) return p.L <= 96 || (p.L <= 256 && ctx->N <= (p.L & (p.L - 1) ? 100000 : 85000));
    return p.L <= 64 || cell_grid(ctx).blocks <= 2 * kSMs;
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
