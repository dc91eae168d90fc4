// Plane-layout demag passes in FP32: the x passes and the sequence (the plane
// and line kernels: mm_plane_f32y.cu).
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f32(mm_ctx* ctx);

int plane_line_len(int P) { return plane_line(P); }

void four_step_table(mm_ctx* ctx, int len, bool z, std::vector<double>& out) {
    const std::vector<double>& c = unit_circle(ctx, len);
    auto put = [&](int L1, int L2) {
        for (int turn = 0; turn < 2; ++turn)
            for (int q = 0; q < len; ++q) {
                const int t = turn ? q / L1 : q % L2, k1 = turn ? q % L1 : q / L2;   // t k1 < len
                out.push_back(c[2 * (size_t)(t * k1)]);
                out.push_back(c[2 * (size_t)(t * k1) + 1]);
            }
    };
    if (z) with_z_length(len, [&](auto A, auto B) { put(decltype(A)::value, decltype(B)::value); });
    else with_length(len, [&](auto A, auto B) { put(decltype(A)::value, decltype(B)::value); });
}

int plane_xfwd_f32(mm_ctx* ctx, const float* m, const float* Ms, float ms) {
    return launch_px_fwd<float>(ctx, m, Ms, ms, (long)ctx->nz * ctx->ny, (float2*)ctx->plane.buf,
                                       3L * ctx->nz * ctx->ny, (const float2*)ctx->plane.tw);
}

int plane_apply_f32(mm_ctx* ctx, const float* m, const float* Ms, float ms, float* H) {
    const PlanePlan& p = ctx->plane;
    int rc = plane_xfwd_f32(ctx, m, Ms, ms);
    if (rc || (rc = plane_yzy_f32(ctx))) return rc;
    const float scale = (float)(1.0 / ((double)p.L * p.P * ctx->Pz));
    return launch_px_inv<float>(ctx, (const float2*)p.buf, H, 3L * ctx->nz * ctx->ny, scale, (const float2*)p.tw);
}

}  // namespace mm
