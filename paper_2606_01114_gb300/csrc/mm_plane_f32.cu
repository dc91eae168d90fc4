// Plane-layout demag passes in FP32: the x passes and the sequence (the plane
// and line kernels: mm_plane_f32y.cu).
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f32(mm_ctx* ctx);

int plane_line_len(int P) { return plane_line(P); }

int plane_apply_f32(mm_ctx* ctx, const float* m, const float* Ms, float ms, float* H) {
    const PlanePlan& p = ctx->plane;
    const long rows = 3L * ctx->nz * ctx->ny;
    const float2* tw = (const float2*)p.tw;
    float2* buf = (float2*)p.buf;
    int rc = launch_px_fwd<float, float>(ctx, m, Ms, ms, (long)ctx->nz * ctx->ny, buf, rows, tw);
    if (rc || (rc = plane_yzy_f32(ctx))) return rc;
    const float scale = (float)(1.0 / ((double)p.L * p.P * ctx->Pz));
    return launch_px_inv<float, float>(ctx, buf, H, rows, scale, tw);
}

}  // namespace mm
