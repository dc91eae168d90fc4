// Plane-layout demag passes in FP32: y forward, z product, y inverse.
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f32(mm_ctx* ctx) {
    const PlanePlan& p = ctx->plane;
    const float2* tw = (const float2*)p.tw;
    float2* buf = (float2*)p.buf;
    const float* kern = (const float*)p.kern;
    if (!p.lines) return launch_plane<float>(ctx, buf, kern, tw);
    float2* wide = (float2*)p.buf2;
    int rc = launch_py<float, -1>(ctx, buf, wide, tw);
    if (rc) return rc;
    const ZLine g{3L * ctx->nz * p.P, (long)ctx->nz * p.P, p.P, 6L * ctx->Pz2 * p.KQ, (long)ctx->Pz2 * p.KQ, p.KQ,
                  ctx->nz, p.P, p.P};
    if ((rc = launch_zline<float, true>(ctx, ctx->Pz, wide, kern, g, p.K, tw + p.off_z4))) return rc;
    return launch_py<float, +1>(ctx, wide, buf, tw);
}

}  // namespace mm
