// Plane-layout demag passes in FP64: y forward, z product, y inverse.
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f64(mm_ctx* ctx) {
    const PlanePlan& p = ctx->plane;
    const double2* tw = (const double2*)p.tw;
    double2* buf = (double2*)p.buf;
    const double* kern = (const double*)p.kern;
    if (!p.lines) return launch_plane<double>(ctx, buf, kern, tw);
    double2* wide = (double2*)p.buf2;
    int rc = launch_py<double, -1>(ctx, buf, wide, tw);
    if (rc) return rc;
    const ZLine g{3L * ctx->nz * p.P, (long)ctx->nz * p.P, p.P, 6L * ctx->Pz2 * p.KQ, (long)ctx->Pz2 * p.KQ, p.KQ,
                  ctx->nz, p.P, p.P};
    if ((rc = launch_zline<double, true>(ctx, ctx->Pz, wide, kern, g, p.K, tw + p.off_z4))) return rc;
    return launch_py<double, +1>(ctx, wide, buf, tw);
}

}  // namespace mm
