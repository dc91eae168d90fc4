// Plane-layout demag passes in FP64: the x passes and the sequence (the plane
// and line kernels: mm_plane_f64y.cu).
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f64(mm_ctx* ctx);

int plane_apply_f64(mm_ctx* ctx, const double* m, const double* Ms, double ms, double* H) {
    const PlanePlan& p = ctx->plane;
    const long rows = 3L * ctx->nz * ctx->ny;
    const double2* tw = (const double2*)p.tw;
    double2* buf = (double2*)p.buf;
    int rc = launch_px_fwd<double, double>(ctx, m, Ms, ms, (long)ctx->nz * ctx->ny, buf, rows, tw);
    if (rc || (rc = plane_yzy_f64(ctx))) return rc;
    return launch_px_inv<double, double>(ctx, buf, H, rows, 1.0 / ((double)p.L * p.P * ctx->Pz), tw);
}

}  // namespace mm
