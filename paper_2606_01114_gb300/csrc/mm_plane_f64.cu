// Plane-layout demag passes in FP64: the x passes and the sequence (the plane
// and line kernels: mm_plane_f64y.cu).
#include "mm_plane_launch.cuh"

namespace mm {

int plane_yzy_f64(mm_ctx* ctx);
// one thread per transform output (mm_plane_lite.cu)
int lite_xfwd(mm_ctx* ctx, const double* m, const double* Ms, double ms);
int lite_xinv(mm_ctx* ctx, double* H);
int lite_plane(mm_ctx* ctx);

// Where one thread per output is the faster form, in complex outputs of a
// pass.  x passes (forward + inverse, four-step -> one output a thread):
// 100x25x1 36.4 -> 17.0 us, 128x128x4 (197 k) 41.2 -> 38.5, 256x128x4 (393 k)
// 69.1 -> 67.0, 256x256x4 (786 k) the four-step.  Plane pass, nz = 1:
// 100x25x1 (19 k) 16.2 -> 10.5 us, 64x64x1 23.3 -> 15.4, 128x128x1 (99 k)
// 33.5 -> 23.1, 200x150x1 (231 k) 47.5 -> 51.0, 256x256x1 (395 k) 72.1 -> 72.6
// (events around single kernels, some 5 us of each are launch).
constexpr long kLiteX = 300000, kLitePlane = 150000;

int plane_apply_f64(mm_ctx* ctx, const double* m, const double* Ms, double ms, double* H) {
    const PlanePlan& p = ctx->plane;
    const long rows = 3L * ctx->nz * ctx->ny;
    const double2* tw = (const double2*)p.tw;
    double2* buf = (double2*)p.buf;
    const bool lite_x = rows * p.L <= kLiteX;
    const bool lite_yz = ctx->nz == 1 && !p.lines && 3L * p.K * p.P <= kLitePlane;
    int rc = lite_x ? lite_xfwd(ctx, m, Ms, ms)
                    : launch_px_fwd<double>(ctx, m, Ms, ms, (long)ctx->nz * ctx->ny, buf, rows, tw);
    if (rc || (rc = lite_yz ? lite_plane(ctx) : plane_yzy_f64(ctx))) return rc;
    if (lite_x) return lite_xinv(ctx, H);
    return launch_px_inv<double>(ctx, buf, H, rows, 1.0 / ((double)p.L * p.P * ctx->Pz), tw);
}

}  // namespace mm
