// The z pass of the [c][z][y][kx] demag passes on long z lines (FP32,
// Pz >= 64): k_zline with kx columns.  The generic pass (k_zconv) ran the
// radix-8 Stockham stages through shared memory at 1024 threads per block:
// 256^3 (Pz = 512) 2815 us, here 950 us.
#include "mm_plane_launch.cuh"

namespace mm {

int zline_f32(mm_ctx* ctx, float2* buf, const float* kern, const float2* tw) {
    const long zs = (long)ctx->Py * ctx->Hs, kz = (long)ctx->Py2 * ctx->Hs;
    const ZLine g{ctx->Hs, ctx->nz * zs, zs, ctx->Hs, ctx->Pz2 * kz, kz, ctx->nz, ctx->Hx, ctx->Py};
    return launch_zline<float, false>(ctx, ctx->Pz, buf, kern, g, ctx->Py, tw);
}

}  // namespace mm
