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

namespace {

template <int L1, int L2, int B, int NT, int MINB>
int zline_ff_t(mm_ctx* ctx, ffc* buf, const ff* kern, const ZLine& g, const ffc* tw) {
    KernelTimer kt(ctx, MM_K_ZCONV);
    auto fn = k_zline<ff, L1, L2, false, B, NT, MINB>;
    const size_t smem = zline_smem<ff, L1, L2, B>();
    int rc = smem_opt_in(ctx, (const void*)fn, smem);
    if (rc) return rc;
    dim3 grid((unsigned)((g.ncol + B - 1) / B), (unsigned)ctx->Py);
    dep(fn, grid, NT, smem, ctx->stream)(buf, kern, g, tw);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

}  // namespace

// Float-float z pass with both levels and the product in registers: the
// Stockham stages (k_zconv) passed every value through shared memory and two
// barriers per stage, and the product once more.  Pz = 32 (512x512x16): 1220
// -> 783 us (32 columns and 256 threads a block; 16 and 128: 801, 8 and 96:
// 885); Pz = 16 (256x256x8): 158 -> 109; Pz = 64 (128x128x32): 206 -> 183.
// Errors against native FP64 are the same (6.40e-15 on 512x512x16).  Longer
// lines do not fit a thread's registers.
bool zline_ff_takes(int Pz) { return Pz == 16 || Pz == 32 || Pz == 64; }

int zline_ff(mm_ctx* ctx, ffc* buf, const ff* kern, const ffc* tw) {
    const long zs = (long)ctx->Py * ctx->Hs, kz = (long)ctx->Py2 * ctx->Hs;
    const ZLine g{ctx->Hs, ctx->nz * zs, zs, ctx->Hs, ctx->Pz2 * kz, kz, ctx->nz, ctx->Hx, ctx->Py};
    switch (ctx->Pz) {
        case 16: return zline_ff_t<4, 4, 16, 128, 4>(ctx, buf, kern, g, tw);
        case 32: return zline_ff_t<8, 4, 32, 256, 2>(ctx, buf, kern, g, tw);
        default: return zline_ff_t<8, 8, 8, 96, 3>(ctx, buf, kern, g, tw);
    }
}

}  // namespace mm
