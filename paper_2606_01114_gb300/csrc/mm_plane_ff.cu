// Plane-layout demag passes in float-float arithmetic (MM_FFT_FF on an FP64
// context): m, Ms and H stay double, the planes hold ffc.  The transforms run
// on the shared-memory Stockham engine (mm_fft.cuh) and not on the register
// four-step: a 32-point float-float DFT unrolled in registers is thousands of
// instructions per kernel, and the radix-8 stages do the same arithmetic.
// Power-of-two meshes only (checked when the mode is set).
#include "mm_fft.cuh"
#include "mm_plane.cuh"

namespace mm {
namespace {

constexpr int kThreads = 256;        // x passes: at most B L / 8 active threads
constexpr int kPlaneThreads = 384;   // plane kernel: 3 nz P / 8

// rows of M -> planes: B = 2^lgB rows per block
__global__ void __launch_bounds__(kThreads)
    k_ffx_fwd(const double* __restrict__ in, int nx, const double* __restrict__ Ms, ff ms, long ms_rows,
              ffc* __restrict__ out, long R, long rows, int lgL, int lgB, const ffc* __restrict__ twL,
              const ffc* __restrict__ twP) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ffc* s = reinterpret_cast<ffc*>(smem_raw);
    const int L = 1 << lgL, B = 1 << lgB;
    const FftGeom g = fft_geom(L, B, 1, sizeof(ffc));
    const long r0 = (long)blockIdx.x << lgB;
    // rows read along x (consecutive threads, consecutive pairs)
    for (int idx = threadIdx.x; idx < (B << lgL); idx += blockDim.x) {
        const int b = idx >> lgL, j = idx & (L - 1);
        const long r = r0 + b;
        ffc v = cmk<ffc>(ff(0), ff(0));
        if (2 * j < nx && r < rows) {
            const double2 d = reinterpret_cast<const double2*>(in + r * nx)[j];
            v = cmk<ffc>(d2ff(d.x), d2ff(d.y));
            if (Ms) {
                const double2 w = reinterpret_cast<const double2*>(Ms + (r % ms_rows) * nx)[j];
                v.x *= d2ff(w.x);
                v.y *= d2ff(w.y);
            } else {
                v.x *= ms;
                v.y *= ms;
            }
        }
        s[sidx(g, 0, j, b)] = v;
    }
    __syncthreads();
    fft_lines<-1, true>(s, g, twL);
    const ff half = ff(0.5f);
    for (int idx = threadIdx.x; idx < (B << (lgL - 1)) + B; idx += blockDim.x) {
        const int b = idx & (B - 1), k = idx >> lgB;        // k = 0 .. L / 2
        const long r = r0 + b;
        if (r >= rows) continue;
        const ffc zk = s[sidx(g, 0, k, b)];
        const ffc zc = cconj(s[sidx(g, 0, (L - k) & (L - 1), b)]);
        const ffc e = cscale(cadd(zk, zc), half);
        const ffc wd = cmul(twP[k], cscale(csub(zk, zc), half));
        out[(long)k * R + r] = cmk<ffc>(e.x + wd.y, e.y - wd.x);
        if (2 * k != L) out[(long)(L - k) * R + r] = cmk<ffc>(e.x - wd.y, -(e.y + wd.x));
    }
}

__global__ void __launch_bounds__(kThreads)
    k_ffx_inv(const ffc* __restrict__ in, long R, double* __restrict__ out, int nx, long rows, ff scale, int lgL,
              int lgB, const ffc* __restrict__ twL, const ffc* __restrict__ twP) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ffc* s = reinterpret_cast<ffc*>(smem_raw);
    const int L = 1 << lgL, B = 1 << lgB;
    const FftGeom g = fft_geom(L, B, 1, sizeof(ffc));
    const long r0 = (long)blockIdx.x << lgB;
    const ff half = ff(0.5f);
    for (int idx = threadIdx.x; idx < (B << (lgL - 1)) + B; idx += blockDim.x) {
        const int b = idx & (B - 1), k = idx >> lgB;
        const long r = r0 + b;
        ffc xk = cmk<ffc>(ff(0), ff(0)), xl = xk;
        if (r < rows) {
            xk = in[(long)k * R + r];
            xl = cconj(in[(long)(L - k) * R + r]);
        }
        const ffc e = cscale(cadd(xk, xl), half);
        const ffc o = cmul(cscale(csub(xk, xl), half), cconj(twP[k]));
        s[sidx(g, 0, k, b)] = cmk<ffc>(e.x - o.y, e.y + o.x);
        if (k > 0 && 2 * k != L) s[sidx(g, 0, L - k, b)] = cmk<ffc>(e.x + o.y, o.x - e.y);
    }
    __syncthreads();
    fft_lines<+1, false, true>(s, g, twL);
    const int half_n = nx >> 1;
    for (int idx = threadIdx.x; idx < B * half_n; idx += blockDim.x) {
        const int b = idx / half_n, j = idx - b * half_n;
        const long r = r0 + b;
        if (r >= rows) continue;
        const ffc z = s[sidx(g, 0, j, b)];
        reinterpret_cast<double2*>(out + r * nx)[j] = make_double2(ff2d(z.x * scale), ff2d(z.y * scale));
    }
}

// one plane per block: y forward, z product, y inverse
template <int NZ>
__global__ void __launch_bounds__(kPlaneThreads)
    k_ff_plane(ffc* __restrict__ buf, const ff* __restrict__ kern, int ny, long R, int KQ, int lgP,
               const ffc* __restrict__ tw) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ffc* s = reinterpret_cast<ffc*>(smem_raw);
    const int P = 1 << lgP;
    constexpr int PZ = NZ > 1 ? 2 * NZ : 1, PZ2 = PZ / 2 + 1;
    const FftGeom g = fft_geom(P, NZ, 3, sizeof(ffc));
    ffc* base = buf + (long)blockIdx.x * R;
    const ff* kp = kern + (long)blockIdx.x * 6 * PZ2 * KQ;
    for (int i = threadIdx.x; i < 3 * NZ * P; i += blockDim.x) {
        const int y = i & (P - 1), line = i >> lgP;
        s[sidx(g, line / NZ, y, line % NZ)] = y < ny ? base[(long)line * ny + y] : cmk<ffc>(ff(0), ff(0));
    }
    __syncthreads();
    fft_lines<-1, true>(s, g, tw);
    for (int ky = threadIdx.x; ky < P; ky += blockDim.x) {
        const bool yodd = 2 * ky > P;
        const ff* kb = kp + (yodd ? P - ky : ky);
        ffc v[3][PZ];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int z = 0; z < NZ; ++z) v[c][z] = s[sidx(g, c, ky, z)];
            dif<PZ, -1, (PZ > 1)>(v[c]);
        }
#pragma unroll
        for (int kz = 0; kz < PZ; ++kz) {
            const int kzp = kz <= PZ / 2 ? kz : PZ - kz;
            const bool zodd = kz > PZ / 2;
            const ff xx = kb[(0 * PZ2 + kzp) * KQ], yy = kb[(1 * PZ2 + kzp) * KQ], zz = kb[(2 * PZ2 + kzp) * KQ];
            ff xy = kb[(3 * PZ2 + kzp) * KQ], xz = kb[(4 * PZ2 + kzp) * KQ], yz = kb[(5 * PZ2 + kzp) * KQ];
            if (yodd) xy = -xy;
            if (zodd) xz = -xz;
            if (yodd != zodd) yz = -yz;
            const int q = dif_pos<PZ>(kz);
            tensor_product<ff>(v[0][q], v[1][q], v[2][q], xx, yy, zz, xy, xz, yz);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ffc u[PZ];
#pragma unroll
            for (int kz = 0; kz < PZ; ++kz) u[kz] = v[c][dif_pos<PZ>(kz)];
            dif<PZ, +1, false>(u);
#pragma unroll
            for (int z = 0; z < NZ; ++z) s[sidx(g, c, ky, z)] = u[dif_pos<PZ>(z)];
        }
    }
    __syncthreads();
    fft_lines<+1, false, true>(s, g, tw);
    for (int i = threadIdx.x; i < 3 * NZ * ny; i += blockDim.x) {
        const int line = i / ny, y = i - line * ny;
        base[i] = s[sidx(g, line / NZ, y, line % NZ)];
    }
}

template <int NZ>
int launch_ff_plane(mm_ctx* ctx, ffc* buf, const ffc* tw) {
    const PlanePlan& p = ctx->plane;
    KernelTimer kt(ctx, MM_K_ZCONV);
    const size_t smem = (size_t)3 * NZ * p.P * sizeof(ffc);
    int rc = smem_opt_in(ctx, (const void*)k_ff_plane<NZ>, smem);
    if (rc) return rc;
    const int nt = (3 * NZ * p.P / 8 + 31) / 32 * 32;     // the Stockham stages need 3 nz P / 8 threads
    dep(k_ff_plane<NZ>, (unsigned)p.K, nt, smem, ctx->stream)(buf, (const ff*)p.kern_ff, ctx->ny, p.R, p.KQ, ilog2(p.P),
                                                             tw + p.off_y);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

}  // namespace

// whether the float-float plane kernel takes this mesh: the Stockham stages
// need 3 nz P / 8 threads, and 384 leave the z phase its 168 registers.  At
// four layers and that size a block fills an SM for longer than the five
// passes take once there are more than two planes an SM (512x128x4 170 us
// against 177; 256x128x4 113 against 92).
bool plane_ff_fits(const mm_ctx* ctx) {
    const PlanePlan& p = ctx->plane;
    const int work = 3 * ctx->nz * p.P;
    if (!p.on || ctx->nz > 4 || ctx->nx % 2 || work > 8 * kPlaneThreads) return false;
    return ctx->nz < 4 || work <= 4 * kPlaneThreads || p.K <= 2 * kSMs;
}

int plane_apply_ff(mm_ctx* ctx, const double* m, const double* Ms, double ms, double* H) {
    const PlanePlan& p = ctx->plane;
    const long rows = 3L * ctx->nz * ctx->ny;
    const ffc* tw = (const ffc*)p.tw_ff;
    ffc* buf = (ffc*)p.buf;
    const int lgL = ilog2(p.L);
    // 64-byte segments per plane (8 rows of short lines); 32-byte ones while the
    // larger blocks are too few to share the SMs evenly (256x256x1: 192 blocks)
    const int lgB = lgL < 6 ? 3 : rows < 16 * kSMs ? 1 : 2;
    const int nt = ((1 << (lgL + lgB - 3)) + 31) / 32 * 32;
    const size_t smem = sizeof(ffc) << (lgL + lgB);
    const unsigned nb = (unsigned)((rows + (1 << lgB) - 1) >> lgB);
    int rc;
    {
        KernelTimer kt(ctx, MM_K_XFWD);
        dep(k_ffx_fwd, nb, nt, smem, ctx->stream)(m, ctx->nx, Ms, ff(ms), (long)ctx->nz * ctx->ny, buf, p.R, rows, lgL,
                                                 lgB, tw, tw + p.off_p);
        MM_LAUNCH_CHECK(ctx);
    }
    switch (ctx->nz) {
        case 1: rc = launch_ff_plane<1>(ctx, buf, tw); break;
        case 2: rc = launch_ff_plane<2>(ctx, buf, tw); break;
        default: rc = launch_ff_plane<4>(ctx, buf, tw); break;
    }
    if (rc) return rc;
    KernelTimer kt(ctx, MM_K_XINV);
    dep(k_ffx_inv, nb, nt, smem, ctx->stream)(buf, p.R, H, ctx->nx, rows, ff(1.0 / ((double)p.L * p.P * ctx->Pz)), lgL,
                                             lgB, tw, tw + p.off_p);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

}  // namespace mm
