// FP64 plane-layout passes for small meshes: one thread per transform output.
//
// An SM sub-partition issues one FP64 warp instruction per 64 cycles, whether
// 32 lanes take part or 3.  The register four-step (mm_plane.cuh) gives a
// 100x25x1 plane to 24 threads with 300 FP64 instructions each: one warp, 14
// us, three sub-partitions idle.  Here a level is a radix-2 step of the
// Stockham autosort (a radix-3 or -5 step last where the length has that
// factor) and every thread forms one output, x0 + w x1 in four fused
// multiply-adds, so each level fills all lanes of all four sub-partitions; the
// levels' shared-memory round trips and barriers hide behind 4 x 64 issue
// cycles.  A fifth more FP64 instructions in all than the four-step, so the
// rule in mm_plane_f64.cu takes these kernels only while the mesh leaves the
// FP64 pipes of the chip idle.
// 100x25x1, one demag field: 38.7 -> 15.8 us; 128x128x1: 56.9 -> 30.8 us.
#include "mm_plane_launch.cuh"

namespace mm {
namespace {

// length n = odd << lg, odd = 1, 3 or 5
struct LiteLen {
    int n, lg, odd;
};
LiteLen lite_len(int n) {
    LiteLen l{n, 0, n};
    while (l.odd % 2 == 0) {
        l.odd /= 2;
        ++l.lg;
    }
    return l;
}

__device__ __forceinline__ double2 fma_c(double2 acc, double2 w, double2 x) {
    return make_double2(fma(w.x, x.x, fma(-w.y, x.y, acc.x)), fma(w.x, x.y, fma(w.y, x.x, acc.y)));
}
__device__ __forceinline__ double flip(double v, int neg) {   // the sign by integer operations
    return __hiloint2double(__double2hiint(v) ^ (neg << 31), __double2loint(v));
}

// Transforms `lines` lines of a, [line][n], whose first `from` radix-2 levels
// are done, with b as the other half of the ping-pong; the last level forms
// outputs o < keep only.  tw = exp(-2 pi i m / n).  Returns where the result
// is (natural order, same pitch).  Starts and ends with a barrier.
template <int DIR>
__device__ double2* lite_fft(double2* a, double2* b, int lines, LiteLen l, int from, int keep,
                             const double2* __restrict__ tw) {
    const int n = l.n, tid = threadIdx.x, nt = blockDim.x;
    __syncthreads();
    for (int lg = from; lg < l.lg; ++lg) {
        const int ns = 1 << lg, step = n >> (lg + 1), kept = lg == l.lg - 1 && l.odd == 1 ? keep : n;
        for (int i = tid; i < lines * kept; i += nt) {
            const int line = i / kept, o = i - line * kept;
            const double2* x = a + line * n + ((o >> (lg + 1)) << lg) + (o & (ns - 1));
            const double2 x0 = x[0], x1 = x[n >> 1];
            const int t = o & (2 * ns - 1);
            double2 y;
            if (lg == 0) {
                y = make_double2(x0.x + flip(x1.x, t), x0.y + flip(x1.y, t));
            } else if (lg == 1) {
                // w^t = 1, DIR i, -1, -DIR i
                const bool rot = t & 1;
                const int neg = t >> 1, nx = rot ? neg ^ (DIR > 0 ? 1 : 0) : neg, ny = rot ? neg ^ (DIR > 0 ? 0 : 1) : neg;
                y = make_double2(x0.x + flip(rot ? x1.y : x1.x, nx), x0.y + flip(rot ? x1.x : x1.y, ny));
            } else {
                double2 w = tw[t * step];
                if (DIR > 0) w.y = -w.y;
                y = fma_c(x0, w, x1);
            }
            b[line * n + o] = y;
        }
        __syncthreads();
        double2* const s = a;
        a = b;
        b = s;
    }
    if (l.odd > 1) {
        const int ns = 1 << l.lg;
        for (int i = tid; i < lines * keep; i += nt) {
            const int line = i / keep, o = i - line * keep;
            const double2* x = a + line * n + (o & (ns - 1));
            double2 y = x[0];
            int m = 0;
            for (int r = 1; r < l.odd; ++r) {
                m += o;
                if (m >= n) m -= n;
                double2 w = tw[m];
                if (DIR > 0) w.y = -w.y;
                y = fma_c(y, w, x[r * ns]);
            }
            b[line * n + o] = y;
        }
        __syncthreads();
        return b;
    }
    return a;
}

__device__ __forceinline__ void lite_table(double2* t, const double2* __restrict__ tw, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = tw[i];
}

// rows of M -> planes, RB rows per block (k_px_fwd's data flow)
__global__ void __launch_bounds__(256)
    k_lx_fwd(const double* __restrict__ in, int nx, const double* __restrict__ Ms, double ms, long ms_rows,
             double2* __restrict__ out, long R, long rows, int RB, LiteLen l, const double2* __restrict__ twL,
             const double2* __restrict__ twP) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* a = reinterpret_cast<double2*>(smem_raw);
    const int L = l.n, H = L >> 1;
    double2* b = a + RB * L;
    double2* t = b + RB * L;
    lite_table(t, twL, L);
    const long r0 = (long)blockIdx.x * RB;
    for (int i = threadIdx.x; i < RB * H; i += blockDim.x) {
        const int br = i / H, x = 2 * (i - br * H);
        const long r = r0 + br;
        double2 v = make_double2(0.0, 0.0);
        if (r < rows && x < nx) {
            const double* mrow = Ms ? Ms + (r % ms_rows) * nx + x : nullptr;
            // the half of the real-to-complex split below, exact here
            v.x = in[r * nx + x] * (0.5 * (Ms ? mrow[0] : ms));
            if (x + 1 < nx) v.y = in[r * nx + x + 1] * (0.5 * (Ms ? mrow[1] : ms));
        }
        a[br * L + x] = v;          // the first level's outputs: its odd inputs are the zero padding
        a[br * L + x + 1] = v;
    }
    const double2* s = lite_fft<-1>(a, b, RB, l, 1, L, t);
    for (int i = threadIdx.x; i < RB * (H + 1); i += blockDim.x) {
        const int k = i / RB, br = i - k * RB;
        const long r = r0 + br;
        if (r >= rows) continue;
        const double2 zk = s[br * L + k], zc = s[br * L + (k ? L - k : 0)], w = twP[k];
        const double2 e = make_double2(zk.x + zc.x, zk.y - zc.y), d = make_double2(zk.x - zc.x, zk.y + zc.y);
        const double2 wd = make_double2(w.x * d.x - w.y * d.y, w.x * d.y + w.y * d.x);
        out[(long)k * R + r] = make_double2(e.x + wd.y, e.y - wd.x);
        if (2 * k != L) out[(long)(L - k) * R + r] = make_double2(e.x - wd.y, -(e.y + wd.x));
    }
}

__global__ void __launch_bounds__(256)
    k_lx_inv(const double2* __restrict__ in, long R, double* __restrict__ out, int nx, long rows, double scale, int RB,
             LiteLen l, const double2* __restrict__ twL, const double2* __restrict__ twP) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* a = reinterpret_cast<double2*>(smem_raw);
    const int L = l.n, H = L >> 1;
    double2* b = a + RB * L;
    double2* t = b + RB * L;
    lite_table(t, twL, L);
    const long r0 = (long)blockIdx.x * RB;
    for (int i = threadIdx.x; i < RB * (H + 1); i += blockDim.x) {
        const int k = i / RB, br = i - k * RB;
        const long r = r0 + br;
        double2 xk = make_double2(0.0, 0.0), xl = xk;
        if (r < rows) {
            xk = in[(long)k * R + r];
            xl = in[(long)(L - k) * R + r];
        }
        const double2 w = twP[k];
        const double2 e = make_double2(xk.x + xl.x, xk.y - xl.y), d = make_double2(xk.x - xl.x, xk.y + xl.y);
        const double2 o = make_double2(d.x * w.x + d.y * w.y, d.y * w.x - d.x * w.y);      // d conj(w)
        a[br * L + k] = make_double2(e.x - o.y, e.y + o.x);                                // E + i O, twice
        if (k > 0 && 2 * k != L) a[br * L + L - k] = make_double2(e.x + o.y, o.x - e.y);
    }
    const int keep = (nx + 1) >> 1;
    const double2* s = lite_fft<+1>(a, b, RB, l, 0, keep, t);
    for (int i = threadIdx.x; i < RB * keep; i += blockDim.x) {
        const int br = i / keep, x = 2 * (i - br * keep);
        const long r = r0 + br;
        if (r >= rows) continue;
        const double2 z = s[br * L + (x >> 1)];
        out[r * nx + x] = z.x * scale;
        if (x + 1 < nx) out[r * nx + x + 1] = z.y * scale;
    }
}

// one plane of a single layer per block: y forward, product, y inverse
// (k_plane's data flow)
__global__ void __launch_bounds__(256)
    k_lplane(double2* __restrict__ buf, const double* __restrict__ kern, int ny, long R, int KQ, LiteLen l,
             const double2* __restrict__ tw) {
    dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = l.n, lines = 3, nk = 6 * KQ;
    double2* a = reinterpret_cast<double2*>(smem_raw);
    double2* b = a + lines * P;
    double2* t = b + lines * P;
    double* kp = reinterpret_cast<double*>(t + P);
    const double* kg = kern + (long)blockIdx.x * nk;
    for (int i = threadIdx.x; i < nk; i += blockDim.x) cp_async_value(kp + i, kg + i);
    lite_table(t, tw, P);
    double2* base = buf + (long)blockIdx.x * R;
    for (int i = threadIdx.x; i < lines * (P >> 1); i += blockDim.x) {
        const int line = i / (P >> 1), y = i - line * (P >> 1);
        const double2 v = y < ny ? base[(long)line * ny + y] : make_double2(0.0, 0.0);
        a[line * P + 2 * y] = v;
        a[line * P + 2 * y + 1] = v;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    double2* s = lite_fft<-1>(a, b, lines, l, 1, P, t);
    double2* const o = s == a ? b : a;
    // one component of one k point per thread
    for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
        const int c = i / P, ky = i - c * P;
        const bool yodd = 2 * ky > P;
        const double* kb = kp + (yodd ? P - ky : ky);
        const int n0 = c == 0 ? 0 : c == 1 ? 3 : 4, n1 = c == 0 ? 3 : c == 1 ? 1 : 5, n2 = c == 0 ? 4 : c == 1 ? 5 : 2;
        const double q0 = flip(kb[n0 * KQ], 1 ^ (yodd && n0 == 3)), q1 = flip(kb[n1 * KQ], 1 ^ (yodd && n1 != 1)),
                     q2 = flip(kb[n2 * KQ], 1 ^ (yodd && n2 == 5));
        const double2 x = s[ky], y = s[P + ky], z = s[2 * P + ky];
        o[i] = make_double2(q0 * x.x + q1 * y.x + q2 * z.x, q0 * x.y + q1 * y.y + q2 * z.y);
    }
    s = lite_fft<+1>(o, s, lines, l, 0, ny, t);
    for (int i = threadIdx.x; i < lines * ny; i += blockDim.x) {
        const int line = i / ny, y = i - line * ny;
        base[i] = s[line * P + y];
    }
}

// rows per block: 128 outputs a level or one row
int lite_rows(int L) { return L >= 128 ? 1 : 128 / L; }
}  // namespace

int lite_xfwd(mm_ctx* ctx, const double* m, const double* Ms, double ms) {
    const PlanePlan& p = ctx->plane;
    const double2* tw = (const double2*)p.tw;
    const long rows = 3L * ctx->nz * ctx->ny;
    const int RB = lite_rows(p.L), nt = RB * p.L >= 256 ? 256 : 128;
    const size_t smem = (size_t)(2 * RB + 1) * p.L * sizeof(double2);
    KernelTimer kt(ctx, MM_K_XFWD);
    dep(k_lx_fwd, (unsigned)((rows + RB - 1) / RB), nt, smem, ctx->stream)(
        m, ctx->nx, Ms, ms, (long)ctx->nz * ctx->ny, (double2*)p.buf, p.R, rows, RB, lite_len(p.L), tw, tw + p.off_p);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

int lite_xinv(mm_ctx* ctx, double* H) {
    const PlanePlan& p = ctx->plane;
    const double2* tw = (const double2*)p.tw;
    const long rows = 3L * ctx->nz * ctx->ny;
    const int RB = lite_rows(p.L), nt = RB * p.L >= 256 ? 256 : 128;
    const size_t smem = (size_t)(2 * RB + 1) * p.L * sizeof(double2);
    KernelTimer kt(ctx, MM_K_XINV);
    // the pack leaves twice the spectrum: half of it belongs to the scale
    dep(k_lx_inv, (unsigned)((rows + RB - 1) / RB), nt, smem, ctx->stream)(
        (const double2*)p.buf, p.R, H, ctx->nx, rows, 0.5 / ((double)p.L * p.P * ctx->Pz), RB, lite_len(p.L), tw,
        tw + p.off_p);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

// single layers only
int lite_plane(mm_ctx* ctx) {
    const PlanePlan& p = ctx->plane;
    const double2* tw = (const double2*)p.tw;
    const size_t smem = (size_t)7 * p.P * sizeof(double2) + (size_t)6 * p.KQ * sizeof(double);
    int rc = smem_opt_in(ctx, (const void*)k_lplane, smem);
    if (rc) return rc;
    const int tasks = 3 * p.P;
    const int nt = tasks >= 256 ? 256 : (tasks + 31) / 32 * 32;
    KernelTimer kt(ctx, MM_K_ZCONV);
    dep(k_lplane, (unsigned)p.K, nt, smem, ctx->stream)((double2*)p.buf, (const double*)p.kern, ctx->ny, p.R,
                                                       p.KQ, lite_len(p.P), tw + p.off_y);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

}  // namespace mm
