// The plane-layout demag path: plan, octant and sequencing (the kernels and
// their layout: mm_plane.cuh).
#include <algorithm>
#include <cmath>
#include <vector>

#include "mm_ff.cuh"

namespace mm {

// per element type (mm_plane_f32.cu, mm_plane_f64.cu, mm_plane_ff.cu)
int plane_apply_f32(mm_ctx* ctx, const float* m, const float* Ms, float ms, float* H);
int plane_apply_f64(mm_ctx* ctx, const double* m, const double* Ms, double ms, double* H);
int plane_apply_ff(mm_ctx* ctx, const double* m, const double* Ms, double ms, double* H);
int plane_xfwd_f32(mm_ctx* ctx, const float* m, const float* Ms, float ms);
int plane_yzy_f32(mm_ctx* ctx);
int plane_line_len(int P);

namespace {

bool pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }

// next of `least` (4 or 8), 8, 16, 32 and {4, 5, 6} 2^k, k >= 3, that is >= n
int next_len(int n, int least) {
    for (int l = least; l <= 32; l *= 2)
        if (n <= l) return l;
    for (int p = 32;; p *= 2)
        for (int q = 4; q <= 6; ++q)
            if (q * p / 4 >= n) return q * p / 4;
}

// One axis of the octant's transform by its definition: the Newell tensor is
// even or odd along each axis, so its DFT over the padded length P is
//   even: N_0 + 2 sum_j N_j cos(2 pi j k / P),  odd: 2 sum_j N_j sin(2 pi j k / P)
// (the factors -i of two odd axes make the -1 that the last axis applies).
// in [O][n][I] -> out [O][m][I]; tab = cos or sin of 2 pi q / P, q < P.
// Setup only: O(n) FP64 multiply-adds per output, any length.
__global__ void k_octant_axis(const double* __restrict__ in, double* __restrict__ out, long O, int n, int I, int m,
                              int P, int odd, const double* __restrict__ tab) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= O * m * I) return;
    const int i = (int)(idx % I);
    const long r = idx / I;
    const int k = (int)(r % m);
    const double* p = in + (r / m) * n * (long)I + i;
    double a0 = 0.0, a1 = 0.0;
    int q = k;
    for (int j = 1; j < n; ++j) {
        const double w = tab[q];
        if (j & 1) a0 += p[(long)j * I] * w;
        else a1 += p[(long)j * I] * w;
        q += k;
        if (q >= P) q -= P;
    }
    out[idx] = (odd ? 0.0 : p[0]) + 2.0 * (a0 + a1);
}

// [kz][ky][kx] of one component -> its place in [K][6][Pz2][KQ]
template <typename T>
__global__ void k_octant_place(const double* __restrict__ in, T* __restrict__ kern, int comp, int K, int Pz2, int Py2,
                               int KQ, double sign) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)K * Pz2 * KQ) return;
    const int ky = (int)(idx % KQ);
    const int kz = (int)(idx / KQ % Pz2);
    const long kx = idx / ((long)KQ * Pz2);
    kern[((kx * 6 + comp) * Pz2 + kz) * KQ + ky] =
        ky < Py2 ? (T)(sign * in[((long)kz * Py2 + ky) * K + kx]) : (T)0;
}

// [kz][ky][kx] of one component -> its part [Pz2][Py2][Hs] of the [c][z][y][kx] octant
template <typename T>
__global__ void k_octant_rows(const double* __restrict__ in, T* __restrict__ kern, int Hx, int Hs, long rows,
                              double sign) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * Hs) return;
    const int kx = (int)(idx % Hs);
    kern[idx] = kx < Hx ? (T)(sign * in[idx / Hs * Hx + kx]) : (T)0;
}

// octant of the [c][z][y][kx] passes, [6][Pz2][Py2][Hs] -> [K][6][Pz2][KQ]
template <typename T>
__global__ void k_octant_turn(const T* __restrict__ in, T* __restrict__ kern, int K, int Pz2, int Py2, int Hs, int KQ) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)K * 6 * Pz2 * KQ) return;
    const int ky = (int)(idx % KQ);
    const long r = idx / KQ;
    const int cz = (int)(r % (6 * Pz2));     // comp Pz2 + kz
    const long kx = r / (6 * Pz2);
    kern[idx] = ky < Py2 ? in[((long)cz * Py2 + ky) * Hs + kx] : (T)0;
}

__global__ void k_split(const double* __restrict__ in, ff* __restrict__ out, long n) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double d = in[i];
    const float h = __double2float_rn(d);
    out[i] = ff(h, __double2float_rn(d - (double)h));
}

unsigned blocks(long n) { return (unsigned)((n + 255) / 256); }
size_t elem(const mm_ctx* ctx) { return ctx->prec == MM_F64 ? 8 : 4; }
long kern_count(const mm_ctx* ctx) { return (long)ctx->plane.K * 6 * ctx->Pz2 * ctx->plane.KQ; }
long tw_count(const mm_ctx* ctx) { return 2 * ctx->plane.tw_len; }

}  // namespace

// Which contexts run in the plane layout: every mesh with nx, ny > 1 and a
// side that is not a power of two, and power-of-two meshes whose plane (3 nz
// lines of the padded y length) fits one block's shared memory with a z
// transform that fits a thread's registers (nz <= 8; FP64 and float-float 4).
// Power-of-two meshes also need two blocks per SM (113 KB a plane) or no more
// than two planes an SM; at one block per SM over more waves the five streaming
// passes are at least as fast: 512x512x8 FP32 153 against 157 us, 512x512x4 FP64
// 1797 against 1795.  On the near side of the line: 256x512x8 FP32 (257 planes)
// 69 against 83 us, 256x512x4 FP64 875 against 962, 64x512x8 29 against 43;
// with two blocks per SM 512x512x4 FP32 61 against 94, 256x256x8 31 against 56.
// The plane is a block's serial work, so few planes of many values leave most
// SMs idle.  In FP64 (one warp instruction per sub-partition and 64 cycles) that
// counts more than the two passes over memory it saves: up to 65 planes of nz P >= 256
// run y, z and y as three kernels.  FP64 demag, plane -> three kernels (-> the
// five passes of the power-of-two meshes): 16x512x4 342 -> 107 (150) us,
// 64x512x4 375 -> 252 (333), 16x256x2 81 -> 62 (115), 64x128x2 49 -> 45 (129),
// 32x64x4 43 -> 36 (123); at 97 planes 96x128x2 53 -> 53 and 96x64x2 37 -> 38.
// A side of three cells beside a power of two and many layers keeps the 2n
// passes: they are direct on that side (2n = 6, here 8) and need no chirp-z,
// and from about 98 k cells in FP64, 197 k in FP32 with ny = 3, the columns
// they save count more than launches: 512x3x256 FP64 939 against 1239 us,
// 3x512x128 654 against 774, 512x3x128 FP32 67 against 78 (256x3x128 47
// against 45, 3x512x512 356 against 271).
int plane_plan(mm_ctx* ctx) {
    PlanePlan& p = ctx->plane;
    p = PlanePlan();
    if (ctx->nx < 2 || ctx->ny < 2) return MM_OK;
    const size_t cs = 2 * elem(ctx);
    p.L = next_len(ctx->nx, 4);
    p.P = next_len(2 * ctx->ny, 8);     // (8: what the float-float stages need)
    const bool regular = pow2(ctx->nx) && pow2(ctx->ny);
    const size_t smem = 3 * (size_t)ctx->nz * plane_line_len(p.P) * cs;
    const bool fits = ctx->nz <= (ctx->prec == MM_F32 ? 8 : 4) && smem <= 227 * 1024;
    if (regular && (!fits || (smem > 113 * 1024 && p.L + 1 > 2 * kSMs))) return MM_OK;
    const bool strip = (ctx->nx == 3 && pow2(ctx->ny)) || (ctx->ny == 3 && pow2(ctx->nx));
    if (strip && (ctx->prec == MM_F64 ? ctx->N >= 98304 : ctx->ny == 3 && ctx->N >= 196608)) return MM_OK;
    p.on = 1;
    p.lines = !fits || (ctx->prec == MM_F64 && ctx->nz > 1 && p.L <= 64 && ctx->nz * p.P >= 256);
    p.K = p.L + 1;
    p.KQ = (p.P / 2 + 1 + 3) / 4 * 4;
    p.R = (3L * ctx->nz * ctx->ny + 3) / 4 * 4;
    p.off_p = p.L;
    p.off_y = p.off_p + 2 * p.L;
    std::vector<double> t;
    unit_circle(ctx, 2 * p.L);       // before L, which it gives
    for (int len : {p.L, 2 * p.L, p.P}) {
        const std::vector<double>& c = unit_circle(ctx, len);
        t.insert(t.end(), c.begin(), c.end());
    }
    long* const off4[3] = {&p.off_x4, &p.off_y4, &p.off_z4};
    const int len4[3] = {p.L, p.P, ctx->Pz};
    for (int a = 0; a < 3; ++a) {
        *off4[a] = (long)t.size() / 2;
        four_step_table(ctx, len4[a], a == 2, t);
    }
    p.tw_len = (long)t.size() / 2;
    int rc;
    if ((rc = dev_alloc(ctx, &p.buf, (size_t)p.K * p.R * cs))) return rc;
    if (p.lines && (rc = dev_alloc(ctx, &p.buf2, (size_t)p.K * 3 * ctx->nz * p.P * cs))) return rc;
    if ((rc = dev_alloc(ctx, &p.kern, (size_t)kern_count(ctx) * elem(ctx)))) return rc;
    if ((rc = dev_alloc(ctx, &p.tw, (size_t)tw_count(ctx) * elem(ctx)))) return rc;
    if (ctx->prec == MM_F64) {
        MM_CUDA_CHECK(ctx, cudaMemcpy(p.tw, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
    } else {
        std::vector<float> f(t.begin(), t.end());
        MM_CUDA_CHECK(ctx, cudaMemcpy(p.tw, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
    }
    return MM_OK;
}

void plane_free(mm_ctx* ctx) {
    PlanePlan& p = ctx->plane;
    void* ptrs[] = {p.buf, p.buf2, p.kern, p.kern_ff, p.tw, p.tw_ff};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    p = PlanePlan();
}

// Fills the plan's octant.  Same padded lengths as the [c][z][y][kx] passes
// (powers of two): their octant, turned.  Otherwise the Newell tensor
// transformed axis by axis from its definition; that also fills
// ctx->newell_host and the octant of the 2n lengths (mm_kspace_product reads it
// and must neither allocate nor wait).
int plane_setup(mm_ctx* ctx) {
    PlanePlan& p = ctx->plane;
    const int Pz2 = ctx->Pz2, Py2 = p.P / 2 + 1;
    if (ctx->kern_ready) {
        const long n = kern_count(ctx);
        if (ctx->prec == MM_F64)
            k_octant_turn<double><<<blocks(n), 256, 0, ctx->stream>>>((const double*)ctx->kern, (double*)p.kern, p.K, Pz2,
                                                                      Py2, ctx->Hs, p.KQ);
        else
            k_octant_turn<float><<<blocks(n), 256, 0, ctx->stream>>>((const float*)ctx->kern, (float*)p.kern, p.K, Pz2,
                                                                     Py2, ctx->Hs, p.KQ);
        MM_LAUNCH_CHECK(ctx);
        return MM_OK;
    }
    const int n[3] = {ctx->nx, ctx->ny, ctx->nz};
    // lengths and kept frequencies of the plan, and of the 2n octant
    const int len[2][3] = {{2 * p.L, p.P, ctx->Pz}, {ctx->Px, ctx->Py, ctx->Pz}};
    const int m[2][3] = {{p.K, Py2, Pz2}, {ctx->Hx, ctx->Py2, Pz2}};
    constexpr int sets = 2;
    std::vector<double> t;
    long off[2][3];
    for (int q = 0; q < sets; ++q)
        for (int a = 0; a < 3; ++a) {
            off[q][a] = (long)t.size();
            const std::vector<double>& e = unit_circle(ctx, len[q][a]);
            for (int s = 0; s < 2; ++s)
                for (int i = 0; i < len[q][a]; ++i) t.push_back(s ? -e[2 * i + 1] : e[2 * i]);   // cos, then sin
        }
    const long fsize = (long)(ctx->nx + 1) * (ctx->ny + 1) * (ctx->nz + 1);
    const size_t K = std::max(p.K, ctx->Hx), Y = std::max(Py2, ctx->Py2);
    void *oct = nullptr, *fg = nullptr, *a1 = nullptr, *a2 = nullptr, *a3 = nullptr, *tab = nullptr;
    auto cleanup = [&]() {
        for (void* q : {oct, fg, a1, a2, a3, tab}) cudaFree(q);
    };
    int rc = MM_OK;
    auto A = [&](void** q, size_t b) {
        if (rc == MM_OK) rc = dev_alloc(ctx, q, b);
    };
    A(&ctx->kern, 6 * (size_t)Pz2 * ctx->Py2 * ctx->Hs * elem(ctx));
    A(&oct, sizeof(double) * 6 * ctx->N);
    A(&fg, sizeof(double2) * fsize);
    A(&a1, sizeof(double) * (size_t)ctx->nz * ctx->ny * K);
    A(&a2, sizeof(double) * (size_t)ctx->nz * Y * K);
    A(&a3, sizeof(double) * (size_t)Pz2 * Y * K);
    A(&tab, sizeof(double) * t.size());
    if (rc == MM_OK && cudaMemcpy(tab, t.data(), sizeof(double) * t.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        rc = fail(ctx, MM_ERR_CUDA, "octant table copy failed");
    for (int c = 0; c < 6 && rc == MM_OK; ++c) {
        double* oc = (double*)oct + c * ctx->N;
        if ((rc = newell_component(ctx, c, nullptr, oc, fg))) break;
        const int odd[3] = {c == 3 || c == 4, c == 3 || c == 5, c == 4 || c == 5};
        const double sign = c >= 3 ? -1.0 : 1.0;
        const double* src[3] = {oc, (const double*)a1, (const double*)a2};
        double* dst[3] = {(double*)a1, (double*)a2, (double*)a3};
        for (int q = 0; q < sets; ++q) {
            const long O[3] = {(long)ctx->nz * ctx->ny, ctx->nz, 1}, I[3] = {1, m[q][0], (long)m[q][1] * m[q][0]};
            for (int a = 0; a < 3; ++a) {
                const long total = O[a] * m[q][a] * I[a];
                k_octant_axis<<<blocks(total), 256, 0, ctx->stream>>>(
                    src[a], dst[a], O[a], n[a], (int)I[a], m[q][a], len[q][a], odd[a],
                    (const double*)tab + off[q][a] + (odd[a] ? len[q][a] : 0));
            }
            if (q == 0) {
                const long total = (long)p.K * Pz2 * p.KQ;
                if (ctx->prec == MM_F64)
                    k_octant_place<double><<<blocks(total), 256, 0, ctx->stream>>>(
                        (const double*)a3, (double*)p.kern, c, p.K, Pz2, Py2, p.KQ, sign);
                else
                    k_octant_place<float><<<blocks(total), 256, 0, ctx->stream>>>((const double*)a3, (float*)p.kern, c,
                                                                                  p.K, Pz2, Py2, p.KQ, sign);
            } else {
                const long rows = (long)Pz2 * ctx->Py2, total = rows * ctx->Hs;
                if (ctx->prec == MM_F64)
                    k_octant_rows<double><<<blocks(total), 256, 0, ctx->stream>>>(
                        (const double*)a3, (double*)ctx->kern + c * total, ctx->Hx, ctx->Hs, rows, sign);
                else
                    k_octant_rows<float><<<blocks(total), 256, 0, ctx->stream>>>(
                        (const double*)a3, (float*)ctx->kern + c * total, ctx->Hx, ctx->Hs, rows, sign);
            }
            ctx->launches += 4;
        }
        if (cudaGetLastError() != cudaSuccess) rc = fail(ctx, MM_ERR_CUDA, "octant kernel launch failed");
    }
    cudaError_t e = cudaSuccess;
    if (rc == MM_OK)
        e = cudaMemcpyAsync(ctx->newell_host, oct, sizeof(double) * 6 * ctx->N, cudaMemcpyDeviceToHost, ctx->stream);
    const cudaError_t es = cudaStreamSynchronize(ctx->stream);
    if (rc == MM_OK && (e != cudaSuccess || es != cudaSuccess))
        rc = fail(ctx, MM_ERR_CUDA, "octant setup failed: %s", cudaGetErrorString(e != cudaSuccess ? e : es));
    cleanup();
    if (rc == MM_OK) ctx->kern_ready = true;
    return rc;
}

// float-float copies of the octant and the tables (MM_FFT_FF)
int plane_prepare_ff(mm_ctx* ctx) {
    PlanePlan& p = ctx->plane;
    if (p.kern_ff && p.tw_ff) return MM_OK;
    const long nk = kern_count(ctx), nt = tw_count(ctx);
    int rc;
    if (!p.kern_ff && (rc = dev_alloc(ctx, &p.kern_ff, nk * sizeof(ff)))) return rc;
    if (!p.tw_ff && (rc = dev_alloc(ctx, &p.tw_ff, nt * sizeof(ff)))) return rc;
    k_split<<<blocks(nk), 256, 0, ctx->stream>>>((const double*)p.kern, (ff*)p.kern_ff, nk);
    MM_LAUNCH_CHECK(ctx);
    k_split<<<blocks(nt), 256, 0, ctx->stream>>>((const double*)p.tw, (ff*)p.tw_ff, nt);
    MM_LAUNCH_CHECK(ctx);
    MM_CUDA_CHECK(ctx, cudaStreamSynchronize(ctx->stream));
    return MM_OK;
}

int plane_apply(mm_ctx* ctx, const void* m, void* H, bool unit) {
    const void* Ms = ctx->has_Ms_cell && !unit ? ctx->Ms_cell : nullptr;
    const double ms = unit ? 1.0 : ctx->Ms;
    if (ctx->prec == MM_F32)
        return plane_apply_f32(ctx, (const float*)m, (const float*)Ms, (float)ms, (float*)H);
    if (ctx->fft_mode == MM_FFT_FF)
        return plane_apply_ff(ctx, (const double*)m, (const double*)Ms, ms, (double*)H);
    return plane_apply_f64(ctx, (const double*)m, (const double*)Ms, ms, (double*)H);
}

// the two parts of a field evaluation before the fused kernel (FP32)
int plane_xfwd(mm_ctx* ctx, const void* m) {
    return plane_xfwd_f32(ctx, (const float*)m, ctx->has_Ms_cell ? (const float*)ctx->Ms_cell : nullptr, (float)ctx->Ms);
}
int plane_yzy(mm_ctx* ctx) { return plane_yzy_f32(ctx); }

}  // namespace mm
