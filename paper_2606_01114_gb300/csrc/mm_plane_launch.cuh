// Launchers of the plane-layout kernels: the length tables and one explicit
// instantiation point per element type (mm_plane_f32*.cu,
// mm_plane_f64*.cu).
#pragma once

#include <algorithm>
#include "mm_plane.cuh"

namespace mm {

// f(integral_constant L1, integral_constant L2) for the four-step split of
// length `len`; false when the length is not in the table.  Both factors are
// even (the zero half of the input is n1 >= L1/2, the dropped half of the
// output k2 >= L2/2).
template <typename F> bool with_length(int len, F&& f) {
#define MM_LEN(N, A, B) \
    case N: f(std::integral_constant<int, A>{}, std::integral_constant<int, B>{}); return true
    switch (len) {
        MM_LEN(4, 2, 2);
        MM_LEN(8, 4, 2);
        MM_LEN(16, 4, 4);
        MM_LEN(32, 8, 4);
        MM_LEN(64, 8, 8);
        MM_LEN(128, 16, 8);
        MM_LEN(256, 16, 16);
        MM_LEN(512, 32, 16);
        MM_LEN(1024, 32, 32);
        MM_LEN(40, 10, 4);
        MM_LEN(48, 12, 4);
        MM_LEN(80, 10, 8);
        MM_LEN(96, 12, 8);
        MM_LEN(160, 16, 10);
        MM_LEN(192, 16, 12);
        MM_LEN(320, 20, 16);
        MM_LEN(384, 24, 16);
        MM_LEN(640, 32, 20);
        MM_LEN(768, 32, 24);
        default: break;
    }
#undef MM_LEN
    return false;
}

// complex stride of a line of length P in the plane kernel's shared memory
inline int plane_line(int P) {
    int lp = 0;
    with_length(P, [&](auto A, auto B) { lp = plane_pitch(decltype(A)::value, decltype(B)::value); });
    return lp;
}

template <typename T>
int launch_px_fwd(mm_ctx* ctx, const T* in, const T* Ms, T ms, long ms_rows, PC<T>* out, long rows, const PC<T>* tw) {
    const PlanePlan& p = ctx->plane;
    int rc = MM_OK;
    KernelTimer kt(ctx, MM_K_XFWD);
    if (!with_length(p.L, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value, L = L1 * L2;
            if constexpr (L <= 512) {
                constexpr int BR = px_rows<T>(L);
                dep(k_px_fwd<T, L1, L2>, (unsigned)((rows + BR - 1) / BR), px_threads(BR, L1, L2), 0, ctx->stream)(
                    in, ctx->nx, Ms, ms, ms_rows, out, p.R, rows, tw + p.off_x4, tw + p.off_p);
            }
        }))
        rc = fail(ctx, MM_ERR_INVALID_ARG, "x length %d", p.L);
    if (rc) return rc;
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

template <typename T>
int launch_px_inv(mm_ctx* ctx, const PC<T>* in, T* out, long rows, T scale, const PC<T>* tw) {
    const PlanePlan& p = ctx->plane;
    int rc = MM_OK;
    KernelTimer kt(ctx, MM_K_XINV);
    if (!with_length(p.L, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value, L = L1 * L2;
            if constexpr (L <= 512) {
                constexpr int BR = px_rows<T>(L);
                dep(k_px_inv<T, L1, L2>, (unsigned)((rows + BR - 1) / BR), px_threads(BR, L1, L2), 0, ctx->stream)(
                    in, p.R, out, ctx->nx, rows, scale, tw + p.off_x4, tw + p.off_p);
            }
        }))
        rc = fail(ctx, MM_ERR_INVALID_ARG, "x length %d", p.L);
    if (rc) return rc;
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

template <typename T>
int launch_plane(mm_ctx* ctx, PC<T>* buf, const T* kern, const PC<T>* tw) {
    const PlanePlan& p = ctx->plane;
    int rc = MM_OK;
    KernelTimer kt(ctx, MM_K_ZCONV);
    if (!with_length(p.P, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value;
            // the fused level 2 holds 3 L2 complex values: single precision, L2 <= 16
            constexpr bool CANF = sizeof(T) == 4 && L2 <= 16;
            const bool fused = CANF && ctx->nz == 1;
            auto fn = fused ? k_plane<T, L1, L2, CANF> : k_plane<T, L1, L2, false>;
            const size_t smem = (size_t)3 * ctx->nz * plane_pitch(L1, L2) * sizeof(PC<T>);
            if ((rc = smem_opt_in(ctx, (const void*)fn, smem))) return;
            const int tasks = 3 * ctx->nz * L1;
            // Rounds of equal size within `cap` threads.  Planes that have an
            // SM each take up to 512 threads; of more planes, blocks of at
            // most 256 put two on an SM (at 128 registers), and smaller ones
            // where that takes every plane into one wave.  Demag, 384 threads
            // -> rule: 256x256x4 20.9 -> 19.1 us, 512x512x4 64.9 -> 61.4,
            // 256x256x8 33.6 -> 30.6, 300x300x2 21.8 -> 19.0 (96 threads: 20.8);
            // 64x512x8 (65 planes) 29.3 at 384, 35.9 at 192; 350x350x4 (385
            // planes, three blocks of 128 on an SM's 228 KB) 36.5 -> 34.9.
            auto even = [&](int cap) {
                const int rounds = (tasks + cap - 1) / cap;
                return ((tasks + rounds - 1) / rounds + 31) / 32 * 32;
            };
            int nt = even(sizeof(T) == 4 ? 512 : 256);
            if (sizeof(T) == 4 && p.K > kSMs) {
                nt = even(256);
                for (int cap : {256, 160, 128}) {
                    const int n = std::max(even(cap), std::min(128, nt));
                    const long fit = std::min<long>(65536 / (128 * n), (228 * 1024) / (long)(smem + 1024));
                    if (kSMs * fit >= p.K) {
                        nt = n;
                        break;
                    }
                }
            }
            dep(fn, (unsigned)p.K, nt, smem, ctx->stream)(buf, kern, ctx->nz, ctx->ny, p.R, p.KQ, tw + p.off_y4);
        }))
        rc = fail(ctx, MM_ERR_INVALID_ARG, "y length %d", p.P);
    if (rc) return rc;
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

template <typename T, int DIR>
int launch_py(mm_ctx* ctx, const PC<T>* in, PC<T>* out, const PC<T>* tw) {
    const PlanePlan& p = ctx->plane;
    int rc = MM_OK;
    KernelTimer kt(ctx, DIR < 0 ? MM_K_YFWD : MM_K_YINV);
    const int lines = 3 * ctx->nz;
    const long nlines = (long)p.K * lines, wide = (long)lines * p.P;
    if (!with_length(p.P, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value;
            auto fn = k_py<T, L1, L2, DIR>;
            const size_t smem = (size_t)kPyLines * plane_pitch(L1, L2) * sizeof(PC<T>);
            if ((rc = smem_opt_in(ctx, (const void*)fn, smem))) return;
            dep(fn, (unsigned)((nlines + kPyLines - 1) / kPyLines), (kPyLines * (L1 > L2 ? L1 : L2) + 31) / 32 * 32, smem, ctx->stream)(in, out, lines, nlines, ctx->ny, DIR < 0 ? p.R : wide, DIR < 0 ? wide : p.R,
                                                      tw + p.off_y4);
        }))
        rc = fail(ctx, MM_ERR_INVALID_ARG, "y length %d", p.P);
    if (rc) return rc;
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}

// the split of a z length: the middle level holds 3 L2 complex values
template <typename F> bool with_z_length(int len, F&& f) {
#define MM_LEN(N, A, B) \
    case N: f(std::integral_constant<int, A>{}, std::integral_constant<int, B>{}); return true
    switch (len) {
        MM_LEN(4, 2, 2);
        MM_LEN(8, 4, 2);
        MM_LEN(16, 4, 4);
        MM_LEN(32, 8, 4);
        MM_LEN(64, 8, 8);
        MM_LEN(128, 16, 8);
        MM_LEN(256, 32, 8);
        MM_LEN(512, 32, 16);
        MM_LEN(1024, 32, 32);
        default: return false;
    }
#undef MM_LEN
}

// B columns per block: 128-byte row segments for short lines, 64 bytes up to
// Pz = 512 (256^3, Pz = 512: 32-byte segments 1980-2230 us, 64-byte 950 us).
// NT threads: level 1 has 3 L2 B tasks, the middle level L1 B.  256^3: 384
// threads 952 us, 256 threads 1050 us (208 registers) or 1450 us (128, two
// blocks per SM, spills), 128 threads 1243 us; 256 x 256 x 32 (Pz = 64,
// whole field): 128 threads 194 us, 256 threads 234 us.  FP64 planes of two
// and four layers that take this pass (mm_plane.cu) have 3 to 6 values a
// column: 32 columns keep a block's warps full.
template <typename T, int L1, int L2, bool COLY, int B, int NT, int MINB>
int launch_zline_b(mm_ctx* ctx, PC<T>* buf, const T* kern, const ZLine& g, int nrows, const PC<T>* tw) {
    auto fn = k_zline<T, L1, L2, COLY, B, NT, MINB>;
    const size_t smem = zline_smem<T, L1, L2, B>();
    int rc = smem_opt_in(ctx, (const void*)fn, smem);
    if (rc) return rc;
    dim3 grid((unsigned)((g.ncol + B - 1) / B), (unsigned)nrows);
    dep(fn, grid, NT, smem, ctx->stream)(buf, kern, g, tw);
    MM_LAUNCH_CHECK(ctx);
    return MM_OK;
}
template <typename T, int L1, int L2, bool COLY>
int launch_zline_t(mm_ctx* ctx, PC<T>* buf, const T* kern, const ZLine& g, int nrows, const PC<T>* tw) {
    constexpr int PZ = L1 * L2, CS = (int)sizeof(PC<T>);
    if constexpr (zline_split<T>(PZ)) {
        // one column a block while four of them would leave SMs idle (5x2x512:
        // 264 us a field with four, 18 blocks; 97 with one)
        if ((long)g.ncol * nrows <= 4 * kSMs) return launch_zline_b<T, L1, L2, COLY, 1, 96, 1>(ctx, buf, kern, g, nrows, tw);
        return launch_zline_b<T, L1, L2, COLY, 4, 384, 1>(ctx, buf, kern, g, nrows, tw);
    } else {
        constexpr int B = PZ <= 8 ? 32 : PZ <= 64 ? 128 / CS : PZ <= 512 ? 64 / CS : 32 / CS;
        constexpr int NT = sizeof(T) == 8 ? (PZ == 512 ? 192 : 128) : PZ == 64 ? 128 : PZ == 256 ? 256 : PZ >= 512 ? 384 : 192;
        constexpr int MINB = sizeof(T) == 8 ? 1 : PZ <= 32 ? 4 : PZ == 64 ? 4 : PZ == 128 ? 3 : PZ == 256 ? 2 : 1;
        return launch_zline_b<T, L1, L2, COLY, B, NT, MINB>(ctx, buf, kern, g, nrows, tw);
    }
}

template <typename T, bool COLY>
int launch_zline(mm_ctx* ctx, int Pz, PC<T>* buf, const T* kern, const ZLine& g, int nrows, const PC<T>* tw) {
    KernelTimer kt(ctx, MM_K_ZCONV);
    int rc = MM_OK;
    if (!with_z_length(Pz, [&](auto A, auto B) {
            constexpr int L1 = decltype(A)::value, L2 = decltype(B)::value;
            // the lengths that reach this pass: FP32 planes from 16 on, kx columns from 64 on
            if constexpr (sizeof(T) == 8 || L1 * L2 >= (COLY ? 16 : 64))
                rc = launch_zline_t<T, L1, L2, COLY>(ctx, buf, kern, g, nrows, tw);
            else
                rc = fail(ctx, MM_ERR_INVALID_ARG, "z length %d", Pz);
        }))
        return fail(ctx, MM_ERR_INVALID_ARG, "z length %d", Pz);
    return rc;
}

}  // namespace mm
