// Runge-Kutta tableaux and the error maximum, shared by the stage kernels
// (mm_llg.cu) and the fused stage of the plane layout (mm_plane_step.cu).
#pragma once

#include "mm_internal.cuh"

namespace mm {

// classic RK4 and Fehlberg's RKF45 (4th-order weights propagated)
__host__ __device__ constexpr double rk_a(int method, int i, int j) {
    if (method == MM_RK4) {
        if (i == 1 && j == 0) return 0.5;
        if (i == 2 && j == 1) return 0.5;
        if (i == 3 && j == 2) return 1.0;
        return 0.0;
    }
    switch (i * 8 + j) {
        case 1 * 8 + 0: return 1.0 / 4.0;
        case 2 * 8 + 0: return 3.0 / 32.0;
        case 2 * 8 + 1: return 9.0 / 32.0;
        case 3 * 8 + 0: return 1932.0 / 2197.0;
        case 3 * 8 + 1: return -7200.0 / 2197.0;
        case 3 * 8 + 2: return 7296.0 / 2197.0;
        case 4 * 8 + 0: return 439.0 / 216.0;
        case 4 * 8 + 1: return -8.0;
        case 4 * 8 + 2: return 3680.0 / 513.0;
        case 4 * 8 + 3: return -845.0 / 4104.0;
        case 5 * 8 + 0: return -8.0 / 27.0;
        case 5 * 8 + 1: return 2.0;
        case 5 * 8 + 2: return -3544.0 / 2565.0;
        case 5 * 8 + 3: return 1859.0 / 4104.0;
        case 5 * 8 + 4: return -11.0 / 40.0;
        default: return 0.0;
    }
}
__host__ __device__ constexpr double rk_b(int method, int j) {
    if (method == MM_RK4) {
        return j == 0 ? 1.0 / 6.0 : j == 1 ? 1.0 / 3.0 : j == 2 ? 1.0 / 3.0 : j == 3 ? 1.0 / 6.0 : 0.0;
    }
    return j == 0 ? 25.0 / 216.0 : j == 2 ? 1408.0 / 2565.0 : j == 3 ? 2197.0 / 4104.0 : j == 4 ? -1.0 / 5.0 : 0.0;
}
// b5 - b4 (RKF45 error weights)
__host__ __device__ constexpr double rk_e(int method, int j) {
    if (method == MM_RK4) return 0.0;
    constexpr double b5[6] = {16.0 / 135.0, 0.0, 6656.0 / 12825.0, 28561.0 / 56430.0, -9.0 / 50.0, 2.0 / 55.0};
    return b5[j] - rk_b(method, j);
}
__host__ __device__ constexpr int rk_stages(int method) { return method == MM_RK4 ? 4 : 6; }

// Block-wide max of a non-negative double, then one atomicMax of its bits.
// Non-negative doubles order like their bit patterns, so the maxima are
// integer reductions and none of it runs on the FP64 pipe.
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
    return ((unsigned long long)mh << 32) | ml;
}
__device__ __forceinline__ void block_max_atomic(double v, unsigned long long* target) {
    __shared__ unsigned long long red[32];
    unsigned long long u = warp_max_bits((unsigned long long)__double_as_longlong(v));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = u;
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        u = warp_max_bits(lane < nw ? red[lane] : 0ull);
        if (lane == 0 && u != 0ull) atomicMax(target, u);
    }
}

// the slope arrays k[0..5]
template <typename T> struct KPtrs {
    T* k[6];
};
template <typename T> KPtrs<T> slopes(const mm_ctx* ctx) {
    KPtrs<T> kb;
    for (int s = 0; s < 6; ++s) kb.k[s] = (T*)ctx->k[s];
    return kb;
}

}  // namespace mm
