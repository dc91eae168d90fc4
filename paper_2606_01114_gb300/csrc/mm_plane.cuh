// Demag convolution in the plane layout: spectra stored [kx][component][z][y]
// (y fastest), one contiguous plane per kept x frequency.
//
// Three kernels take a field evaluation:
//   k_px_fwd   rows of M: real-to-complex x transform, written transposed
//              into the planes (B consecutive rows of the block land in one
//              32- or 64-byte segment of every plane);
//   k_plane    one block per plane, everything on chip: y forward, z forward,
//              the 3x3 tensor product, z inverse, y inverse, in place;
//   k_px_inv   planes back to real rows of H.
// Planes too large for one block's shared memory (or nz > 8), and FP64 planes
// too few to fill the SMs, run y forward, z product and y inverse as three
// kernels in the same layout (k_py, k_zline).
//
// Lengths.  The convolution is linear, so the padded length P may be any
// length >= 2n: it is the next of 8 (x: 2 L, L = 4), 16, 32 and {4, 5, 6} 2^k
// from 32 on, not 2n itself.  Meshes whose sides are not powers of two
// therefore run the same four-step transforms as the others and need no
// chirp-z convolution of length >= 4n - 1.  The padding is at most a third more
// above 32 (2n = 770 takes 1024); lengths 12, 20 and 24 below it were slower
// than the 16 and 32 that hold them (FP64 12x11x16, P = 24: 33 us against 28).
//
// Every transform is a four-step L = L1 x L2 with both levels in registers:
// level 1 (thread t < L2) DFT over n1 of x[t + L2 n1], twiddle w^(t k1);
// level 2 (thread k1 < L1) DFT over n2, X[k1 + L1 k2].  Element (k1, t) sits
// at k1 (L2 + 1) + t of its line: both levels read and write the same places
// (no barrier between a level's loads and stores), and the odd pitch keeps
// the row accesses of level 2 off each other's banks.  The twiddles w^(t k1)
// come from tables laid out [k1][t] and, behind it, [t][k1]: every load of a
// level sits at a compile-time offset from one pointer, and the lanes of a
// warp (consecutive t, or consecutive k1) read consecutive values.
#pragma once

#include "mm_ff.cuh"
#include "mm_regfft.cuh"

namespace mm {

template <typename T> using PC = typename cx<T>::type;

constexpr int plane_pitch(int L1, int L2) { return L1 * (L2 + 1); }

// rows per block of the x passes
template <typename T> constexpr int px_rows(int L) { return L <= 64 ? 8 : 4; }
constexpr int px_threads(int B, int L1, int L2) { return (B * (L1 > L2 ? L1 : L2) + 31) / 32 * 32; }

// ---------------------------------------------------------------- x forward
template <typename T, int L1, int L2>
__global__ void __launch_bounds__(px_threads(px_rows<T>(L1 * L2), L1, L2))
    k_px_fwd(const T* __restrict__ in, int nx, const T* __restrict__ Ms, T ms, long ms_rows, PC<T>* __restrict__ out,
             long R, long rows, const PC<T>* __restrict__ twL, const PC<T>* __restrict__ twP) {
    dep_wait();
    using C = PC<T>;
    constexpr int L = L1 * L2, B = px_rows<T>(L), LP = plane_pitch(L1, L2) + (sizeof(T) == 4 ? 4 : 2);
    __shared__ C Sm[B * LP];
    const int tid = threadIdx.x;
    const long r0 = (long)blockIdx.x * B;
    if (tid < B * L2) {
        const int t = tid % L2, b = tid / L2;
        const long r = r0 + b;
        const bool act = r < rows;
        const T* row = in + (act ? r : 0) * nx;
        const T* mrow = Ms ? Ms + (long)((unsigned)(act ? r : 0) % (unsigned)ms_rows) * nx : nullptr;
        // pairs in one access where every row starts on a pair boundary (the
        // library's own Ms array always does)
        const bool even = nx % 2 == 0 && reinterpret_cast<uintptr_t>(in) % (2 * sizeof(T)) == 0;
        C v[L1], w[L1 / 2];
#pragma unroll
        for (int n1 = 0; n1 < L1 / 2; ++n1) {
            const int x = 2 * (t + L2 * n1);
            v[n1] = cmk<C>((T)0, (T)0);
            w[n1] = cmk<C>(ms, ms);
            if (act && x < nx) {
                if (even) {
                    v[n1] = *reinterpret_cast<const C*>(row + x);
                    if (mrow) w[n1] = *reinterpret_cast<const C*>(mrow + x);
                } else {
                    const bool two = x + 1 < nx;
                    v[n1] = cmk<C>(row[x], two ? row[x + 1] : (T)0);
                    if (mrow) w[n1] = cmk<C>(mrow[x], two ? mrow[x + 1] : (T)0);
                }
            }
        }
#pragma unroll
        for (int n1 = 0; n1 < L1 / 2; ++n1) v[n1] = cmk<C>(v[n1].x * w[n1].x, v[n1].y * w[n1].y);
        const C* tq = twL + t;
        dif<L1, -1, true>(v);
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) {
            C y = v[dif_pos<L1>(k1)];
            if (k1 > 0) y = cmul(y, tq[k1 * L2]);
            Sm[b * LP + k1 * (L2 + 1) + t] = y;
        }
    }
    __syncthreads();
    if (tid < B * L1) {
        const int k1 = tid % L1, b = tid / L1;
        C* s = Sm + b * LP + k1 * (L2 + 1);
        C u[L2];
#pragma unroll
        for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2];
        dif<L2, -1, false>(u);
#pragma unroll
        for (int k2 = 0; k2 < L2; ++k2) s[k2] = u[dif_pos<L2>(k2)];
    }
    __syncthreads();
    // X_k = E - i w^k D and X_(L-k) = conj(E + i w^k D) from Z_k, Z_(L-k)
    const T half = (T)0.5;
    for (int idx = tid; idx < B * (L / 2 + 1); idx += blockDim.x) {
        const int b = idx % B, k = idx / B;
        const long r = r0 + b;
        if (r >= rows) continue;
        const int kc = k == 0 ? 0 : L - k;
        const C zk = Sm[b * LP + (k % L1) * (L2 + 1) + k / L1];
        const C zc = cconj(Sm[b * LP + (kc % L1) * (L2 + 1) + kc / L1]);
        const C e = cscale(cadd(zk, zc), half);
        const C wd = cmul(twP[k], cscale(csub(zk, zc), half));
        out[(long)k * R + r] = cmk<C>(e.x + wd.y, e.y - wd.x);
        if (2 * k != L) out[(long)(L - k) * R + r] = cmk<C>(e.x - wd.y, -(e.y + wd.x));
    }
}

// ---------------------------------------------------------------- x inverse
template <typename T, int L1, int L2>
__global__ void __launch_bounds__(px_threads(px_rows<T>(L1 * L2), L1, L2))
    k_px_inv(const PC<T>* __restrict__ in, long R, T* __restrict__ out, int nx, long rows, T scale,
             const PC<T>* __restrict__ twL, const PC<T>* __restrict__ twP) {
    dep_wait();
    using C = PC<T>;
    constexpr int L = L1 * L2, B = px_rows<T>(L), LP = plane_pitch(L1, L2) + (sizeof(T) == 4 ? 4 : 2);
    __shared__ C Sm[B * LP];
    const int tid = threadIdx.x;
    const long r0 = (long)blockIdx.x * B;
    const T half = (T)0.5;
    for (int idx = tid; idx < B * (L / 2 + 1); idx += blockDim.x) {
        const int b = idx % B, k = idx / B;
        const long r = r0 + b;
        C xk = cmk<C>((T)0, (T)0), xl = xk;
        if (r < rows) {
            xk = in[(long)k * R + r];
            xl = cconj(in[(long)(L - k) * R + r]);
        }
        const C e = cscale(cadd(xk, xl), half);
        const C o = cmul(cscale(csub(xk, xl), half), cconj(twP[k]));
        Sm[b * LP + (k / L2) * (L2 + 1) + k % L2] = cmk<C>(e.x - o.y, e.y + o.x);          // E + i O
        const int kc = L - k;
        if (k > 0 && kc != k) Sm[b * LP + (kc / L2) * (L2 + 1) + kc % L2] = cmk<C>(e.x + o.y, o.x - e.y);
    }
    __syncthreads();
    if (tid < B * L2) {
        const int t = tid % L2, b = tid / L2;
        C* s = Sm + b * LP + t;
        C v[L1];
#pragma unroll
        for (int n1 = 0; n1 < L1; ++n1) v[n1] = s[n1 * (L2 + 1)];
        const C* tq = twL + t;
        dif<L1, +1, false>(v);
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) {
            C y = v[dif_pos<L1>(k1)];
            if (k1 > 0) y = cmul(y, cconj(tq[k1 * L2]));
            s[k1 * (L2 + 1)] = y;
        }
    }
    __syncthreads();
    if (tid < B * L1) {
        const int k1 = tid % L1, b = tid / L1;
        const C* s = Sm + b * LP + k1 * (L2 + 1);
        C u[L2];
#pragma unroll
        for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2];
        dif<L2, +1, false>(u);
        const long r = r0 + b;
        if (r < rows) {
            T* row = out + r * nx;
            const bool even = nx % 2 == 0 && reinterpret_cast<uintptr_t>(out) % (2 * sizeof(T)) == 0;
#pragma unroll
            for (int k2 = 0; k2 < L2 / 2; ++k2) {
                const C z = u[dif_pos<L2>(k2)];
                const int x = 2 * (k1 + L1 * k2);
                const T a = z.x * scale, c = z.y * scale;
                if (x + 1 < nx) {
                    if (even) {
                        *reinterpret_cast<C*>(row + x) = cmk<C>(a, c);
                    } else {
                        row[x] = a;
                        row[x + 1] = c;
                    }
                } else if (x < nx) {
                    row[x] = a;
                }
            }
        }
    }
}

// ------------------------------------------------------------- the product
// H^ = -N^ M^ at one k point: n = the six real octant values with the signs
// of the odd components already applied (xy, xz, yz)
template <typename T, typename C>
__device__ __forceinline__ void tensor_product(C& mx, C& my, C& mz, T xx, T yy, T zz, T xy, T xz, T yz) {
    const C a = mx, b = my, c = mz;
    mx = cmk<C>(-(xx * a.x + xy * b.x + xz * c.x), -(xx * a.y + xy * b.y + xz * c.y));
    my = cmk<C>(-(xy * a.x + yy * b.x + yz * c.x), -(xy * a.y + yy * b.y + yz * c.y));
    mz = cmk<C>(-(xz * a.x + yz * b.x + zz * c.x), -(xz * a.y + yz * b.y + zz * c.y));
}

// z transform, product and inverse of one (kx, ky) column of the plane: the
// 3 NZ values s[(c NZ + z) LP], octant values kb[(comp PZ2 + kz) KQ]; sy = -1
// where ky is in the upper half (xy and yz are odd in ky, xz and yz in kz)
template <typename T, int PZ>
__device__ __forceinline__ void z_point(PC<T>* s, int LP, const T* __restrict__ kb, int KQ, bool yodd) {
    using C = PC<T>;
    constexpr int NZ = PZ > 1 ? PZ / 2 : 1, PZ2 = PZ / 2 + 1;
    C v[3][PZ];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int z = 0; z < NZ; ++z) v[c][z] = s[(c * NZ + z) * LP];
        dif<PZ, -1, (PZ > 1)>(v[c]);
    }
#pragma unroll
    for (int kz = 0; kz < PZ2; ++kz) {
        const T xx = kb[(0 * PZ2 + kz) * KQ], yy = kb[(1 * PZ2 + kz) * KQ], zz = kb[(2 * PZ2 + kz) * KQ];
        T xy = kb[(3 * PZ2 + kz) * KQ], yz = kb[(5 * PZ2 + kz) * KQ];
        const T xz = kb[(4 * PZ2 + kz) * KQ];
        if (yodd) {
            xy = -xy;
            yz = -yz;
        }
        const int q = dif_pos<PZ>(kz);
        tensor_product<T>(v[0][q], v[1][q], v[2][q], xx, yy, zz, xy, xz, yz);
        if (kz > 0 && 2 * kz < PZ) {
            const int qc = dif_pos<PZ>(PZ - kz);
            tensor_product<T>(v[0][qc], v[1][qc], v[2][qc], xx, yy, zz, xy, -xz, -yz);
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        C u[PZ];
#pragma unroll
        for (int kz = 0; kz < PZ; ++kz) u[kz] = v[c][dif_pos<PZ>(kz)];
        dif<PZ, +1, false>(u);
#pragma unroll
        for (int z = 0; z < NZ; ++z) s[(c * NZ + z) * LP] = u[dif_pos<PZ>(z)];
    }
}

// ------------------------------------------------------------------ plane
// One block per kx.  FUSED (nz = 1): level 2 holds all three components of a
// row k1, so its DFT, the product and the inverse DFT need no shared memory
// in between.
template <typename T, int L1, int L2, bool FUSED>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 512 : 256)
    k_plane(PC<T>* __restrict__ buf, const T* __restrict__ kern, int nz, int ny, long R, int KQ,
            const PC<T>* __restrict__ tw) {
    dep_wait();
    using C = PC<T>;
    constexpr int P = L1 * L2, LP = plane_pitch(L1, L2);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* Sm = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x, nt = blockDim.x;
    C* base = buf + (long)blockIdx.x * R;
    const int lines = 3 * nz;
    const int PZ2 = nz > 1 ? nz + 1 : 1;
    const T* kp = kern + (long)blockIdx.x * 6 * PZ2 * KQ;
    for (int i = tid; i < lines * L2; i += nt) {
        const int t = i % L2, line = i / L2;
        const C* ib = base + (long)line * ny;
        C v[L1];
#pragma unroll
        for (int n1 = 0; n1 < L1 / 2; ++n1) {
            const int y = t + L2 * n1;
            v[n1] = y < ny ? ib[y] : cmk<C>((T)0, (T)0);
        }
        dif<L1, -1, true>(v);
        C* s = Sm + line * LP + t;
        const C* tq = tw + t;
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) {
            C y = v[dif_pos<L1>(k1)];
            if (k1 > 0) y = cmul(y, tq[k1 * L2]);
            s[k1 * (L2 + 1)] = y;
        }
    }
    __syncthreads();
    if constexpr (FUSED) {
        for (int k1 = tid; k1 < L1; k1 += nt) {
            C* s = Sm + k1 * (L2 + 1);
            const C* tq = tw + P + k1;
            C u[3][L2];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
                for (int n2 = 0; n2 < L2; ++n2) u[c][n2] = s[c * LP + n2];
                dif<L2, -1, false>(u[c]);
            }
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) {
                const int ky = k1 + L1 * k2;
                const bool yodd = 2 * ky > P;
                const T* kb = kp + (yodd ? P - ky : ky);
                const T xx = kb[0], yy = kb[KQ], zz = kb[2 * KQ];
                T xy = kb[3 * KQ], yz = kb[5 * KQ];
                const T xz = kb[4 * KQ];
                if (yodd) {
                    xy = -xy;
                    yz = -yz;
                }
                const int q = dif_pos<L2>(k2);
                tensor_product<T>(u[0][q], u[1][q], u[2][q], xx, yy, zz, xy, xz, yz);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                C w[L2];
#pragma unroll
                for (int k2 = 0; k2 < L2; ++k2) w[k2] = u[c][dif_pos<L2>(k2)];
                dif<L2, +1, false>(w);
#pragma unroll
                for (int t = 0; t < L2; ++t) {
                    C y = w[dif_pos<L2>(t)];
                    if (t > 0) y = cmul(y, cconj(tq[t * L1]));
                    s[c * LP + t] = y;
                }
            }
        }
    } else {
        for (int i = tid; i < lines * L1; i += nt) {
            C* s = Sm + (i / L1) * LP + (i % L1) * (L2 + 1);
            C u[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2];
            dif<L2, -1, false>(u);
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) s[k2] = u[dif_pos<L2>(k2)];
        }
        __syncthreads();
        for (int ky = tid; ky < P; ky += nt) {
            C* s = Sm + (ky % L1) * (L2 + 1) + ky / L1;
            const bool yodd = 2 * ky > P;
            const T* kb = kp + (yodd ? P - ky : ky);
            switch (nz) {
                case 1: z_point<T, 1>(s, LP, kb, KQ, yodd); break;
                case 2: z_point<T, 4>(s, LP, kb, KQ, yodd); break;
                case 4: z_point<T, 8>(s, LP, kb, KQ, yodd); break;
                default:
                    if constexpr (sizeof(T) == 4) z_point<T, 16>(s, LP, kb, KQ, yodd);
                    break;
            }
        }
        __syncthreads();
        for (int i = tid; i < lines * L1; i += nt) {
            const int k1 = i % L1;
            C* s = Sm + (i / L1) * LP + k1 * (L2 + 1);
            const C* tq = tw + P + k1;
            C u[L2];
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) u[k2] = s[k2];
            dif<L2, +1, false>(u);
#pragma unroll
            for (int t = 0; t < L2; ++t) {
                C y = u[dif_pos<L2>(t)];
                if (t > 0) y = cmul(y, cconj(tq[t * L1]));
                s[t] = y;
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < lines * L2; i += nt) {
        const int t = i % L2, line = i / L2;
        const C* s = Sm + line * LP + t;
        C v[L1];
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) v[k1] = s[k1 * (L2 + 1)];
        dif<L1, +1, false>(v);
        C* ob = base + (long)line * ny;
#pragma unroll
        for (int n1 = 0; n1 < L1 / 2; ++n1) {
            const int y = t + L2 * n1;
            if (y < ny) ob[y] = v[dif_pos<L1>(n1)];
        }
    }
}

// ------------------------------------------------- y lines (large planes)
// DIR -1: ny values of a line of `in` (plane stride in_plane, line stride ny)
// -> P values of `out` (plane stride 3 nz P); DIR +1 the reverse, keeping ny.
// Line q of the grid: plane q / lines, line q % lines.
constexpr int kPyLines = 4;
template <typename T, int L1, int L2, int DIR>
__global__ void __launch_bounds__((kPyLines * (L1 > L2 ? L1 : L2) + 31) / 32 * 32)
    k_py(const PC<T>* __restrict__ in, PC<T>* __restrict__ out, int lines, long nlines, int ny, long in_plane,
         long out_plane, const PC<T>* __restrict__ tw) {
    dep_wait();
    using C = PC<T>;
    constexpr int P = L1 * L2, LP = plane_pitch(L1, L2), B = kPyLines;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* Sm = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x;
    const long q0 = (long)blockIdx.x * B;
    if (tid < B * L2) {
        const int t = tid % L2, b = tid / L2;
        const long q = q0 + b;
        if (q < nlines) {
            const C* ib = in + (q / lines) * in_plane + (q % lines) * (long)(DIR < 0 ? ny : P);
            C v[L1];
            constexpr int NI = DIR < 0 ? L1 / 2 : L1;
#pragma unroll
            for (int n1 = 0; n1 < NI; ++n1) {
                const int y = t + L2 * n1;
                v[n1] = (DIR > 0 || y < ny) ? ib[y] : cmk<C>((T)0, (T)0);
            }
            dif<L1, DIR, (DIR < 0)>(v);
            C* s = Sm + b * LP + t;
            const C* tq = tw + t;
#pragma unroll
            for (int k1 = 0; k1 < L1; ++k1) {
                C y = v[dif_pos<L1>(k1)];
                if (k1 > 0) {
                    C w = tq[k1 * L2];
                    if (DIR > 0) w = cconj(w);
                    y = cmul(y, w);
                }
                s[k1 * (L2 + 1)] = y;
            }
        }
    }
    __syncthreads();
    if (tid < B * L1) {
        const int k1 = tid % L1, b = tid / L1;
        const long q = q0 + b;
        if (q < nlines) {
            const C* s = Sm + b * LP + k1 * (L2 + 1);
            C u[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2];
            dif<L2, DIR, false>(u);
            C* ob = out + (q / lines) * out_plane + (q % lines) * (long)(DIR < 0 ? P : ny);
            constexpr int NO = DIR < 0 ? L2 : L2 / 2;
#pragma unroll
            for (int k2 = 0; k2 < NO; ++k2) {
                const int y = k1 + L1 * k2;
                if (DIR < 0 || y < ny) ob[y] = u[dif_pos<L2>(k2)];
            }
        }
    }
}

// -------------------------------------------------------------- z columns
// z forward, product, z inverse of B adjacent columns (innermost index of
// the layout), in place.  Element (c, z, col) of block row `row` at
// buf + row * row_s + c * c_s + z * z_s + col; octant value (comp, kz) of
// column col at kern + krow(row) + comp * kc_s + kz * kz_s + kcol.
// COLY (plane layout): row = kx, columns = ky, kcol = min(ky, P - ky) with
// the sign of the columns above P/2.  Otherwise row = ky (mirrored the same
// way), columns = kx.
struct ZLine {
    long row_s, c_s, z_s, k_row, kc_s, kz_s;
    int nz, ncol, P;      // P: length of the mirrored axis (y)
};

// The tile's octant values are copied into shared memory by asynchronous
// copies that land while level 1 runs: read from global memory they sat on
// the critical path of the middle level (6 L2 dependent loads per thread).
template <typename T> __device__ __forceinline__ void cp_async_value(T* smem, const T* gmem) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(a), "l"(gmem), "n"(sizeof(T)) : "memory");
}
// FP64 at Pz = 1024: three components of 32 values are 384 registers, which
// spilled (12x12x512 477 us a field).  The middle level then goes one component
// at a time, with the product between two barriers, and the octant is read from
// global memory, so that four columns fit an SM (342; 60x60x512 6781 -> 4856).
template <typename T> constexpr bool zline_split(int PZ) { return std::is_same<T, double>::value && PZ == 1024; }
template <typename T, int L1, int L2, int B> constexpr size_t zline_smem() {
    return (size_t)3 * L1 * (L2 + 1) * B * sizeof(PC<T>) +
           (zline_split<T>(L1 * L2) ? 0 : (size_t)6 * (L1 * L2 / 2 + 1) * B * sizeof(T));
}

template <typename T, int L1, int L2, bool COLY, int B, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_zline(PC<T>* __restrict__ buf, const T* __restrict__ kern, ZLine g, const PC<T>* __restrict__ tw) {
    dep_wait();
    using C = PC<T>;
    constexpr int PZ = L1 * L2, PZ2 = PZ / 2 + 1, LQ = L2 + 1, CP = L1 * LQ * B;   // component pitch
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* Sm = reinterpret_cast<C*>(smem_raw);                 // [3][L1][L2 + 1][B]
    T* Kn = reinterpret_cast<T*>(Sm + 3 * CP);              // [6][PZ2][B]
    const int tid = threadIdx.x;
    const int col0 = blockIdx.x * B;
    int row = blockIdx.y;
    int krow = row;
    bool rodd = false;
    if (!COLY) {
        // rows 0, P/2, 1, P-1, 2, P-2, ...: the two rows of an octant row run
        // back to back, the second one reads it from L2
        row = row == 0 ? 0 : row == 1 ? (g.P >> 1) : ((row & 1) ? g.P - (row >> 1) : (row >> 1));
        rodd = 2 * row > g.P;
        krow = rodd ? g.P - row : row;
    }
    C* base = buf + (long)row * g.row_s + col0;
    const T* kbase = kern + (long)krow * g.k_row;
    constexpr bool SPLIT = zline_split<T>(PZ);
    auto octant_col = [&](int b) {
        const int col = col0 + b < g.ncol ? col0 + b : g.ncol - 1;
        return COLY && 2 * col > g.P ? g.P - col : col;
    };
    if constexpr (!SPLIT) {
        for (int i = tid; i < 6 * PZ2 * B; i += NT) {
            const int b = i % B, ck = i / B, kz = ck % PZ2, c = ck / PZ2;
            cp_async_value(Kn + i, kbase + c * g.kc_s + kz * g.kz_s + octant_col(b));
        }
    }
#pragma unroll 1
    for (int i = tid; i < 3 * L2 * B; i += NT) {
        const int b = i % B, ct = i / B, t = ct % L2, c = ct / L2;
        C* s = Sm + c * CP + t * B + b;
        const C* tq = tw + t;
        const C* p = base + c * g.c_s + b;
        const bool act = col0 + b < g.ncol;
        C v[L1];
#pragma unroll
        for (int n1 = 0; n1 < L1 / 2; ++n1) v[n1] = act ? p[(t + L2 * n1) * g.z_s] : cmk<C>((T)0, (T)0);
        dif<L1, -1, true>(v);
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) {
            C y = v[dif_pos<L1>(k1)];
            if (k1 > 0) y = cmul(y, tq[k1 * L2]);
            s[k1 * LQ * B] = y;
        }
    }
    if constexpr (!SPLIT) {
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    __syncthreads();
    if constexpr (SPLIT) {
#pragma unroll 1
        for (int i = tid; i < 3 * L1 * B; i += NT) {
            const int b = i % B, ck = i / B, k1 = ck % L1;
            C* s = Sm + (ck / L1) * CP + k1 * LQ * B + b;
            C u[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2 * B];
            dif<L2, -1, false>(u);
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) s[k2 * B] = u[dif_pos<L2>(k2)];
        }
        __syncthreads();
#pragma unroll 2
        for (int i = tid; i < PZ * B; i += NT) {
            const int b = i % B, kz = i / B, k2 = kz / L1, k1 = kz - k2 * L1;
            const bool yodd = COLY ? 2 * (col0 + b) > g.P : rodd, zodd = 2 * kz > PZ;
            const T* kk = kbase + (zodd ? PZ - kz : kz) * g.kz_s + octant_col(b);
            const T xx = kk[0], yy = kk[g.kc_s], zz = kk[2 * g.kc_s];
            T xy = kk[3 * g.kc_s], xz = kk[4 * g.kc_s], yz = kk[5 * g.kc_s];
            if (yodd) xy = -xy;
            if (zodd) xz = -xz;
            if (yodd != zodd) yz = -yz;
            C* s = Sm + (k1 * LQ + k2) * B + b;
            tensor_product<T>(s[0], s[CP], s[2 * CP], xx, yy, zz, xy, xz, yz);
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < 3 * L1 * B; i += NT) {
            const int b = i % B, ck = i / B, k1 = ck % L1;
            C* s = Sm + (ck / L1) * CP + k1 * LQ * B + b;
            const C* tq = tw + PZ + k1;
            C w[L2];
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) w[k2] = s[k2 * B];
            dif<L2, +1, false>(w);
#pragma unroll
            for (int t = 0; t < L2; ++t) {
                C y = w[dif_pos<L2>(t)];
                if (t > 0) y = cmul(y, cconj(tq[t * L1]));
                s[t * B] = y;
            }
        }
    } else {
#pragma unroll 1
        for (int i = tid; i < L1 * B; i += NT) {
            const int b = i % B, k1 = i / B;
            const bool yodd = COLY ? 2 * (col0 + b) > g.P : rodd;
            C* s = Sm + k1 * LQ * B + b;
            const C* tq = tw + PZ + k1;
            C u[3][L2];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
                for (int n2 = 0; n2 < L2; ++n2) u[c][n2] = s[c * CP + n2 * B];
                dif<L2, -1, false>(u[c]);
            }
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) {
                const int kz = k1 + L1 * k2;
                const bool zodd = 2 * kz > PZ;
                const T* kk = Kn + (zodd ? PZ - kz : kz) * B + b;
                const T xx = kk[0], yy = kk[PZ2 * B], zz = kk[2 * PZ2 * B];
                T xy = kk[3 * PZ2 * B], xz = kk[4 * PZ2 * B], yz = kk[5 * PZ2 * B];
                if (yodd) xy = -xy;
                if (zodd) xz = -xz;
                if (yodd != zodd) yz = -yz;
                const int q = dif_pos<L2>(k2);
                tensor_product<T>(u[0][q], u[1][q], u[2][q], xx, yy, zz, xy, xz, yz);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                C w[L2];
#pragma unroll
                for (int k2 = 0; k2 < L2; ++k2) w[k2] = u[c][dif_pos<L2>(k2)];
                dif<L2, +1, false>(w);
#pragma unroll
                for (int t = 0; t < L2; ++t) {
                    C y = w[dif_pos<L2>(t)];
                    if (t > 0) y = cmul(y, cconj(tq[t * L1]));
                    s[c * CP + t * B] = y;
                }
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < 3 * L2 * B; i += NT) {
        const int b = i % B, ct = i / B, t = ct % L2, c = ct / L2;
        const C* s = Sm + c * CP + t * B + b;
        C v[L1];
#pragma unroll
        for (int k1 = 0; k1 < L1; ++k1) v[k1] = s[k1 * LQ * B];
        dif<L1, +1, false>(v);
        C* p = base + c * g.c_s + b;
        if (col0 + b < g.ncol) {
#pragma unroll
            for (int n1 = 0; n1 < L1 / 2; ++n1) p[(t + L2 * n1) * g.z_s] = v[dif_pos<L1>(n1)];
        }
    }
}

}  // namespace mm
