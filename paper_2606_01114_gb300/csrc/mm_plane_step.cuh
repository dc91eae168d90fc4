// x inverse, local fields and Runge-Kutta stage, x forward in one kernel
// (plane layout, FP32).
//
// A stage of a small or middling mesh was four dependent kernels (x forward,
// plane, x inverse, stage) of 2 to 10 us each, most of it launch gap, ramp and
// tail.  The inverse x transform of a cell row needs only that row of the
// planes, the stage needs the row's field and m_in around it, and the next
// evaluation's x forward needs the row's new state: one block takes B cell rows
// (all three components) through all of it.  The planes are updated in place
// (a block reads and writes its own rows), and the demag field stays in shared
// memory.
#pragma once

#include "mm_fields.cuh"
#include "mm_plane.cuh"
#include "mm_rk.cuh"

namespace mm {

// one Runge-Kutta stage, by value: coefficients of the next trial state, or of
// the new state and its error after the last stage
template <typename T> struct RkStage {
    int s, last, adaptive, forward;
    T a[6], e[6];
    T cs, es;                  // weights of this stage's own slope
    const T* m0;
    T* out;
    T* hd;                     // demag field recorded here, or NULL
    KPtrs<T> kb;
};

// The stage at cell i with demag field d; returns the stored state (of which
// the next field is taken) and the error norm over dt.
template <typename T>
__device__ __forceinline__ V3<T> rk_cell(const Params<T>& p, const RkStage<T>& g, const T* __restrict__ m_in, long i,
                                         int x, int y, int z, T Msi, bool folded, const V3<T>& d, T dt, T& err,
                                         bool& bad) {
    V3<T> ks = {0, 0, 0};
    const V3<T> mi = load3(m_in, i, p.N);
    V3<T> kj[5];
#pragma unroll
    for (int j = 0; j < 5; ++j)
        if (j < g.s && (g.a[j] != (T)0 || g.e[j] != (T)0)) kj[j] = load3((const T*)g.kb.k[j], i, p.N);
        else kj[j] = {0, 0, 0};
    const V3<T> a0 = g.s == 0 ? mi : load3(g.m0, i, p.N);
    if (Msi != (T)0) {
        const T inv = inv_ms_at(p, Msi);
        V3<T> h = exchange_at(p, m_in, i, x, y, z, mi, folded ? (T)1 : inv);
        const V3<T> l = local_at(p, mi, inv);
        h = {h.x + l.x + d.x, h.y + l.y + d.y, h.z + l.z + d.z};
        if (p.dmi) {
            const V3<T> q = dmi_at(p, m_in, i, x, y, z, inv);
            h = {h.x + q.x, h.y + q.y, h.z + q.z};
        }
        ks = llg_rhs(p, mi, h);
        if (p.stt) {
            const V3<T> q = stt_at(p, mi, inv);
            ks = {ks.x + q.x, ks.y + q.y, ks.z + q.z};
        }
    }
    V3<T> acc = {0, 0, 0}, e = {0, 0, 0};
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        acc = {acc.x + g.a[j] * kj[j].x, acc.y + g.a[j] * kj[j].y, acc.z + g.a[j] * kj[j].z};
        if (g.adaptive) e = {e.x + g.e[j] * kj[j].x, e.y + g.e[j] * kj[j].y, e.z + g.e[j] * kj[j].z};
    }
    acc = {acc.x + g.cs * ks.x, acc.y + g.cs * ks.y, acc.z + g.cs * ks.z};
    V3<T> mn = {a0.x + dt * acc.x, a0.y + dt * acc.y, a0.z + dt * acc.z};
    if (!g.last) {
        store3(g.kb.k[g.s], i, p.N, ks);
    } else {
        const T nrm = sqrt(mn.x * mn.x + mn.y * mn.y + mn.z * mn.z);
        if (Msi != (T)0 && nrm > (T)0) {
            const T inv = (T)1 / nrm;
            mn = {mn.x * inv, mn.y * inv, mn.z * inv};
        }
        bad |= !(isfinite(mn.x) && isfinite(mn.y) && isfinite(mn.z));
        if (g.adaptive) {
            e = {e.x + g.es * ks.x, e.y + g.es * ks.y, e.z + g.es * ks.z};
            const T v = sqrt(e.x * e.x + e.y * e.y + e.z * e.z);
            bad |= !isfinite(v);
            err = v > err ? v : err;
        }
    }
    store3(g.out, i, p.N, mn);
    return mn;
}

// the effective field at cell i with demag field d
template <typename T>
__device__ __forceinline__ V3<T> field_cell(const Params<T>& p, const T* __restrict__ m, long i, int x, int y, int z,
                                            T Msi, bool folded, const V3<T>& d) {
    if (Msi == (T)0) return d;      // vacuum: only the stray field
    const V3<T> mi = load3(m, i, p.N);
    const T inv = inv_ms_at(p, Msi);
    V3<T> h = exchange_at(p, m, i, x, y, z, mi, folded ? (T)1 : inv);
    const V3<T> l = local_at(p, mi, inv);
    h = {h.x + l.x + d.x, h.y + l.y + d.y, h.z + l.z + d.z};
    if (p.dmi) {
        const V3<T> q = dmi_at(p, m, i, x, y, z, inv);
        h = {h.x + q.x, h.y + q.y, h.z + q.z};
    }
    return h;
}

// 3 B lines a block: component c of row r0 + b is line c B + b.  STAGE: g and
// ctl; otherwise the effective field to H.  folded: A / Ms is in the axis
// constants of p already (uniform material: one rounding a bond fewer).
// MAXT: the bound, not the block.  512 keeps the stage within 128 registers (112
// to 116 but for the longest rows), two blocks of 256 threads to an SM; at 384 it
// took 130 to 132, one block, and more rows than SMs went in two waves
// (300x300x1 21.3 us a stage, now 15.4).
template <typename T, int L1, int L2, bool STAGE, int MAXT>
__global__ void __launch_bounds__(MAXT)
    k_px_cell(PC<T>* __restrict__ buf, long R, Params<T> p, bool folded, int lgB, T scale, const PC<T>* __restrict__ twL,
              const PC<T>* __restrict__ twP, const T* __restrict__ m_in, T* __restrict__ H, RkStage<T> g, Control* ctl) {
    dep_wait();
    using C = PC<T>;
    constexpr int L = L1 * L2, LP = plane_pitch(L1, L2) + 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* Sm = reinterpret_cast<C*>(smem_raw);
    // (one answer for the block: an RK4 stage of another block may raise the status now)
    if (STAGE && __syncthreads_or(ctl->status != 0 || ctl->done)) return;
    const T dt = STAGE ? (T)ctl->dt : (T)0;
    const int tid = threadIdx.x, nt = blockDim.x, B = 1 << lgB, lines = 3 * B;
    const int nrows = p.ny * p.nz, r0 = (int)blockIdx.x << lgB;
    const T half = (T)0.5;
    // planes -> packed half-length spectra (k_px_inv)
    for (int idx = tid; idx < lines * (L / 2 + 1); idx += nt) {
        const int b = idx & (B - 1), ck = idx >> lgB, c = ck % 3, k = ck / 3;
        const int r = r0 + b;
        C xk = cmk<C>((T)0, (T)0), xl = xk;
        if (r < nrows) {
            const C* q = buf + (long)c * nrows + r;
            xk = q[(long)k * R];
            xl = cconj(q[(long)(L - k) * R]);
        }
        const C e = cscale(cadd(xk, xl), half);
        const C o = cmul(cscale(csub(xk, xl), half), cconj(twP[k]));
        C* s = Sm + ((c << lgB) + b) * LP;
        s[(k / L2) * (L2 + 1) + k % L2] = cmk<C>(e.x - o.y, e.y + o.x);
        const int kc = L - k;
        if (k > 0 && kc != k) s[(kc / L2) * (L2 + 1) + kc % L2] = cmk<C>(e.x + o.y, o.x - e.y);
    }
    __syncthreads();
    if (tid < lines * L2) {
        const int t = tid % L2;
        C* s = Sm + (tid / L2) * LP + t;
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
    {
        // the kept half of the line as plain reals, x = 0, 1, ... from the line's start
        const bool act = tid < lines * L1;
        const int k1 = tid % L1;
        C* line = Sm + (act ? tid / L1 : 0) * LP;
        C u[L2];
        if (act) {
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) u[n2] = line[k1 * (L2 + 1) + n2];
        }
        __syncthreads();
        if (act) {
            dif<L2, +1, false>(u);
#pragma unroll
            for (int k2 = 0; k2 < L2 / 2; ++k2) line[k1 + L1 * k2] = cscale(u[dif_pos<L2>(k2)], scale);
        }
    }
    __syncthreads();
    // cells: demag field in, state times Ms out, at the same place
    T* F = reinterpret_cast<T*>(Sm);
    constexpr int LF = 2 * LP;
    T err = 0;
    bool bad = false;
    for (int i = tid; i < B * L; i += nt) {
        const int b = i / L, x = i - b * L, r = r0 + b;
        T* f = F + b * LF + x;
        const int fs = LF << lgB;
        V3<T> w = {0, 0, 0};
        if (r < nrows && x < p.nx) {
            const long cell = (long)r * p.nx + x;
            const int z = r / p.ny, y = r - z * p.ny;
            const T Msi = p.Ms_cell ? p.Ms_cell[cell] : p.Ms;
            const V3<T> d = {f[0], f[fs], f[2 * fs]};
            if constexpr (STAGE) {
                if (g.hd) store3(g.hd, cell, p.N, d);
                const V3<T> mn = rk_cell(p, g, m_in, cell, x, y, z, Msi, folded, d, dt, err, bad);
                w = {mn.x * Msi, mn.y * Msi, mn.z * Msi};
            } else {
                store3(H, cell, p.N, field_cell(p, m_in, cell, x, y, z, Msi, folded, d));
            }
        }
        if (STAGE && g.forward) {
            f[0] = w.x;
            f[fs] = w.y;
            f[2 * fs] = w.z;
        }
    }
    if constexpr (STAGE) {
        if (g.last) {
            if (g.adaptive) {
                // a trial that overflowed is rejected (infinite error)
                double v = (double)dt * (double)err;
                if (bad || !isfinite(v)) v = INFINITY;
                block_max_atomic(v, &ctl->err_bits);
            } else if (bad) {
                atomicCAS(&ctl->status, 0, (int)MM_ERR_NONFINITE);
            }
        }
        if (!g.forward) return;
        __syncthreads();
        // x forward of the new state (k_px_fwd)
        {
            const bool act = tid < lines * L2;
            const int t = tid % L2;
            C* line = Sm + (act ? tid / L2 : 0) * LP;
            C v[L1];
            if (act) {
#pragma unroll
                for (int n1 = 0; n1 < L1 / 2; ++n1) v[n1] = line[t + L2 * n1];
            }
            __syncthreads();
            if (act) {
                const C* tq = twL + t;
                dif<L1, -1, true>(v);
#pragma unroll
                for (int k1 = 0; k1 < L1; ++k1) {
                    C y = v[dif_pos<L1>(k1)];
                    if (k1 > 0) y = cmul(y, tq[k1 * L2]);
                    line[k1 * (L2 + 1) + t] = y;
                }
            }
        }
        __syncthreads();
        if (tid < lines * L1) {
            C* s = Sm + (tid / L1) * LP + (tid % L1) * (L2 + 1);
            C u[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) u[n2] = s[n2];
            dif<L2, -1, false>(u);
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) s[k2] = u[dif_pos<L2>(k2)];
        }
        __syncthreads();
        for (int idx = tid; idx < lines * (L / 2 + 1); idx += nt) {
            const int b = idx & (B - 1), ck = idx >> lgB, c = ck % 3, k = ck / 3;
            const int r = r0 + b;
            if (r >= nrows) continue;
            const int kc = k == 0 ? 0 : L - k;
            const C* s = Sm + ((c << lgB) + b) * LP;
            const C zk = s[(k % L1) * (L2 + 1) + k / L1];
            const C zc = cconj(s[(kc % L1) * (L2 + 1) + kc / L1]);
            const C e = cscale(cadd(zk, zc), half);
            const C wd = cmul(twP[k], cscale(csub(zk, zc), half));
            C* q = buf + (long)c * nrows + r;
            q[(long)k * R] = cmk<C>(e.x + wd.y, e.y - wd.x);
            if (2 * k != L) q[(long)(L - k) * R] = cmk<C>(e.x - wd.y, -(e.y + wd.x));
        }
    }
}

}  // namespace mm
