// gp_pcr.cuh -- FP64 line solves by truncated parallel cyclic reduction.
//
// One FP64 warp instruction takes 64 clock cycles on this part (measured: 64.4
// with independent operations, 66 in a dependent chain, the same for 1 to 32
// active lanes), up to four warps of an SM side by side, more sharing the
// pipe, and a one-thread-per-line Thomas solve of a small grid leaves most of
// the SMs' room for 608 idle: 64x48x40 has 60 warps of x lines.  Here a block keeps
// `tl` whole lines in shared memory and every node is a work item: the kick,
// the right-hand side and each reduction level run over all (node, line)
// pairs, with one barrier between them.
//
// A sweep is solved for the change d = phi - p it makes to the kicked values p:
// (1 + K) phi = (1 - K) p is (1 + K) d = -2 K p, the same matrix.  Every
// rounding and the truncation below are then relative to the change, and the
// one rounding at the size of the field is that of phi = p + d; reducing phi
// itself rounded each node twice a level at the size of the field and was 1.4
// to 3 times as far from extended-precision sweeps as the two-pass solve
// (48x56x40 real, 10 steps: 2.9e-15 of max|psi| against 1.0e-15).
//
// Cyclic reduction on the CN matrix (-a, D, -c): level l (distance e = 2^l)
// eliminates the neighbours at distance e,
//     R[t] <- R[t] + A_l[t] R[t-e] + C_l[t] R[t+e],
// with A_l, C_l (and the final 1/D) precomputed per node on the host.  The
// coupling that is left after level l is about |cp|^(2^(l+1)) of the diagonal
// (cp the Thomas multiplier), so the levels stop when it is below 2^-55 of it,
// a quarter of the unit roundoff of the change: 4 levels at c = 0.025
// (dt = 0.1 d^2), 3 at c = 0.005i, whatever the length of the line.  The tables
// carry the ends of the line (zero beyond them), so every length is served.
// Real coefficients cost 3 + 2 levels + 1 operations per component and node
// against 6 for Thomas: the host takes this form where its better balance
// outweighs that (choose_pcr).
#pragma once

#include "gp_async.cuh"
#include "gp_optin.h"
#include "gp_sweep.cuh"

namespace gpcn {

__device__ __forceinline__ double pcr_mac(double acc, double c, double v) { return fma(c, v, acc); }
__device__ __forceinline__ cx<double> pcr_mac(cx<double> acc, double c, cx<double> v) {
    return cx<double>{fma(c, v.re, acc.re), fma(c, v.im, acc.im)};
}
__device__ __forceinline__ cx<double> pcr_mac(cx<double> acc, cx<double> c, cx<double> v) {
    return cx<double>{fma(c.re, v.re, fma(-c.im, v.im, acc.re)), fma(c.re, v.im, fma(c.im, v.re, acc.im))};
}
// 2 c (pm + p1 - 2 p0), c = k / 2 (imaginary time) or i k / 2 (real time)
template <class F> __device__ __forceinline__ double pcr_rhs(double pm, double p0, double p1, double k) {
    return k * fma(-2.0, p0, pm + p1);
}
template <class F> __device__ __forceinline__ cx<double> pcr_rhs(cx<double> pm, cx<double> p0, cx<double> p1, double k) {
    const double re = k * fma(-2.0, p0.re, pm.re + p1.re), im = k * fma(-2.0, p0.im, pm.im + p1.im);
    return real_time<F>() ? cx<double>{-im, re} : cx<double>{re, im};
}
__device__ __forceinline__ double pcr_mul(double c, double v) { return c * v; }
__device__ __forceinline__ cx<double> pcr_mul(double c, cx<double> v) { return cx<double>{c * v.re, c * v.im}; }
__device__ __forceinline__ cx<double> pcr_mul(cx<double> c, cx<double> v) {
    return cx<double>{fma(c.re, v.re, -c.im * v.im), fma(c.re, v.im, c.im * v.re)};
}
__device__ __forceinline__ double pcr_sub(double a, double b) { return a - b; }
__device__ __forceinline__ cx<double> pcr_sub(cx<double> a, cx<double> b) { return cx<double>{a.re - b.re, a.im - b.im}; }

// The block's sum of v over its first `count` threads (through `buf`, `count`
// values of shared memory), then the last block's sum of the partials, in
// fixed orders; four warps add, one per sub-partition (a warp sum of every
// warp would cost the FP64 pipe five instructions for each).
__device__ __forceinline__ void pcr_norm(double v, double *buf, int count, const SweepArgs &a) {
    __shared__ double red[4];
    __shared__ int is_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, quad = min((int)blockDim.x, 128);
    if ((int)threadIdx.x < count) buf[threadIdx.x] = v;
    __syncthreads();
    if ((int)threadIdx.x < quad) {
        double t = 0.0;
        for (int q = threadIdx.x; q < count; q += quad) t += buf[q];
        t = warp_sum(t);
        if (lane == 0) red[wid] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = red[0];
        for (int w = 1; w < quad / 32; ++w) t += red[w];
        a.partials[blockIdx.x] = t;
        __threadfence();
        is_last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if ((int)threadIdx.x < quad) {
        double t = 0.0;
        for (unsigned b = threadIdx.x; b < gridDim.x; b += quad) t += __ldcg(a.partials + b);
        t = warp_sum(t);
        if (lane == 0) red[wid] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = red[0];
        for (int w = 1; w < quad / 32; ++w) t += red[w];
        const double nrm = a.dV * t;
        *a.norm_out = nrm;
        if (a.want_scale) *a.scale_out = 1.0 / sqrt(nrm);
        *a.counter = 0u;
    }
}

// NS work items per thread (its nodes stay in registers from level to level;
// shared memory holds what the neighbours read, and the tables).
// RADIAL: the lines' matrix varies along the line and the right-hand side is
// 2 A (pm - p0) + 2 C (p1 - p0) with 2 A, 2 C from p.rhs; the first and the
// last line (the z boundary) are zero whatever the input holds.
template <class F, int KIND, bool RADIAL, int NS>
__global__ void __launch_bounds__(1024) lines_pcr_kernel(SweepArgs a, PcrArgs p) {
    using V = typename F::V;
    using C = typename F::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.N - 2, T = blockDim.x;
    const unsigned L0 = blockIdx.x * (unsigned)p.tl, lines = (unsigned)a.n_lines;
    const int nl = (int)min((unsigned)p.tl, lines - L0);
    const int total = nl * n;
    const int step = KIND == K_Z ? 1 : nl;  // distance of neighbouring nodes in shared memory
    V *x = reinterpret_cast<V *>(smem_raw), *y = x + (size_t)p.tl * n;
    C *tab = reinterpret_cast<C *>(y + (size_t)p.tl * n);  // levels, final inverse, radial right-hand side
    const int ntab = 2 * p.levels * n;
    C *inv = tab + ntab, *rhs = inv + n;
    double *lk = reinterpret_cast<double *>(rhs + (RADIAL ? 2 * n : 0));  // the kick's factor or phase of each line
    const V *in = static_cast<const V *>(a.psi);
    V *out = static_cast<V *>(a.psi_out);
    auto origin = [&](int l) -> long long {
        const unsigned L = L0 + l;
        if (KIND == K_X) return L;
        if (KIND == K_Z) return (long long)L * a.N;
        const unsigned o = L / (unsigned)a.inner;
        return (long long)o * a.outer_stride + (L - o * (unsigned)a.inner);
    };
    // the tables, which no launch writes, while the previous sweep ends
    pdl_trigger();
    for (int q = threadIdx.x; q < ntab; q += T) tab[q] = ldc(static_cast<const C *>(p.lv) + q);
    for (int q = threadIdx.x; q < n; q += T) inv[q] = ldc(static_cast<const C *>(p.inv) + q);
    if (RADIAL)
        for (int q = threadIdx.x; q < 2 * n; q += T) rhs[q] = ldc(static_cast<const C *>(p.rhs) + q);
    pdl_wait();
    // item i of the thread: node t of line l of the block (the global
    // accesses of a warp run along the contiguous axis), all ones past the end
    int tt[NS], ll[NS];
    V p0[NS], v[NS];  // the kicked value, its change
    KickState<double> ks;
    if (KIND == K_X) {
        for (int l = threadIdx.x; l < nl; l += T) {
            kick_init<double, KIND>(ks, a, (long long)(L0 + l));
            lk[l] = a.kick_ex ? ks.eyz : ks.pyz;
        }
        kick_init<double, KIND>(ks, a, (long long)L0);
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int s = threadIdx.x + i * T;
        tt[i] = -1;
        ll[i] = 0;
        p0[i] = v[i] = F::zero();
        if (s < total) {
            const int m = KIND == K_Z ? n : nl, q = s / m, r = s - q * m;
            tt[i] = KIND == K_Z ? r : q;
            ll[i] = KIND == K_Z ? q : r;
            if (!RADIAL || (L0 + ll[i] > 0 && L0 + ll[i] < lines - 1))
                p0[i] = in[origin(ll[i]) + (long long)(tt[i] + 1) * a.stride];
        }
    }
    for (int q = threadIdx.x; q < 2 * nl; q += T)  // the line ends
        out[origin(q >> 1) + (q & 1 ? (long long)(a.N - 1) * a.stride : 0)] = F::zero();
    if (KIND == K_X) __syncthreads();  // lk
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        if (tt[i] < 0) continue;
        if (KIND == K_X && (!RADIAL || (L0 + ll[i] > 0 && L0 + ll[i] < lines - 1))) {
            ks.eyz = ks.pyz = lk[ll[i]];
            p0[i] = F::kick(p0[i], ks, tt[i] + 1);
        }
        x[threadIdx.x + i * T] = p0[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int t = tt[i], s = threadIdx.x + i * T;
        if (t < 0) continue;
        const V pm = t > 0 ? x[s - step] : F::zero(), p1 = t < n - 1 ? x[s + step] : F::zero();
        if (RADIAL) v[i] = pcr_mac(pcr_mul(rhs[2 * t], pcr_sub(pm, p0[i])), rhs[2 * t + 1], pcr_sub(p1, p0[i]));
        else v[i] = pcr_rhs<F>(pm, p0[i], p1, 2.0 * a.kappa);
        y[s] = v[i];
    }
    for (int lv = 0; lv < p.levels; ++lv) {
        __syncthreads();
        const C *tl = tab + (size_t)lv * n * 2;
        const int d = 1 << lv;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const int t = tt[i], s = threadIdx.x + i * T;
            if (t < 0) continue;
            // beyond an end the coefficient is zero: any value of the line will do
            const int lo = t >= d ? s - d * step : s, hi = t + d < n ? s + d * step : s;
            v[i] = pcr_mac(pcr_mac(v[i], tl[2 * t], y[lo]), tl[2 * t + 1], y[hi]);
            if (lv < p.levels - 1) x[s] = v[i];
        }
        V *z = x;
        x = y;
        y = z;
    }
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        if (tt[i] < 0) continue;
        const V r = pcr_mac(p0[i], inv[tt[i]], v[i]);
        out[origin(ll[i]) + (long long)(tt[i] + 1) * a.stride] = r;
        if (KIND == K_Z && !real_time<F>()) acc = p.line_w ? fma(__ldg(p.line_w + L0 + ll[i]), F::abs2(r), acc) : acc + F::abs2(r);
    }
    // after the last level's swap y is the buffer that no thread reads any more
    if (KIND == K_Z && !real_time<F>()) pcr_norm(acc, reinterpret_cast<double *>(y), min(T, total), a);
}

template <class F, int KIND, bool RADIAL, int NS>
inline cudaError_t launch_pcr_ns(const SweepArgs &a, const PcrArgs &p, int threads, size_t smem, cudaStream_t s) {
    const unsigned grid = (unsigned)((a.n_lines + p.tl - 1) / p.tl);
    static SmemOptIn kept;
    const cudaError_t e = opt_in_smem(kept, lines_pcr_kernel<F, KIND, RADIAL, NS>, kPcrSmem);
    if (e != cudaSuccess) return e;
    if (p.dependent) return launch_dependent(lines_pcr_kernel<F, KIND, RADIAL, NS>, grid, threads, smem, s, a, p);
    lines_pcr_kernel<F, KIND, RADIAL, NS><<<grid, threads, smem, s>>>(a, p);
    return cudaGetLastError();
}

// As few items per thread as 1024 threads allow: more warps cover the
// barriers and the shared-memory reads between the FP64 instructions.
template <class F, int KIND, bool RADIAL>
inline cudaError_t launch_pcr(const SweepArgs &a, const PcrArgs &p, cudaStream_t s) {
    const long long total = (long long)p.tl * (a.N - 2);
    const size_t smem = pcr_smem((int)sizeof(typename F::V), (int)sizeof(typename F::C), p.levels, p.tl, a.N);
    const int ns = total <= 1024 ? 1 : total <= 2048 ? 2 : total <= 4096 ? 4 : 8;
    const int threads = (int)(((total + ns - 1) / ns + 31) / 32 * 32);
    if (smem > kPcrSmem || total > kPcrItems) return cudaErrorInvalidValue;
    switch (ns) {
    case 1: return launch_pcr_ns<F, KIND, RADIAL, 1>(a, p, threads, smem, s);
    case 2: return launch_pcr_ns<F, KIND, RADIAL, 2>(a, p, threads, smem, s);
    case 4: return launch_pcr_ns<F, KIND, RADIAL, 4>(a, p, threads, smem, s);
    default:
        // 16-byte elements have at most 3200 pairs in kPcrSmem
        if constexpr (sizeof(typename F::V) == 8) return launch_pcr_ns<F, KIND, RADIAL, 8>(a, p, threads, smem, s);
        else return cudaErrorInvalidValue;
    }
}

}  // namespace gpcn
