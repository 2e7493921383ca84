// gp_res.cuh -- FP32 line solves of short lines held whole in shared memory.
//
// The streaming sweeps give a line one thread, which alternates between its
// copies, its kick and its recurrences; on grids of 30..130 nodes a side that
// leaves each launch waiting for one dependent chain after another (a sweep
// of 64 condensates ran 30-60 us at 13-43 % of the HBM rate, a 48x40x32 x sweep
// 20 us).  Here a block loads `tl` whole lines at once, and each part of the
// solve takes the parallelism it has:
//  1. load and kick, the right-hand sides: every node a work item;
//  2. the forward recurrence: one thread per line, values prefetched in
//     chunks, nothing but the recurrence on the chain;
//  3. the windowed backward recurrence: one thread per (line, chunk of B
//     nodes), since every chunk starts from its own dp;
//  4. the store (and the norm): every node a work item.
// The arithmetic per node, the chunk length B and the window W are those of
// the streaming form that the same settings select, so the results are the
// same bit for bit; only the norm's partial sums are grouped differently.
// Taken for lines of one segment (at most 128 interior nodes).
#pragma once

#include "gp_sweep.cuh"

namespace gpcn {

constexpr int kResThreads = 128;

// Shared-memory pitch of a line (K_Z: lines contiguous, an odd number of
// values, so that the threads of a warp on different lines meet different
// banks) and distance between neighbouring nodes.
template <int KIND> __device__ __forceinline__ int res_index(int t, int l, int tl, int pitch) {
    return KIND == K_Z ? l * pitch + t : t * tl + l;
}

template <class F, typename R, int KIND>
__device__ __forceinline__ double res_body(const SweepArgs &a, unsigned block, unsigned char *smem_raw) {
    using V = typename F::V;
    using C = typename F::C;
    const int n = a.N - 2, tl = a.res_tl, B = a.res_chunk, W = a.res_window, T = kResThreads;
    const int pitch = n | 1, step = KIND == K_Z ? 1 : tl;
    const long long L0 = (long long)block * tl;
    const int nl = (int)min((long long)tl, a.n_lines - L0);
    V *x = reinterpret_cast<V *>(smem_raw), *y = x + (KIND == K_Z ? tl * pitch : tl * n);
    const V *in = static_cast<const V *>(a.psi);
    V *out = static_cast<V *>(a.psi_out);
    const C *cp = static_cast<const C *>(a.cp), *ipm1 = static_cast<const C *>(a.ip);
    const R kap = (R)a.kappa;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // The nodes of the block's lines, four at a time: f(t, l, offset of node t + 1).
    // K_X, K_Y: a thread keeps one line (threads of a warp adjacent lines);
    // K_Z: a warp takes a line, its lanes adjacent nodes.
    long long off = 0;
    int l = 0;
    if (KIND != K_Z) {
        l = threadIdx.x & (tl - 1);
        const long long L = L0 + min(l, nl - 1);
        off = KIND == K_X ? L : (L / a.inner) * a.outer_stride + (L % a.inner);
    }
    KickState<R> ks;
    if (KIND == K_X) kick_init<R, KIND>(ks, a, L0 + min(l, nl - 1));
    if (KIND == K_Z) {
        for (int q = wid; q < nl; q += T / 32) {
            const V *g = in + (L0 + q) * a.N + 1;
            for (int t = lane; t < n; t += 32) x[q * pitch + t] = g[t];
        }
    } else if (l < nl) {
        const int dt = T / tl;
        const V *g = in + off + a.stride;
        int t = threadIdx.x / tl;
        auto kick = [&](V v, int node) {
            if constexpr (KIND == K_X) {
                if constexpr (std::is_same<F, FRealTime<float>>::value) {
                    // the pair form's phase of the node (computed, not from the table)
                    return a.res_pair ? F::kick_at(v, ks, PRealTimeF::px_of(ks, node)) : F::kick(v, ks, node);
                } else {
                    return F::kick(v, ks, node);
                }
            } else {
                return v;
            }
        };
        for (; t + 7 * dt < n; t += 8 * dt) {  // eight loads in flight
            V v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = g[(long long)(t + q * dt) * a.stride];
#pragma unroll
            for (int q = 0; q < 8; ++q) x[(t + q * dt) * tl + l] = kick(v[q], t + q * dt + 1);
        }
        for (; t < n; t += dt) x[t * tl + l] = kick(g[(long long)t * a.stride], t + 1);
    }
    __syncthreads();
    // right-hand sides
    auto rhs = [&](int t, int s) {
        const V pm = t > 0 ? x[s - step] : F::zero(), p1 = t < n - 1 ? x[s + step] : F::zero();
        y[s] = F::rhs(pm, x[s], p1, kap);
    };
    if (KIND == K_Z) {
        for (int q = wid; q < nl; q += T / 32)
            for (int t = lane; t < n; t += 32) rhs(t, q * pitch + t);
    } else if (l < nl) {
#pragma unroll 4
        for (int t = threadIdx.x / tl; t < n; t += T / tl) rhs(t, t * tl + l);
    }
    __syncthreads();
    // forward: dp over the right-hand sides
    if ((int)threadIdx.x < nl) {
        V *c = y + (KIND == K_Z ? threadIdx.x * pitch : threadIdx.x);
        const C ips = ldc(ipm1 + n - 1);
        V dp = F::zero();
        int t = 0;
        for (; t < n && t < a.t_const; ++t) {
            dp = F::fwd(c[t * step], dp, kap, ldc(ipm1 + t));
            c[t * step] = dp;
        }
        for (; t + 8 <= n; t += 8) {
            V r[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) r[q] = c[(t + q) * step];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                dp = F::fwd(r[q], dp, kap, ips);
                c[(t + q) * step] = dp;
            }
        }
        for (; t < n; ++t) {
            dp = F::fwd(c[t * step], dp, kap, ips);
            c[t * step] = dp;
        }
    }
    __syncthreads();
    // backward: full chunks start W nodes ahead with phi = dp; the rest of the
    // line (from node B full) is exact from phi[n-1] = dp[n-1]
    {
        const int full = n >= B + W ? (n - W) / B : 0, items = (full + 1) * nl;
        const C cps = ldc(cp + n - 1);
        for (int it = threadIdx.x; it < items; it += T) {
            const int c = it / nl, q = it - c * nl, t0 = c * B;
            const int s0 = KIND == K_Z ? q * pitch : q;
            const V *d = y + s0;
            V *o = x + s0;
            int t = c < full ? t0 + B + W - 1 : n - 1;
            const int te = c < full ? t0 + B : n;  // results below te are kept
            V phi = d[t * step];
            if (t < te) o[t * step] = phi;
            if (t0 >= a.t_const) {
#pragma unroll 4
                for (--t; t >= t0; --t) {
                    phi = F::back(d[t * step], cps, phi);
                    if (t < te) o[t * step] = phi;
                }
            } else {
                for (--t; t >= t0; --t) {
                    phi = F::back(d[t * step], ldc(cp + t), phi);
                    if (t < te) o[t * step] = phi;
                }
            }
        }
    }
    __syncthreads();
    Acc<R> acc;
    if (KIND == K_Z) {
        for (int q = wid; q < nl; q += T / 32) {
            V *g = out + (L0 + q) * a.N + 1;
            for (int t = lane; t < n; t += 32) {
                const V v = x[q * pitch + t];
                g[t] = v;
                acc.add(F::abs2(v));
            }
            if (lane == 0) g[-1] = F::zero();
            if (lane == 1) g[n] = F::zero();
        }
    } else if (l < nl) {
        V *g = out + off + a.stride;
#pragma unroll 4
        for (int t = threadIdx.x / tl; t < n; t += T / tl) g[(long long)t * a.stride] = x[t * tl + l];
        if ((int)threadIdx.x < tl) {
            out[off] = F::zero();
            out[off + (long long)(a.N - 1) * a.stride] = F::zero();
        }
    }
    return acc.value();
}

template <class F, typename R, int KIND>
__global__ void __launch_bounds__(kResThreads) sweep_res_kernel(SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const double v = res_body<F, R, KIND>(a, blockIdx.x, smem_raw);
    if (KIND == K_Z && !real_time<F>()) norm_finalize(v, a, blockIdx.x, gridDim.x);
}

// Many condensates in one launch (see BatchDesc).
template <class F, typename R, int KIND>
__global__ void __launch_bounds__(kResThreads) batch_res_kernel(BatchDesc d) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int i = find_instance(d, blockIdx.x);
    const SweepArgs a = d.args[i];
    const unsigned local = blockIdx.x - __ldg(d.first + i);
    const unsigned nblocks = __ldg(d.first + i + 1) - __ldg(d.first + i);
    const double v = res_body<F, R, KIND>(a, local, smem_raw);
    if (KIND == K_Z) norm_finalize(v, a, local, nblocks);
}

}  // namespace gpcn
