// gp_async.cuh -- mbarrier and bulk-copy helpers shared by the kernels that
// stage global memory in shared memory through the tensor memory accelerator
// (the TMA z sweep, the bulk-copy observables reduction of real fields, the
// bounded-wait self-test).  Hand-written inline PTX of the documented instruction forms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gpcn {

// Bound of every mbarrier wait: about a second of SM clock cycles.
constexpr long long kSpinCycles = 1LL << 31;

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for the phase of `bar` with the given parity, for at most `cycles`
// clock cycles (none at all once `ok` is false).  Returns false on expiry.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity, bool ok,
                                                  long long cycles = kSpinCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    if (!ok) return false;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > cycles) return false;
    return true;
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// Programmatic dependent launch: let the next launch of the stream begin, and
// wait until the previous one has completed and its writes are visible
// (nothing to wait for in a launch without the attribute).  What the previous
// launch writes (psi, the renormalisation factor) is read by ordinary loads
// after the wait; __ldg is for tables alone: its non-coherent load is defined
// only where nobody writes during the whole life of the kernel, which here
// begins before the previous launch has ended.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// One untiled bulk copy of `bytes` (a multiple of 16; both addresses
// 16-byte aligned) from global memory into this CTA's shared memory,
// completing on the transaction count of mbarrier `bar`.
__device__ __forceinline__ void bulk_load(unsigned dst, const void *src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Launch a kernel so that its blocks may be placed while the previous launch's
// last ones run.  The kernel calls pdl_wait() before it touches anything that
// the previous launch writes or reads.  For launches into a stream only (axial
// steps: 21.8 -> 20.2 us a step of two launches on 120x241): in captured graphs
// the same attribute slowed every step (64x48x40 FP64 25.8 -> 35.6 us, 200x160x120
// complex64 62 -> 84 us), and those launches go without it.
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                                    const A &...args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace gpcn
