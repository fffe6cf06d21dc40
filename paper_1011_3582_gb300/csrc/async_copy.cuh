// Asynchronous global -> shared staging for the row and column kernels:
// 1-D bulk copies (cp.async.bulk) and 2-D tensor-map copies
// (cp.async.bulk.tensor) completing on shared-memory mbarriers, with waits
// that give up after a bounded number of polls instead of spinning forever.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fftlb {

// A stage whose copies have not landed after this many nanoseconds of
// polling (read from the %globaltimer nanosecond clock) is declared stuck;
// kWaitPolls caps the polls as well, in case that clock does not advance.
constexpr unsigned long long kWaitNs = 2000000000ull;
constexpr unsigned kWaitPolls = 1u << 28;

// bits of the device error word
constexpr int kErrWaitTimeout = 1;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make barrier initialisation visible to the async proxy
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// order this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (bulk copy) accesses
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may start before the kernel before it on the stream has been
// retired.  grid_dep_wait() returns once that kernel has completed and its
// memory operations are visible; every read or write of memory the previous
// kernels touch comes after it.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// PEER: the phase also orders what other blocks of the cluster wrote
template <bool PEER = false> __device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (PEER)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    else asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounded wait by this thread; false if the phase did not complete within
// limit_ns of %globaltimer time (or kWaitPolls polls)
template <bool PEER = false>
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  unsigned long long limit_ns = kWaitNs) {
    if (mbar_try_wait<PEER>(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned i = 1; i < kWaitPolls; ++i) {
        if (mbar_try_wait<PEER>(bar, parity)) return true;
        if ((i & 63u) == 0 && global_ns() - t0 > limit_ns) return false;
    }
    return false;
}

// Block-wide wait for one phase.  Returns false in every thread if any
// thread gave up; the caller then records the error and drains.
__device__ __forceinline__ bool block_wait(uint64_t *bar, uint32_t parity, int *err,
                                           unsigned long long limit_ns = kWaitNs) {
    const bool ok = mbar_wait_bounded(bar, parity, limit_ns);
    const int bad = __syncthreads_or(ok ? 0 : 1);
    if (bad && threadIdx.x == 0) atomicOr(err, kErrWaitTimeout);
    return bad == 0;
}

// 1-D bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 2-D tiled tensor copy of one box at coordinates (x, y) (x in elements of
// the innermost dimension; x * element size must be a multiple of 16)
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// L2 prefetch of `bytes` (multiple of 16, 16-byte aligned) of global
// memory: no destination, no barrier, nothing to wait for
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

}  // namespace fftlb
