// cluster_device.cuh -- thread-block cluster and mbarrier primitives of the tails
// (cluster.cu, dense.cu): ranks, remote shared-memory accesses, asynchronous
// stores that complete on the receiver's mbarrier, L2 prefetches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cl_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// all threads of every CTA of the cluster; release/acquire orders the
// shared-memory writes (local and remote) before it against reads after it
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the shared::cluster address of 'p' (this CTA's shared memory) in CTA 'rank'
__device__ __forceinline__ uint32_t cl_map(const void *p, unsigned rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t o;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(rank));
    return o;
}

__device__ __forceinline__ unsigned cl_ld_u16(uint32_t a) {
    unsigned short v;
    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void cl_st_u32(uint32_t a, unsigned x) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}

// 16 bytes into another CTA's shared memory, completing (as 16 transaction
// bytes) on the mbarrier at 'mbar' in that CTA
__device__ __forceinline__ void cl_st_async_v4(uint32_t a, uint32_t mbar, unsigned x, unsigned y, unsigned z,
                                               unsigned w) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mb_init(unsigned long long *mb, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(mb)), "r"(count)
                 : "memory");
}

// this thread's arrival, announcing 'tx' transaction bytes for the current phase
__device__ __forceinline__ void mb_arrive_expect_tx(unsigned long long *mb, unsigned tx) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
            (unsigned)__cvta_generic_to_shared(mb)),
        "r"(tx)
        : "memory");
}

// has the phase of parity 'parity' completed? (acquire at cluster scope: the
// asynchronous stores that completed it are visible)
__device__ __forceinline__ bool mb_try_wait(unsigned long long *mb, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, "
        "1, 0, p;\n\t}"
        : "=r"(done)
        : "r"((unsigned)__cvta_generic_to_shared(mb)), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ void cl_st_u64(uint32_t a, unsigned long long x) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(x) : "memory");
}

// L2 prefetch of bytes [off, off + len) of an array of 'total' bytes, in
// 16-byte granules inside the array (one bulk request, no data returned)
__device__ __forceinline__ void prefetch_l2(const void *base, unsigned long long total, unsigned long long off,
                                            unsigned long long len) {
    const unsigned long long a = off & ~15ull;
    unsigned long long b = (off + len + 15) & ~15ull;
    const unsigned long long end = total & ~15ull;
    if (b > end) b = end;
    if (b > a)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((const char *)base + a), "r"((unsigned)(b - a))
                     : "memory");
}
