// common.cuh -- device helpers shared by the SwitchSD kernels (sm_103a).
//
// Thin inline-PTX wrappers for the Blackwell features the kernels use: mbarriers with transaction
// counts, bulk (TMA) global->shared copies, and split arrive/wait cluster barriers.  Every wait on an
// mbarrier is bounded: after kWaitLimit polls it gives up and reports failure to the caller, which
// records SWITCHSD_ROW_TIMEOUT instead of hanging.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "switchsd.h"

namespace switchsd {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;
// Polls of mbarrier.try_wait before a wait is declared failed.  Each poll may suspend the thread
// for a hardware-chosen interval, so the limit bounds the wait to well under a second.
constexpr uint32_t kWaitLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

// Makes barrier initialisation visible to the async (TMA) proxy and the rest of the cluster.
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// A plain arrive (release at CTA scope): the arriving thread's earlier shared-memory writes are visible to a
// thread that then observes the phase complete.
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}

// The same for a barrier that only counts an asynchronous copy's bytes: the arriving thread publishes
// nothing through it, so the arrive needs no release ordering.
__device__ __forceinline__ void mbar_expect_tx_relaxed(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// Bounded wait for phase `parity` of the barrier to complete.  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    const uint32_t addr = smem_addr(bar);
    for (uint32_t it = 0; it < kWaitLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// mbar_wait with a caller's poll count (0: give up at once).
__device__ __forceinline__ bool mbar_wait_polls(uint64_t *bar, uint32_t parity, uint32_t polls) {
    const uint32_t addr = smem_addr(bar);
    for (uint32_t it = 0; it < polls; ++it) {
        uint32_t done;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Bulk asynchronous copy global -> this CTA's shared memory, completing `bytes` of transaction on
// `bar`.  dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// L2 policy for data read once per launch (the context): evicted before anything else, so the
// small per-step arrays (lengths, drafts, targets) stay cached while the contexts stream through.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void bulk_g2s_hint(void *dst, const void *src, uint32_t bytes, uint64_t *bar,
                                              uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], "
        "%4;\n" ::"r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}

// Split cluster barrier.  Every thread of every CTA in the cluster executes each arrive and each
// wait the same number of times.
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_release() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_nctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(r));
    return r;
}

// Address of the same shared variable in CTA `rank` of the cluster (shared::cluster window).
__device__ __forceinline__ uint32_t map_to_rank(const void *p, uint32_t rank) {
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(out) : "r"(smem_addr(p)), "r"(rank));
    return out;
}

// Programmatic dependent launch.  Every kernel of the library is launched with programmatic stream
// serialization: it waits for the preceding kernel (griddepcontrol.wait) before its first read of
// data that kernel may have written, and lets the next kernel start launching right after
// (griddepcontrol.launch_dependents), so launch latency overlaps execution.  Both are no-ops when the
// launch carries no programmatic dependency.  A grid may so be resident while the kernel before it writes the
// grid's inputs: they are read with plain loads, bulk copies or through L2, never through the non-coherent path
// (__ldg), which asks for data that nothing writes while the grid runs.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// Asynchronous 16-byte store into another CTA's shared memory that completes 16 bytes of transaction
// on that CTA's mbarrier (both addresses in the shared::cluster window).
__device__ __forceinline__ void st_async_v4(uint32_t cluster_addr, uint4 v, uint32_t cluster_mbar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
            cluster_addr),
        "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(cluster_mbar)
        : "memory");
}

// Bulk copy of `bytes` from this CTA's shared memory to another CTA's (cluster address), completing that
// many bytes of transaction on the destination's mbarrier (cluster address).  Both addresses 16-byte
// aligned, bytes a multiple of 16.  The source is read asynchronously: generic writes to it need
// fence_proxy_async() first, and it stays untouched until bulk_wait_read() returns.
__device__ __forceinline__ void bulk_s2c(uint32_t dst_cluster, const void *src, uint32_t bytes, uint32_t mbar_cluster) {
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
        "cp.async.bulk.commit_group;\n" ::"r"(dst_cluster),
        "r"(smem_addr(src)), "r"(bytes), "r"(mbar_cluster)
        : "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }

// Generic accesses to shared memory before it are ordered before asynchronous accesses to it after it.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// Launches `kernel` on `stream` with programmatic stream serialization and, when cluster_x >= 1, an
// explicit cluster shape of cluster_x CTAs (1 included: the cluster instructions of the rescan kernel,
// st.async into shared::cluster in particular, need an explicit cluster launch).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              unsigned cluster_x, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
    if (cluster_x >= 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster_x;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// The per-mode tallies of switchsd_params.counters for one row: its step chose `mode`; when its
// verification appended (acc >= 0) the draft it verified came from the previous step's mode `prev`.
__device__ __forceinline__ void count_row(unsigned long long *ctr, int32_t mode, bool verified, int32_t prev,
                                          int32_t acc) {
    atomicAdd(&ctr[SWITCHSD_CTR_STEPS + mode], 1ull);
    if (verified && acc >= 0) {
        const int slot = prev == SWITCHSD_MODE_COPY ? SWITCHSD_CTR_COPY_DRAFTS : SWITCHSD_CTR_NEURAL_DRAFTS;
        atomicAdd(&ctr[slot], 1ull);
        atomicAdd(&ctr[slot + 1], static_cast<unsigned long long>(acc));
    }
}

__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ float warp_sum_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

}  // namespace switchsd
