// hc_async.cuh -- shared-memory mbarriers and 1-D TMA bulk copies (sm_90+ PTX),
// with bounded waits.
//
// A bulk copy moves a contiguous, 16-byte aligned block whose size is a
// multiple of 16 bytes from global to shared memory on the TMA engine; its
// completion is counted in bytes on an mbarrier (complete_tx).  Waits spin on
// mbarrier.try_wait with an iteration limit: a wait that runs out returns
// false, and the caller reports HC_ERR_TIMEOUT through a device flag instead
// of hanging the GPU.
#pragma once

#include <cstdint>

namespace hc {

constexpr uint32_t kWaitLimit = 1u << 22;  // try_wait attempts before giving up

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// make mbarrier initialisation visible to the async (TMA) proxy
__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// order earlier generic-proxy shared-memory accesses before later async-proxy ones
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// one arrival that also announces `bytes` of transactions to come
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_addr(bar)),
        "r"(bytes)
        : "memory");
}

// one arrival
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
                 : "memory");
}

// global -> shared bulk copy, completion counted on bar
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// L2 policy for data read exactly once (evict first), for bulk_g2s_stream
__device__ __forceinline__ uint64_t l2_evict_first_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// bulk_g2s with an L2 cache policy: data streamed once (the MAC's weights) goes
// first when L2 evicts, so that what the next kernel reads (the MAC's outputs,
// read by the inverse NTT) stays
__device__ __forceinline__ void bulk_g2s_stream(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t pol)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(pol)
        : "memory");
}

// ---- thread-block clusters: rank, barrier, stores into a peer's shared memory ----
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// every thread of every CTA of the cluster; orders the shared-memory writes
// (own and remote) before it with the reads after it
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the shared::cluster address of p (a shared-memory address of this CTA) in CTA rank
__device__ __forceinline__ uint32_t cluster_map(const void *p, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}

__device__ __forceinline__ void st_cluster_u64(uint32_t addr, uint64_t v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ uint64_t ld_cluster_u64(uint32_t addr)
{
    uint64_t v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}

// ---- programmatic dependent launch ------------------------------------------------
// The next kernel of the stream, if it was launched with the programmatic attribute,
// may start once every CTA of this grid has come here (or ended) ...
__device__ __forceinline__ void pdl_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ... and waits here until the grids before it have ended and their stores are visible.
// Returns at once in a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// first statement of a kernel that is launched as a programmatic dependent and may have
// dependents of its own
__device__ __forceinline__ void pdl_begin()
{
    pdl_launch_dependents();
    pdl_wait();
}

// Loads of what an earlier launch, or another CTA of this one, may have written: through L2,
// and never on the read-only path, whose loads the compiler may move above the wait.  It may
// move the load intrinsic too, which it does not see touching memory, unless the address
// comes from after_wait.
template <class T>
__device__ __forceinline__ const T *after_wait(const T *p)
{
    asm volatile("" : "+l"(p)::"memory");
    return p;
}
__device__ __forceinline__ uint64_t ld_data(const uint64_t *p)
{
    return __ldcg((const unsigned long long *)p);
}
__device__ __forceinline__ ulonglong2 ld_data(const ulonglong2 *p) { return __ldcg(p); }
// an ordinary load, through L1, for what several warps or CTAs of an SM read (the sums' term
// lists and operands, weights).  p must not come from a __restrict__ parameter, which would
// make it a read-only one.  Sums of four products through L2 instead, 64 of them at
// N = 16384, L = 4, into 16: 131 -> 169 us.
template <class T>
__device__ __forceinline__ T ld_near(const T *p)
{
    return *p;
}

// host: launch kern, as the programmatic dependent of the launch before it if asked to
template <class... P, class... A>
cudaError_t launch_programmatic(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool dependent,
                                A &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// per-thread asynchronous 8-byte global -> shared copy (completes with cp_async_wait_all)
__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// this thread's committed copies have landed (other threads': after a barrier)
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// bounded wait for the phase with the given parity to complete
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit = kWaitLimit)
{
    const uint32_t a = smem_addr(bar);
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

}  // namespace hc
