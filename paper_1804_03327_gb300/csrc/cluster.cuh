// Thread-block cluster building blocks of the small-frontier kernels (bfs_cluster.cu,
// sssp_cluster.cu): distributed shared memory, and the exchange of the blocks' counts that ends
// a level.
#pragma once

#include "gbx_internal.cuh"

namespace gbx {

constexpr int kClusterMax = 16;  // blocks of a cluster (8 where 16 do not fit)

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of shared variable p in block `rank` of the cluster.
__device__ __forceinline__ uint32_t remote_smem(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(a)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void st_remote(uint32_t a, int32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// Stores v at a (another block's or this one's shared memory) and counts its bytes on the
// mbarrier at m of the same block.
__device__ __forceinline__ void st_async(uint32_t a, int32_t v, uint32_t m) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(a), "r"(v),
                 "r"(m)
                 : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long* m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(m)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(m)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long* m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"((uint32_t)__cvta_generic_to_shared(m)), "r"(parity)
        : "memory");
    return ok != 0u;
}
__device__ __forceinline__ int32_t ld_remote(uint32_t a) {
    int32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t or_remote(uint32_t a, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared::cluster.or.b32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}

// Waits, at most timeout_ns, until the phase `parity` of mbarrier m of this block is complete;
// the whole block calls it and gets one answer.
__device__ __forceinline__ bool mbar_wait_block(unsigned long long* m, uint32_t parity, unsigned long long timeout_ns) {
    bool ok = true;
    if (threadIdx.x < 32) {
        ok = mbar_try(m, parity);
        for (unsigned long long t0 = 0ull; !ok; ok = mbar_try(m, parity)) {
            const unsigned long long now = global_timer_ns();
            if (t0 == 0ull) t0 = now;
            if (now - t0 > timeout_ns) break;
        }
    }
    return __syncthreads_and(ok) != 0;
}

// A bounded wait of this block ran out: records it in `status` and tells every block, which
// sees it (*abort, its own shared variable) at its next cluster barrier -- its own wait
// runs out, or it is at a barrier of the level.  Nobody touches another block after that one.
__device__ __forceinline__ void cluster_give_up(int32_t* abort, int blocks, int32_t* status) {
    if ((int)threadIdx.x < blocks) st_remote(remote_smem(abort, threadIdx.x), 1);
    if (threadIdx.x == 0) atomicCAS(status + ST_ERROR, 0, (int)GBX_ERR_TIMEOUT);
    cluster_barrier();
}

// The block of the cluster, and the place in its queue, of entry g of all queues one after
// another: lane r of the warp holds in inc where block r's queue ends.  All lanes call.
__device__ __forceinline__ void cluster_locate(int32_t inc, int32_t g, int32_t& block, int32_t& place) {
    int32_t o = 0;
#pragma unroll
    for (int s = kClusterMax / 2; s > 0; s >>= 1) {
        const int32_t y = __shfl_sync(0xffffffffu, inc, o + s - 1);
        if (g >= y) o += s;
    }
    const int32_t y = __shfl_sync(0xffffffffu, inc, o > 0 ? o - 1 : 0);
    block = o;
    place = g - (o > 0 ? y : 0);
}

// The number of blocks (16 or 8) of the largest cluster of fn that fits the device, -1 if none
// does.  Sets fn's shared memory limit.
gbx_status cluster_fit(const void* fn, int threads, size_t smem, int* blocks);
gbx_status cluster_launch(const void* fn, int blocks, int threads, size_t smem, void** args, cudaStream_t s);

}  // namespace gbx
