// Launch geometry of the thread-block cluster kernels.
#include "cluster.cuh"

namespace gbx {

static void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int blocks, int threads, size_t smem,
                           cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

gbx_status cluster_fit(const void* fn, int threads, size_t smem, int* blocks) {
    GBX_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    *blocks = -1;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        for (int c = kClusterMax; c >= 8 && *blocks < 0; c >>= 1) {
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute at[1];
            cluster_config(cfg, at, c, threads, smem, nullptr);
            int k = 0;
            if (cudaOccupancyMaxActiveClusters(&k, fn, &cfg) == cudaSuccess && k >= 1) *blocks = c;
        }
    cudaGetLastError();  // a size that does not fit is no error of this call
    return GBX_OK;
}

gbx_status cluster_launch(const void* fn, int blocks, int threads, size_t smem, void** args, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, blocks, threads, smem, s);
    GBX_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
    return GBX_OK;
}

}  // namespace gbx
