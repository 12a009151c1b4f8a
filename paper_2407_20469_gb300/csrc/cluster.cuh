// cluster.cuh - kernels whose unit of work is taken by one block or by a cluster of K
// blocks: device helpers, set-up and launch (K = 1: plain blocks).
#pragma once

#include "common.cuh"

namespace apic {

__device__ __forceinline__ uint32_t cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cta_count() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Barrier of all threads of the unit's blocks (release / acquire at cluster scope); a
// block barrier without a cluster.
template <bool CL>
__device__ __forceinline__ void tile_sync() {
    if constexpr (!CL) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// Load of global data that another block of the cluster may have written: from L2.
template <bool CL, class T>
__device__ __forceinline__ T ldx(const T* p) {
    if constexpr (CL)
        return __ldcg(p);
    else
        return *p;
}

// Stores a value at this address of shared memory in the cluster's first block.
template <class T>
__device__ __forceinline__ void st_first(T* p, T v) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    if constexpr (sizeof(T) == 8)
        asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(*reinterpret_cast<long long*>(&v)) : "memory");
    else
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(*reinterpret_cast<int*>(&v)) : "memory");
}

inline void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int K, int slots, int threads,
                           size_t smem, cudaStream_t st) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = K;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(K * slots, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = K > 1 ? 1 : 0;
}

// Blocks (K = 1) or clusters of K blocks of kernel f that run at once on the current
// device, 0 on error; raises the kernel's shared-memory limit.
inline int cluster_slots(const void* f, int threads, size_t smem, int K) {
    if (!f || raise_smem_limit(f, smem) != cudaSuccess) return 0;
    if (K == 1) {
        int occ = 0, dev = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, threads, smem) != cudaSuccess ||
            cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 0;
        return occ * sms;
    }
    if (K > 8 && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cluster_config(cfg, attr, K, 256, threads, smem, nullptr);
    int clusters = 0;
    return cudaOccupancyMaxActiveClusters(&clusters, f, &cfg) == cudaSuccess ? clusters : 0;
}

template <class... P, class... A>
cudaError_t cluster_launch(void (*f)(P...), int K, int slots, int threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cluster_config(cfg, attr, K, slots, threads, smem, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, f, args...);
    if (e != cudaSuccess) cudaGetLastError();       // returned here, not by a later launch's check as well
    return e;
}

}  // namespace apic
