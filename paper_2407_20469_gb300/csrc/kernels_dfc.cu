// kernels_dfc.cu - the cluster darkfield kernel (dfc.cuh): tiles of 128 pixels, set-up
// and launch.
#include "dfc.cuh"

namespace apic {

namespace {

ClKernel cl_kernel(const DevPlan& P) {
    const int B = P.mr / 16;
    if (P.h != P.w || P.n_used == 0) return nullptr;
    if (P.h == 256) return cl_kernel_256(B);
    if (P.h == 128 && B == 6) return k_darkfield_cluster<8, 6>;
    if (P.h == 128 && B == 8) return k_darkfield_cluster<8, 8>;
    return nullptr;
}

// Dynamic shared memory of a launch: more than half an SM's, so that one block runs per
// SM (each allocates all of its SM's tensor memory)
size_t cl_smem_bytes(const ClSmem& L) { return std::max(L.total, (size_t)116 * 1024); }

ClSmem cl_layout(const DevPlan& P, int K) {
    return cl_smem_layout(P.h / 16, P.mr / 16, K, P.cl_maxB, P.cl_mx, P.band_u, P.band_p, P.band_q, P.max_N);
}

}  // namespace

size_t dfc_scratch_bytes(const DevPlan& P) {
    return (cl_scratch_layout(P.h, P.mr, P.band_p, P.band_q, P.max_M).total * sizeof(float2) + 255) & ~(size_t)255;
}

int configure_dfc(const DevPlan& P, int K) {
    ClKernel f = cl_kernel(P);
    int dev = 0, most = 0;
    if (!f || K < 2 || K > kMaxCluster || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    const size_t smem = cl_smem_bytes(cl_layout(P, K));
    // TMEM columns of a thread: 32 per round of its columns; 1 KB for the static shared memory
    if (cl_share(cl_share(P.cl_mx, K), kClHW) * 32 > kClTmemSlot || smem + 1024 > (size_t)most) return 0;
    return cluster_slots((const void*)f, kClThreads, smem, K);
}

cudaError_t launch_darkfield_cluster(const DevPlan& P, int K, int slots, int n_tiles, const float* I, const float* phi,
                                     float2* spec, void* scratch, int iters, float tol, int32_t* status,
                                     unsigned long long* counters, cudaStream_t st, DfTiles tiles) {
    ClKernel f = cl_kernel(P);
    slots = std::min(slots, n_tiles);
    if (!f) return cudaErrorInvalidValue;
    if (slots < 1) return cudaErrorInvalidConfiguration;
    const ClSmem L = cl_layout(P, K);
    return cluster_launch(f, K, slots, kClThreads, cl_smem_bytes(L), st, P, L, n_tiles, I, phi, spec, (char*)scratch,
                          dfc_scratch_bytes(P), iters, tol, status, counters, tiles);
}

}  // namespace apic
