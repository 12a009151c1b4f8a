// kernels_dfc256.cu - the cluster darkfield kernel (dfc.cuh) of 256-pixel tiles.
#include "dfc.cuh"

namespace apic {

ClKernel cl_kernel_256(int B) {
    if (B == 12) return k_darkfield_cluster<16, 12>;
    if (B == 16) return k_darkfield_cluster<16, 16>;
    return nullptr;
}

}  // namespace apic
