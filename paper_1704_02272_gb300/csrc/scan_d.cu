// Instances of the dense scan kernel: prefix entries through L2 or in shared
// memory.
#include "kernels_d.cuh"

namespace pfac {

void *scan_kernel_d(bool entries_in_smem) {
    return entries_in_smem ? (void *)k_scand<1> : (void *)k_scand<0>;
}

}  // namespace pfac
