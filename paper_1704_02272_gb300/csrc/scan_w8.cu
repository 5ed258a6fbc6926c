// Instances of the window kernel with stride 8.
#include "kernels_w.cuh"

namespace pfac {

template <int TB>
static void *pick(bool packed, uint32_t nb, bool g5) {
    if (g5) return nullptr;
    switch ((packed ? 4u : 0u) + nb) {
        case 1: return (void *)k_scanw<0, 8, 1, 0, TB>;
        case 2: return (void *)k_scanw<0, 8, 2, 0, TB>;
        case 3: return (void *)k_scanw<0, 8, 3, 0, TB>;
        case 5: return (void *)k_scanw<1, 8, 1, 0, TB>;
        case 6: return (void *)k_scanw<1, 8, 2, 0, TB>;
        default: return nullptr;
    }
}

void *scan_kernel_w8(bool packed, uint32_t nb, bool g5, int tb) {
    if (tb == WT_L2) return pick<WT_L2>(packed, nb, g5);
    return tb == WT_ONE ? pick<WT_ONE>(packed, nb, g5) : pick<WT_COPIES>(packed, nb, g5);
}

}  // namespace pfac
