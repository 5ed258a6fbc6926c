// Instances of the resolver kernels, one per record format.
#include "kernels_w.cuh"

namespace pfac {

void *resolve_kernel(int w) {
    switch (w) {
        case 0: return (void *)k_resolve<0>;
        case 1: return (void *)k_resolve<1>;
        case 2: return (void *)k_resolve<2>;
        case 3: return (void *)k_resolve<3>;
        case 8: return (void *)k_resolve<8>;
        default: return nullptr;
    }
}

void *wresolve_kernel(int w) {
    switch (w) {
        case 0: return (void *)k_wresolve<0, 0>;
        case 1: return (void *)k_wresolve<1, 0>;
        case 2: return (void *)k_wresolve<2, 0>;
        case 3: return (void *)k_wresolve<3, 0>;
        case 8: return (void *)k_wresolve<8, 0>;
        default: return nullptr;
    }
}

// pending records of the dense scan kernel (2-bit symbols)
void *dresolve_kernel(int w) {
    switch (w) {
        case 0: return (void *)k_wresolve<0, 1>;
        case 1: return (void *)k_wresolve<1, 1>;
        case 3: return (void *)k_wresolve<3, 1>;
        default: return nullptr;
    }
}

}  // namespace pfac
