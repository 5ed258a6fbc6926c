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
        case 0: return (void *)k_wresolve<0>;
        case 1: return (void *)k_wresolve<1>;
        case 2: return (void *)k_wresolve<2>;
        case 3: return (void *)k_wresolve<3>;
        case 8: return (void *)k_wresolve<8>;
        default: return nullptr;
    }
}

}  // namespace pfac
