// sne_d3b.cu -- instantiations of the semi-normal-equation stencil kernel: divergence-free 3D, degree 4.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneD3b[] = {GMLS_SNE(1, 3, 4, 3, 32, 36, 2, false, 256)};
extern const int kSneD3bCount = sizeof(kSneD3b) / sizeof(kSneD3b[0]);
}  // namespace gmls
