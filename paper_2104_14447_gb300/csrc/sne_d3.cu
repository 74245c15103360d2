// sne_d3.cu -- instantiations of the semi-normal-equation stencil kernel: divergence-free 3D, degrees 2 and 3.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneD3[] = {GMLS_SNE(1, 3, 2, 3, 8, 44, 2, false, 384),
                              GMLS_SNE(1, 3, 3, 3, 16, 40, 2, false, 384)};
extern const int kSneD3Count = sizeof(kSneD3) / sizeof(kSneD3[0]);
}  // namespace gmls
