// sne_d2.cu -- instantiations of the semi-normal-equation stencil kernel: divergence-free 2D.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneD2[] = {GMLS_SNE(1, 2, 2, 2, 8, 24, 4, false, 384),
                              GMLS_SNE(1, 2, 3, 2, 8, 36, 4, false, 384),
                              GMLS_SNE(1, 2, 4, 2, 8, 24, 2, false, 384)};
extern const int kSneD2Count = sizeof(kSneD2) / sizeof(kSneD2[0]);
}  // namespace gmls
