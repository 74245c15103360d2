// sne_n2.cu -- instantiations of the semi-normal-equation stencil kernel: scalar 2D with the Neumann constraint.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneN2[] = {GMLS_SNE(0, 2, 2, 3, 8, 12, 4, true, 384),
                              GMLS_SNE(0, 2, 3, 3, 8, 20, 4, true, 384),
                              GMLS_SNE(0, 2, 4, 3, 8, 36, 2, true, 384)};
extern const int kSneN2Count = sizeof(kSneN2) / sizeof(kSneN2[0]);
}  // namespace gmls
