// sne_n3.cu -- instantiations of the semi-normal-equation stencil kernel: scalar 3D with the Neumann constraint.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneN3[] = {GMLS_SNE(0, 3, 2, 4, 8, 20, 2, true, 384),
                              GMLS_SNE(0, 3, 3, 4, 8, 20, 2, true, 384),
                              GMLS_SNE(0, 3, 4, 4, 16, 28, 2, true, 256)};
extern const int kSneN3Count = sizeof(kSneN3) / sizeof(kSneN3[0]);
}  // namespace gmls
