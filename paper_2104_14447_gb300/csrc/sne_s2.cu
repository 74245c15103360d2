// sne_s2.cu -- instantiations of the semi-normal-equation stencil kernel: scalar 2D.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneS2[] = {GMLS_SNE(0, 2, 2, 2, 8, 12, 2, false, 512),
                              GMLS_SNE(0, 2, 2, 3, 8, 12, 4, false, 512),
                              GMLS_SNE(0, 2, 3, 2, 8, 20, 2, false, 512),
                              GMLS_SNE(0, 2, 3, 3, 8, 20, 4, false, 384),
                              GMLS_SNE(0, 2, 4, 2, 8, 36, 2, false, 384),
                              GMLS_SNE(0, 2, 4, 3, 8, 36, 2, false, 384)};
extern const int kSneS2Count = sizeof(kSneS2) / sizeof(kSneS2[0]);
}  // namespace gmls
