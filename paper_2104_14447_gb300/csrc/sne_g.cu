// sne_g.cu -- instantiations of the semi-normal-equation stencil kernel: staggered.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneG[] = {GMLS_SNE(2, 2, 2, 3, 8, 12, 4, false, 384),
                              GMLS_SNE(2, 2, 3, 3, 8, 36, 2, false, 384),
                              GMLS_SNE(2, 2, 4, 3, 8, 24, 2, false, 384),
                              GMLS_SNE(2, 3, 2, 4, 8, 20, 2, false, 384),
                              GMLS_SNE(2, 2, 2, 1, 8, 12, 2, false, 384),
                              GMLS_SNE(2, 2, 3, 1, 8, 36, 2, false, 384)};
extern const int kSneGCount = sizeof(kSneG) / sizeof(kSneG[0]);
}  // namespace gmls
