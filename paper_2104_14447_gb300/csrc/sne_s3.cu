// sne_s3.cu -- instantiations of the semi-normal-equation stencil kernel: scalar 3D, degrees 2 and 3.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneS3[] = {GMLS_SNE(0, 3, 2, 3, 8, 20, 4, false, 384),
                              GMLS_SNE(0, 3, 2, 4, 8, 20, 4, false, 384),
                              GMLS_SNE(0, 3, 3, 3, 8, 20, 2, false, 384),
                              GMLS_SNE(0, 3, 3, 4, 8, 20, 2, false, 384)};
extern const int kSneS3Count = sizeof(kSneS3) / sizeof(kSneS3[0]);
}  // namespace gmls
