// sne_s3b.cu -- instantiations of the semi-normal-equation stencil kernel: scalar 3D, degree 4.
// (Kernel in stencil_sne.cuh; split over several files so they compile in parallel.)
#include "stencil_sne.cuh"

namespace gmls {
extern const SneEntry kSneS3b[] = {GMLS_SNE(0, 3, 4, 3, 16, 28, 2, false, 256),
                              GMLS_SNE(0, 3, 4, 4, 16, 28, 2, false, 256)};
extern const int kSneS3bCount = sizeof(kSneS3b) / sizeof(kSneS3b[0]);
}  // namespace gmls
