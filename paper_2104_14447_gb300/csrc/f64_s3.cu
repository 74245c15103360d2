// f64_s3.cu -- instantiations of the FP64 stencil kernel: scalar 3D.
// (Kernel in stencil_f64.cuh; split over several files so they compile in parallel.)
#include "stencil_f64.cuh"

namespace gmls {
extern const F64Entry kF64S3[] = {GMLS_F64(0, 3, 2, 4, 20), GMLS_F64(0, 3, 3, 4, 16), GMLS_F64(0, 3, 4, 8, 16)};
extern const int kF64S3Count = sizeof(kF64S3) / sizeof(kF64S3[0]);
}  // namespace gmls
