// f64_d2.cu -- instantiations of the FP64 stencil kernel: divergence-free 2D.
// (Kernel in stencil_f64.cuh; split over several files so they compile in parallel.)
#include "stencil_f64.cuh"

namespace gmls {
extern const F64Entry kF64D2[] = {GMLS_F64(1, 2, 2, 4, 24), GMLS_F64(1, 2, 3, 4, 20), GMLS_F64(1, 2, 4, 4, 16)};
extern const int kF64D2Count = sizeof(kF64D2) / sizeof(kF64D2[0]);
}  // namespace gmls
