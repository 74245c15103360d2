// f64_s2.cu -- instantiations of the FP64 stencil kernel: scalar 2D.
// (Kernel in stencil_f64.cuh; split over several files so they compile in parallel.)
#include "stencil_f64.cuh"

namespace gmls {
extern const F64Entry kF64S2[] = {GMLS_F64(0, 2, 2, 4, 12), GMLS_F64(0, 2, 3, 4, 20), GMLS_F64(0, 2, 4, 4, 20)};
extern const int kF64S2Count = sizeof(kF64S2) / sizeof(kF64S2[0]);
}  // namespace gmls
