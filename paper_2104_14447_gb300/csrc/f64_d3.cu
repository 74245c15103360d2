// f64_d3.cu -- instantiations of the FP64 stencil kernel: divergence-free 3D.
// (Kernel in stencil_f64.cuh; split over several files so they compile in parallel.)
#include "stencil_f64.cuh"

namespace gmls {
extern const F64Entry kF64D3[] = {GMLS_F64(1, 3, 2, 8, 16), GMLS_F64(1, 3, 4, 16, 12)};
extern const int kF64D3Count = sizeof(kF64D3) / sizeof(kF64D3[0]);
}  // namespace gmls
