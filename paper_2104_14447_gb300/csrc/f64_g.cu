// f64_g.cu -- instantiations of the FP64 stencil kernel: staggered.
// (Kernel in stencil_f64.cuh; split over several files so they compile in parallel.)
#include "stencil_f64.cuh"

namespace gmls {
extern const F64Entry kF64G[] = {GMLS_F64(2, 2, 2, 4, 24), GMLS_F64(2, 2, 3, 4, 20), GMLS_F64(2, 2, 4, 4, 16), GMLS_F64(2, 3, 2, 4, 16)};
extern const int kF64GCount = sizeof(kF64G) / sizeof(kF64G[0]);
}  // namespace gmls
