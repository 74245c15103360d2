// f64.cu -- dispatch of the FP64 stencil kernel (stencil_f64.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "stencil_f64.cuh"

namespace gmls {

#define GMLS_F64_TABLES(X) X(S2) X(D2) X(D3)
#define GMLS_F64_DECL(T)            \
  extern const F64Entry kF64##T[];  \
  extern const int kF64##T##Count;
GMLS_F64_TABLES(GMLS_F64_DECL)

namespace {

struct F64Table {
  const F64Entry* e;
  const int* n;
};
#define GMLS_F64_ROW(T) {kF64##T, &kF64##T##Count},
const F64Table kTables[] = {GMLS_F64_TABLES(GMLS_F64_ROW)};

const F64Entry* f64_entry(int kind, int dim, int deg, int L) {
  for (const F64Table& t : kTables)
    for (int i = 0; i < *t.n; ++i) {
      const F64Entry& e = t.e[i];
      if (e.kind == kind && e.dim == dim && e.deg == deg && L >= 1 && L <= e.lmax) return &e;
    }
  return nullptr;
}

constexpr size_t kSmemPerBlock = 227 * 1024;

int f64_kp(int kmax) { return (kmax + 3) & ~3; }

size_t warp_bytes(const F64Entry& e, int kp) { return (size_t)(32 / e.G) * e.stride(kp) * sizeof(double); }

}  // namespace

bool f64_path_available(int kind, int dim, int deg, int kmax, int L) {
  const F64Entry* e = f64_entry(kind, dim, deg, L);
  return e && warp_bytes(*e, f64_kp(kmax)) <= kSmemPerBlock;
}

// targets in flight on the whole chip (0: not available)
int64_t f64_wave_targets(int kind, int dim, int deg, int kmax, int L, int sms) {
  const F64Entry* e = f64_entry(kind, dim, deg, L);
  if (!e) return 0;
  const size_t w = std::min<size_t>(kSmemPerBlock / warp_bytes(*e, f64_kp(kmax)), (size_t)e->maxt / 32);
  return (int64_t)w * (32 / e->G) * sms;
}

// One block per SM of as many warps as its registers and shared memory allow,
// fewer when there are not enough targets to give every SM such a block.
cudaError_t launch_stencils_f64(const Launch& L, const StencilJob& j, int deg, int kmax, int sms) {
  const F64Entry* e = f64_entry(j.kind, j.dim, deg, j.L);
  if (!e || !j.gen_items || !j.gen_count || !whole_half_power(j)) return cudaErrorInvalidValue;
  int kp = f64_kp(kmax);
  const size_t wb = warp_bytes(*e, kp);
  int64_t w = (int64_t)std::min<size_t>(kSmemPerBlock / wb, (size_t)e->maxt / 32);
  if (w < 1) return cudaErrorInvalidConfiguration;
  const int64_t gpw = 32 / e->G, warps = (j.n_tgt + gpw - 1) / gpw;
  w = std::max<int64_t>(1, std::min(w, (warps + sms - 1) / sms));
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (warps + w - 1) / w));
  cudaError_t r = cudaFuncSetAttribute(e->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemPerBlock);
  if (r != cudaSuccess) return r;
  const F64Tab tab = e->tab();
  void* args[] = {(void*)&j, (void*)&tab, (void*)&kp};
  r = cudaLaunchKernel(e->fn, dim3(grid), dim3((unsigned)(32 * w)), args, (size_t)w * wb, L.stream);
  *L.counter += 1;
  return r;
}

}  // namespace gmls
