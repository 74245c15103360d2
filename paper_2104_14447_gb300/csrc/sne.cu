// sne.cu -- dispatch of the semi-normal-equation stencil kernel
// (stencil_sne.cuh).
#include <cuda_runtime.h>

#include "stencil_sne.cuh"

namespace gmls {

#define GMLS_SNE_TABLES(X) X(S2) X(S3) X(S3b) X(N2) X(N3) X(G) X(D2) X(D3) X(D3b)
#define GMLS_SNE_DECL(T)             \
  extern const SneEntry kSne##T[];   \
  extern const int kSne##T##Count;
GMLS_SNE_TABLES(GMLS_SNE_DECL)

namespace {

struct SneTable {
  const SneEntry* e;
  const int* n;
};
#define GMLS_SNE_ROW(T) {kSne##T, &kSne##T##Count},
const SneTable kTables[] = {GMLS_SNE_TABLES(GMLS_SNE_ROW)};

const SneEntry* sne_entry(int kind, int dim, int deg, int L, bool neu) {
  for (const SneTable& t : kTables)
    for (int i = 0; i < *t.n; ++i) {
      const SneEntry& e = t.e[i];
      if (e.kind == kind && e.dim == dim && e.deg == deg && e.L == L && (e.neu != 0) == neu) return &e;
    }
  return nullptr;
}

constexpr size_t kSmemPerBlock = 227 * 1024;

int sne_kp(int kmax) { return (kmax + 3) & ~3; }

size_t warp_bytes(const SneEntry& e, int kp) { return (size_t)(32 / e.G) * e.stride(kp) * sizeof(float); }

}  // namespace

bool sne_path_available(int kind, int dim, int deg, int kmax, int L, bool neu) {
  const SneEntry* e = sne_entry(kind, dim, deg, L, neu);
  return e && warp_bytes(*e, sne_kp(kmax)) <= kSmemPerBlock;
}

// One block per SM of as many warps as its registers (the kernel's thread
// bound) and shared memory allow; fewer warps a block when there are not
// enough targets to give every SM such a block.
cudaError_t sne_launch_shape(int kind, int dim, int deg, int L, bool neu, int kmax, int64_t n_tgt, int sms,
                             SneShape* s) {
  const SneEntry* e = sne_entry(kind, dim, deg, L, neu);
  if (!e) return cudaErrorInvalidValue;
  const int kp = sne_kp(kmax);
  const size_t wb = warp_bytes(*e, kp);
  int64_t w = (int64_t)std::min<size_t>(kSmemPerBlock / wb, (size_t)e->maxt / 32);
  if (w < 1) return cudaErrorInvalidConfiguration;
  const int64_t gpw = 32 / e->G, warps = (n_tgt + gpw - 1) / gpw;
  w = std::max<int64_t>(1, std::min(w, (warps + sms - 1) / sms));
  s->warps = (int)w;
  s->grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (warps + w - 1) / w));
  s->smem = (size_t)w * wb;
  s->scratch = (size_t)s->grid * w * gpw * e->rhs * kp * sizeof(float2);
  s->kp = kp;
  return cudaSuccess;
}

cudaError_t launch_stencils_sne(const Launch& L, const StencilJob& j, int deg, const SneShape& s, bool neu) {
  const SneEntry* e = sne_entry(j.kind, j.dim, deg, j.L, neu);
  if (!e || !j.dscratch || !whole_half_power(j)) return cudaErrorInvalidValue;
  cudaError_t r = cudaFuncSetAttribute(e->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemPerBlock);
  if (r != cudaSuccess) return r;
  const SneTab tab = e->tab();
  int kp = s.kp;
  void* args[] = {(void*)&j, (void*)&tab, (void*)&kp};
  r = cudaLaunchKernel(e->fn, dim3(s.grid), dim3(32 * s.warps), args, s.smem, L.stream);
  *L.counter += 1;
  return r;
}

}  // namespace gmls
