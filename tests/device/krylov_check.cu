// Launches of GMRES iterations queued past the end of a cycle leave every vector
// as it is (tests/test_gpu_device_checks.py builds this against libgmls.so).
#include <cstdio>
#include <vector>

#include "gmls_internal.cuh"

using namespace gmls;

int main() {
  const int64_t n = 5000;
  const int m = 12;
  int64_t launches = 0;
  const Launch L{nullptr, &launches};
  double *w, *z, *dinv, *a;
  int32_t* flags;
  cudaMalloc(&w, n * sizeof(double));
  cudaMalloc(&z, n * sizeof(double));
  cudaMalloc(&dinv, n * sizeof(double));
  cudaMalloc(&a, 4096 * sizeof(double));
  cudaMalloc(&flags, 2 * sizeof(int32_t));
  const std::vector<double> ones(n, 1.0), sevens(n, 7.0), st0(4096, 0.5);
  GmresState st;
  st.H = a;
  st.cs = a + 1024;
  st.sn = a + 1100;
  st.g = a + 1200;
  st.h1 = a + 1300;
  st.h2 = a + 1400;
  st.nrm2 = a + 1500;
  st.jdone = flags;
  st.done = flags + 1;
  int bad = 0;
  // the cycle ended with iteration 2 (three of them): iterations 3 and later do
  // nothing, also to what iteration 2 left
  for (int j = 3; j < 9; ++j) {
    const int32_t f[2] = {3, 3};
    cudaMemcpy(flags, f, sizeof(f), cudaMemcpyHostToDevice);
    cudaMemcpy(w, sevens.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(z, sevens.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(dinv, ones.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(a, st0.data(), 4096 * sizeof(double), cudaMemcpyHostToDevice);
    if (krylov_step(L, n, j, m, w, dinv, z, st, 1e-12) != cudaSuccess) return 2;
    std::vector<double> hw(n), hz(n), ha(4096);
    int32_t g[2];
    cudaMemcpy(hw.data(), w, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaMemcpy(hz.data(), z, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaMemcpy(ha.data(), a, 4096 * sizeof(double), cudaMemcpyDeviceToHost);
    if (cudaMemcpy(g, flags, sizeof(g), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    bad += hw != sevens || hz != sevens || ha != st0 || g[0] != 3 || g[1] != 3;
  }
  std::printf("%d of 6 iterations past the end of a cycle wrote something\n", bad);
  return bad ? 1 : 0;
}
