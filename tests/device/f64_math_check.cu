// f64_rsqrt and f64_rcp against the quotients in extended precision on the host
// (tests/test_gpu_device_checks.py builds this): the largest errors in units of the
// last place over exponents of -290 to 290 decimal orders.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "stencil_f64.cuh"

__global__ void eval(const double* x, double* rs, double* rc, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    rs[i] = gmls::f64_rsqrt(x[i]);
    rc[i] = gmls::f64_rcp(x[i]);
  }
}

static double ulps(double got, long double want) {
  int e;
  std::frexp((double)want, &e);
  return (double)std::fabs(((long double)got - want) / std::ldexp(1.0L, e - 53));
}

int main() {
  static_assert(sizeof(long double) > sizeof(double), "a reference of more than 53 bits");
  std::vector<double> x;
  unsigned long long s = 88172645463325252ull;
  for (int e = -963; e <= 963; ++e)
    for (int i = 0; i < 400; ++i) {
      s ^= s << 13, s ^= s >> 7, s ^= s << 17;  // (Marsaglia's xorshift)
      unsigned long long man = s >> 12;
      if (i == 0) man = 0;
      if (i == 1) man = (1ull << 52) - 1;
      if (i == 2) man = (1ull << 32) - 1;  // the bits below those the approximations read
      if (i == 3) man = ~((1ull << 32) - 1) & ((1ull << 52) - 1);
      const unsigned long long b = (unsigned long long)(e + 1023) << 52 | man;
      double v;
      std::memcpy(&v, &b, sizeof(v));
      x.push_back(v);
    }
  const int n = (int)x.size();
  double *dx, *ds, *dc;
  cudaMalloc(&dx, n * sizeof(double));
  cudaMalloc(&ds, n * sizeof(double));
  cudaMalloc(&dc, n * sizeof(double));
  cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
  eval<<<(n + 255) / 256, 256>>>(dx, ds, dc, n);
  std::vector<double> rs(n), rc(n);
  cudaMemcpy(rs.data(), ds, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (cudaMemcpy(rc.data(), dc, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  double es = 0.0, ec = 0.0;
  for (int i = 0; i < n; ++i) {
    es = std::fmax(es, ulps(rs[i], 1.0L / std::sqrt((long double)x[i])));
    ec = std::fmax(ec, ulps(rc[i], 1.0L / (long double)x[i]));
    if (!std::isfinite(rs[i]) || !std::isfinite(rc[i])) es = ec = INFINITY;
  }
  std::printf("%.3f %.3f\n", es, ec);
  return 0;
}
