// krylov.cu -- restarted GMRES on the GPU for the collocation system of
// Sec. 3.2 (the global solve of Sec. 3.3; the paper uses a block-
// preconditioned Krylov method, this is a plain right-Jacobi-preconditioned
// GMRES(m), optionally on the row-equilibrated system R A D y = R b).
//
// Vectors are FP64 device arrays.  The Krylov basis V ([m + 1][n], basis
// vector i contiguous) lives in the context arena.  Orthogonalisation is
// classical Gram-Schmidt applied twice (CGS2).  An iteration is six launches:
// A z (rows scaled on the way out), dots, update, dots, update with the norm, and
// the new basis vector with its preconditioned copy; every reduction ends in the
// block that finishes last, and the Hessenberg column's Givens rotations run
// beside the normalisation on the device.  The host queues kGmresChunk iterations
// ahead and reads their columns and whether the solve has converged; the launches of
// iterations queued past that point return at once.  (One column read back per iteration and a
// single-block sum of 304 partials per column took 270 us an iteration on 55,297
// unknowns, of which the matrix and the basis need about 20.)
// Every reduction has a fixed order (partial sums over fixed row ranges, then
// lanes over the partials and a butterfly), so a solve is reproducible bit for
// bit.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "gmls_internal.cuh"

namespace gmls {

namespace {

constexpr int kDotThreads = 128;   // small blocks: an even share of the FP64 work per SM at 50,000 rows
constexpr int kDotChunk = 8;       // basis vectors per block of the dots
constexpr int kDotRows = 1024;     // rows per block, up to kDotMaxBlocks row ranges
constexpr int kAxpyThreads = 128;
constexpr int kDotMaxBlocks = 272;  // (with these partials and the columns of one chunk a solve needs no more of
                                    // the arena than it did with 304 partials and one column)

// row ranges of the dots: a function of n alone, so the summation order does not
// depend on the device
int dot_ranges(int64_t n) {
  const int64_t b = (n + kDotRows - 1) / kDotRows;
  return (int)(b < 1 ? 1 : b > kDotMaxBlocks ? kDotMaxBlocks : b);
}

// blocks of the updates, a function of n alone too (the order of the norm's sum)
constexpr int kAxpyMaxBlocks = 2432;
unsigned axpy_blocks(int64_t n) {
  const int64_t b = (n + kAxpyThreads - 1) / kAxpyThreads;
  return (unsigned)(b < 1 ? 1 : b > kAxpyMaxBlocks ? kAxpyMaxBlocks : b);
}

__device__ __forceinline__ double warp_sum(double s) {
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// true in the block that arrives last (its reads see every block's writes); the
// counter is back at zero for the next launch
__device__ __forceinline__ bool last_block(int32_t* counter, int blocks) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1) == blocks - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// out[i] = V_i . w (i < ncols): block (b, c) takes row range b and kDotChunk
// columns; the last block adds the ranges' partials
__global__ void __launch_bounds__(kDotThreads) multi_dot_kernel(int64_t n, int ncols, const double* __restrict__ V,
                                                                const double* __restrict__ w,
                                                                double* __restrict__ partial, double* __restrict__ out,
                                                                int32_t* counter, const int32_t* __restrict__ done) {
  __shared__ double red[kDotThreads / 32][kDotChunk];
  if (done && *done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nr = gridDim.x, i0 = blockIdx.y * kDotChunk;
  const int64_t a = n * blockIdx.x / nr, e = n * (blockIdx.x + 1) / nr;
  double acc[kDotChunk];
#pragma unroll
  for (int c = 0; c < kDotChunk; ++c) acc[c] = 0.0;
#pragma unroll 2
  for (int64_t p = a + threadIdx.x; p < e; p += kDotThreads) {
    const double wp = w[p];
#pragma unroll
    for (int c = 0; c < kDotChunk; ++c)
      if (i0 + c < ncols) acc[c] = fma(V[(int64_t)(i0 + c) * n + p], wp, acc[c]);
  }
  // recursive halving over the lanes: 9 FP64 additions a lane instead of the 40
  // of eight butterflies, which cost more than the dots themselves at 1/64 of the
  // FP32 rate; total c ends on lane 4 c
  static_assert(kDotChunk == 8, "three halving stages");
#pragma unroll
  for (int st = 0; st < 3; ++st) {
    const int o = 16 >> st, h = 4 >> st;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int c = 0; c < h; ++c) {
      const double send = up ? acc[c] : acc[c + h];
      acc[c] = (up ? acc[c + h] : acc[c]) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
  if ((lane & 3) == 0) red[warp][lane >> 2] = acc[0];
  __syncthreads();
  if (threadIdx.x < kDotChunk && i0 + (int)threadIdx.x < ncols) {
    double s = 0.0;
    for (int wi = 0; wi < kDotThreads / 32; ++wi) s += red[wi][threadIdx.x];
    partial[(int64_t)(i0 + threadIdx.x) * nr + blockIdx.x] = s;
  }
  if (!last_block(counter, gridDim.x * gridDim.y)) return;
  // four lanes a column
  const int quad = threadIdx.x & 3;
  for (int i = threadIdx.x >> 2; i - (int)(threadIdx.x >> 2) < ncols; i += kDotThreads / 4) {
    double s = 0.0;
    if (i < ncols) {
#pragma unroll 8
      for (int b = quad; b < nr; b += 4) s += __ldcg(partial + (int64_t)i * nr + b);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (i < ncols && quad == 0) out[i] = s;
  }
}

// w -= sum_i h[i] V_i   (i < ncols); NORM: out = |w|^2 after it (the last block
// adds the blocks' partials)
template <bool NORM>
__global__ void __launch_bounds__(kAxpyThreads) multi_axpy_kernel(int64_t n, int ncols, const double* __restrict__ V,
                                                         const double* __restrict__ h, double* __restrict__ w,
                                                         double* __restrict__ partial, double* __restrict__ out,
                                                         int32_t* counter, const int32_t* __restrict__ done) {
  __shared__ double red[kAxpyThreads / 32], hs[258];
  if (done && *done) return;
  for (int i = threadIdx.x; i < ncols; i += blockDim.x) hs[i] = -h[i];
  __syncthreads();
  double nn = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    double s = w[p];
#pragma unroll 8
    for (int i = 0; i < ncols; ++i) s = fma(hs[i], __ldg(V + (int64_t)i * n + p), s);
    w[p] = s;
    if (NORM) nn = fma(s, s, nn);
  }
  if (NORM) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    nn = warp_sum(nn);
    if (lane == 0) red[warp] = nn;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int i = 0; i < kAxpyThreads / 32; ++i) s += red[i];
      partial[blockIdx.x] = s;
    }
    if (!last_block(counter, gridDim.x)) return;
    if (warp == 0) {
      double s = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(partial + b);
      s = warp_sum(s);
      if (lane == 0) *out = s;
    }
  }
}

// End of iteration j: v_{j+1} = w / |w| in place and z = dinv .* v_{j+1}; the
// last block applies the earlier rotations to the new Hessenberg column, forms
// the next one and the residual estimate, and sets done to j + 1 when that is at
// most target (or w vanished).  The other blocks see zero or j + 1 there in the
// iteration that ends the cycle, and leave in those queued after it.
__global__ void __launch_bounds__(256) arnoldi_step_kernel(int64_t n, int j, int m, double* __restrict__ w,
                                                           const double* __restrict__ dinv, double* __restrict__ z,
                                                           GmresState st, double target) {
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double h[258], cs[256], sn[256], ch[256], sh[256];
    if (*st.done) return;  // set by an earlier iteration: this block alone writes it
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
      h[i] = st.h1[i] + st.h2[i];
      cs[i] = i < j ? st.cs[i] : 0.0;
      sn[i] = i < j ? st.sn[i] : 0.0;
    }
    const double hn = sqrt(fmax(*st.nrm2, 0.0));
    __syncthreads();
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
      ch[i] = cs[i] * h[i + 1];
      sh[i] = sn[i] * h[i + 1];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double prev = h[0];
      // previous rotations, one dependent FMA each
#pragma unroll 4
      for (int i = 0; i < j; ++i) {
        h[i] = fma(cs[i], prev, sh[i]);
        prev = fma(-sn[i], prev, ch[i]);
      }
      const double r = hypot(prev, hn);
      const double c = r > 0.0 ? prev / r : 1.0, s = r > 0.0 ? hn / r : 0.0;
      st.cs[j] = c;
      st.sn[j] = s;
      h[j] = r;
      const double g = st.g[j];
      st.g[j + 1] = -s * g;
      st.g[j] = c * g;
      *st.jdone = j + 1;
      if (fabs(s * g) <= target || !(hn > 0.0)) *st.done = j + 1;
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= j; i += blockDim.x) st.H[(int64_t)(j % kGmresChunk) * (m + 1) + i] = h[i];
    return;
  }
  const int32_t ended = *static_cast<volatile const int32_t*>(st.done);
  if (ended != 0 && ended <= j) return;
  const double hn = sqrt(fmax(*st.nrm2, 0.0));
  if (!(hn > 0.0)) return;
  const double inv = 1.0 / hn;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)(gridDim.x - 1) * blockDim.x) {
    const double v = w[p] * inv;
    w[p] = v;
    z[p] = dinv[p] * v;
  }
}

// start of a cycle: g = (beta, 0, ..), nothing done
__global__ void arnoldi_start_kernel(GmresState st, int m, double beta) {
  for (int i = threadIdx.x; i <= m; i += blockDim.x) st.g[i] = i == 0 ? beta : 0.0;
  if (threadIdx.x == 0) {
    *st.done = 0;
    *st.jdone = 0;
  }
}

// x += dinv .* (sum_i y[i] V_i)
__global__ void update_solution_kernel(int64_t n, int ncols, const double* __restrict__ V,
                                       const double* __restrict__ y, const double* __restrict__ dinv,
                                       double* __restrict__ x) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int i = 0; i < ncols; ++i) s = fma(y[i], V[(int64_t)i * n + p], s);
    x[p] = fma(dinv[p], s, x[p]);
  }
}

// z = dinv .* v
__global__ void scale_kernel(int64_t n, const double* __restrict__ dinv, const double* __restrict__ v,
                             double* __restrict__ z) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    z[p] = dinv[p] * v[p];
}

// dst = src * s
__global__ void scaled_copy_kernel(int64_t n, const double* __restrict__ src, double s, double* __restrict__ dst) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    dst[p] = src[p] * s;
}

// r = b - r (r holds A x on entry)
__global__ void residual_kernel(int64_t n, const double* __restrict__ b, double* __restrict__ r) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    r[p] = b[p] - r[p];
}

// dinv[r] = 1 / A[r][r] (1 where the diagonal entry is absent or zero).  A
// row may list column r more than once; as in A x, the entries add up, so
// the diagonal is their sum (the same in both scalings).
// SCALE, row equilibration: rinv[r] = 1 / max_j |A[r][j]| (1 for an empty or
// zero row), and dinv[r] = 1 / (rinv[r] A[r][r]), the Jacobi scaling of the
// equilibrated matrix (1 where that diagonal entry is absent or zero).
// Eight lanes a row; a row of more than kRowLong entries (the zero-mean row of
// the Stokes system) by the whole block (a thread a row took 1.6 ms on a row of
// 13,824 entries).
constexpr int64_t kRowLong = 2048;
template <bool SCALE>
__global__ void __launch_bounds__(256) row_scales_kernel(int64_t n, const int64_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col, const double* __restrict__ val,
                                                         double* __restrict__ rinv, double* __restrict__ dinv) {
  __shared__ double ra[8], rd[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = threadIdx.x & 7;
  auto finish = [&](int64_t r, double amax, double d) {
    const double ri = SCALE ? (amax > 0.0 ? 1.0 / amax : 1.0) : 1.0;
    const double ds = SCALE ? ri * d : d;
    if (SCALE) rinv[r] = ri;
    dinv[r] = ds != 0.0 ? 1.0 / ds : 1.0;
  };
  for (int64_t r0 = blockIdx.x * 32ll; r0 < n; r0 += gridDim.x * 32ll) {
    const int64_t r = r0 + (threadIdx.x >> 3);
    double amax = 0.0, d = 0.0;
    int64_t a = 0, e = 0;
    if (r < n) {
      a = row_ptr[r];
      e = row_ptr[r + 1];
    }
    const bool is_long = e - a > kRowLong;
    if (!is_long)
      for (int64_t p = a + sub; p < e; p += 8) {
        if (SCALE) amax = fmax(amax, fabs(val[p]));
        if (col[p] == (int32_t)r) d += val[p];
      }
    for (int o = 4; o > 0; o >>= 1) {
      amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      d += __shfl_xor_sync(0xffffffffu, d, o);
    }
    if (r < n && !is_long && sub == 0) finish(r, amax, d);
    if (!__syncthreads_or(is_long)) continue;
    for (int q = 0; q < 32 && r0 + q < n; ++q) {
      const int64_t la = row_ptr[r0 + q], le = row_ptr[r0 + q + 1];
      if (le - la <= kRowLong) continue;
      amax = d = 0.0;
      for (int64_t p = la + threadIdx.x; p < le; p += blockDim.x) {
        if (SCALE) amax = fmax(amax, fabs(val[p]));
        if (col[p] == (int32_t)(r0 + q)) d += val[p];
      }
      for (int o = 16; o > 0; o >>= 1) {
        amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        d += __shfl_xor_sync(0xffffffffu, d, o);
      }
      __syncthreads();
      if (lane == 0) {
        ra[warp] = amax;
        rd[warp] = d;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
          ra[0] = fmax(ra[0], ra[w]);
          rd[0] += rd[w];
        }
        finish(r0 + q, ra[0], rd[0]);
      }
    }
    __syncthreads();
  }
}

// v = d .* v
__global__ void scale_in_place_kernel(int64_t n, const double* __restrict__ d, double* v,
                                      const int32_t* __restrict__ done) {
  if (done && *done) return;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    v[p] = d[p] * v[p];
}

unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > (int64_t)device_sm_count() * 16) b = (int64_t)device_sm_count() * 16;
  return (unsigned)b;
}

}  // namespace

cudaError_t krylov_dots(const Launch& L, int64_t n, int ncols, const double* V, const double* w, double* partial,
                        double* out, int32_t* counter, const int32_t* done) {
  const dim3 grid(dot_ranges(n), (ncols + kDotChunk - 1) / kDotChunk);
  multi_dot_kernel<<<grid, kDotThreads, 0, L.stream>>>(n, ncols, V, w, partial, out, counter, done);
  *L.counter += 1;
  return cudaGetLastError();
}

size_t krylov_partial_elems(int max_cols) { return (size_t)kDotMaxBlocks * max_cols; }

cudaError_t krylov_axpy(const Launch& L, int64_t n, int ncols, const double* V, const double* h, double* w,
                        const int32_t* done) {
  multi_axpy_kernel<false><<<axpy_blocks(n), kAxpyThreads, 0, L.stream>>>(n, ncols, V, h, w, nullptr, nullptr, nullptr, done);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_axpy_norm(const Launch& L, int64_t n, int ncols, const double* V, const double* h, double* w,
                             double* partial, double* out, int32_t* counter, const int32_t* done) {
  multi_axpy_kernel<true><<<axpy_blocks(n), kAxpyThreads, 0, L.stream>>>(n, ncols, V, h, w, partial, out, counter, done);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_step(const Launch& L, int64_t n, int j, int m, double* w, const double* dinv, double* z,
                        const GmresState& st, double target) {
  arnoldi_step_kernel<<<grid_for(n) + 1, 256, 0, L.stream>>>(n, j, m, w, dinv, z, st, target);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_start(const Launch& L, const GmresState& st, int m, double beta) {
  arnoldi_start_kernel<<<1, 256, 0, L.stream>>>(st, m, beta);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_update(const Launch& L, int64_t n, int ncols, const double* V, const double* y, const double* dinv,
                          double* x) {
  update_solution_kernel<<<grid_for(n), 256, 0, L.stream>>>(n, ncols, V, y, dinv, x);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_scale(const Launch& L, int64_t n, const double* dinv, const double* v, double* z) {
  scale_kernel<<<grid_for(n), 256, 0, L.stream>>>(n, dinv, v, z);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_scaled_copy(const Launch& L, int64_t n, const double* src, double s, double* dst) {
  scaled_copy_kernel<<<grid_for(n), 256, 0, L.stream>>>(n, src, s, dst);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_residual(const Launch& L, int64_t n, const double* b, double* r) {
  residual_kernel<<<grid_for(n), 256, 0, L.stream>>>(n, b, r);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_inverse_diagonal(const Launch& L, int64_t n, const int64_t* row_ptr, const int32_t* col,
                                    const double* val, double* dinv) {
  row_scales_kernel<false><<<grid_for(n * 8), 256, 0, L.stream>>>(n, row_ptr, col, val, nullptr, dinv);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_row_equilibration(const Launch& L, int64_t n, const int64_t* row_ptr, const int32_t* col,
                                     const double* val, double* rinv, double* dinv) {
  row_scales_kernel<true><<<grid_for(n * 8), 256, 0, L.stream>>>(n, row_ptr, col, val, rinv, dinv);
  *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t krylov_scale_in_place(const Launch& L, int64_t n, const double* d, double* v, const int32_t* done) {
  scale_in_place_kernel<<<grid_for(n), 256, 0, L.stream>>>(n, d, v, done);
  *L.counter += 1;
  return cudaGetLastError();
}

}  // namespace gmls
