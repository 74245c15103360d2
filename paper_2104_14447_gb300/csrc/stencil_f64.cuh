// stencil_f64.cuh -- GMLS stencils in FP64: R factor in column-owning lanes,
// several targets per warp.
//
// The systems of stencil_sne.cuh in plain FP64: the same columns (orthogonal
// under the target's own weighted neighbours), the same factored form of the
// divergence-free basis (A = Q_A R_A of the scalar columns, then the
// component-0 rows of (I (x) R_A) C against the triangle).  s = B y with y =
// R^-1 R^-T lambda: the semi-normal equations of a least-norm problem, whose
// forward error is O(kappa u) as that of a solve with Q (Paige 1973; Demmel &
// Higham 1993), so Q is neither kept nor applied and no correction is needed.
//
// Bound: the FP64 pipe, two lanes a clock and SM: a warp instruction costs 16
// clocks whether its lanes have work or not, and everything else (shared
// memory, integer work, latency at three or four warps) hides behind it.  So
// the layout counts FP64 warp instructions only:
//  * a target has few lanes (4 for bases up to 20, else 8 or 16), each owning
//    whole columns: no cross-lane additions (the shared-memory kernel's
//    butterflies were a third of its FP64 work) and the triangle's idle lanes
//    cost 4 / n rather than 32 / n;
//  * rows stream through registers P at a time, in chunks of four that a short
//    last block leaves out;
//  * one reflector costs ten FP64 operations: reciprocal square root and
//    reciprocal from the hardware's approximations and one third-order
//    (Householder's method) step each;
//  * the divergence-free systems factor k x Q scalar columns instead of
//    d k x N, 2.4 times fewer operations (2D degree 4).
// Measured (GB300, 32,761 targets, ncu: FP64 pipe 81 to 85 % busy): 2D degree 4
// divergence-free 2.64 ms, scalar 1.39 ms; the operators from cloud to CSR 12.4 ->
// 4.3 ms, of 1,024 targets at degree 2 159 -> 116 us; error against 64-bit
// references unchanged (3.1e-14, 5.9e-16).
// G and P as in stencil_sne.cuh, in FP64: P is what 255 registers hold beside the
// column slots.
// Taken where the error against 64-bit weights is that of a solve with Q within a
// few percent (measured, new / old): 2D scalar 0.9 to 1.07, 2D divergence-free 0.92
// to 1.02, 3D divergence-free degree 2 1.03, degree 4 1.04.  Not built: 3D scalar
// (1.1 to 1.6), 3D divergence-free degree 3 (1.2) and the staggered basis (4 to 8:
// its columns vanish at the target and have no constant to be orthogonal to).
// Not taken besides: Neumann rows, odd weight powers, lists shorter than the basis,
// systems with max / min |r_ii| above 1e5: those targets keep the
// shared-memory kernel (their status bits come from its factor).
#pragma once
#include "stencil_sne.cuh"

namespace gmls {

struct F64Tab {
  SneTab t;
  double mc[72];  // main coefficient of column i's component-0 part
};
template <int D, int LO, int HI>
F64Tab make_f64_tab() {
  F64Tab f{};
  f.t = make_sne_tab<D, LO, HI>();
  constexpr int Q = SneMono<D, LO, HI>::Q;
  if (LO == 0)
    for (int i = 0; i < (D - 1) * Q && i < 72; ++i) {
      const int c = 1 + i / Q, g = i % Q;
      f.mc[i] = (double)f.t.e[c][g] / (double)(f.t.e[0][g] + 1);
    }
  return f;
}

// 1 / sqrt(x) and 1 / x for normal x > 0: the hardware's approximation y
// (about 20 bits) and one step of Householder's third-order iteration,
// y + y e (1/2 + 3/8 e), e = 1 - x y^2, and y + y e (1 + e), e = 1 - x y.  Measured
// over 1e-290 to 1e290: within 0.98 and 0.51 units of the last place (correct
// rounding: 0.5)
__device__ __forceinline__ double f64_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(fma(0.375, e, 0.5), e * y, y);
}
__device__ __forceinline__ double f64_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(fma(e, e, e), y, y);
}

// Householder elimination of 4 nch <= P rows against the packed upper triangle
// R (N columns): sne_append in FP64, a row a register pair.
template <int P, int SN, int N, int G>
__device__ __forceinline__ void f64_append(double (&a)[SN][P], double* R, double* vbuf, int lane, int& par, int nch) {
  constexpr int PV = P + 2;
#pragma unroll
  for (int s = 0; s < SN; ++s) {
    constexpr int last = N - (SN - 1) * G;  // columns of the last slot
    double* rrow = R + rpk<N>(s * G, 0);    // row k of R: entry c at rrow[c]
#pragma unroll 1
    for (int o = 0; o < (s < SN - 1 ? G : last); ++o) {
      const int k = s * G + o;
      double* vb = vbuf + par * PV;
      par ^= 1;
      if (lane == o) {
#pragma unroll
        for (int i = 0; i < P / 2; ++i) reinterpret_cast<double2*>(vb)[i] = make_double2(a[s][2 * i], a[s][2 * i + 1]);
        vb[P] = rrow[k];
      }
      __syncwarp();
      const double alpha = vb[P];
      double d[SN], e[SN];
#pragma unroll
      for (int u = s; u < SN; ++u) d[u] = e[u] = 0.0;
#pragma unroll
      for (int h = 0; h < P / 4; ++h) {
        if (h >= nch) break;
        const double2 p = reinterpret_cast<const double2*>(vb)[2 * h], q = reinterpret_cast<const double2*>(vb)[2 * h + 1];
#pragma unroll
        for (int u = s; u < SN; ++u) {
          d[u] = fma(p.x, a[u][4 * h], d[u]);
          e[u] = fma(p.y, a[u][4 * h + 1], e[u]);
          d[u] = fma(q.x, a[u][4 * h + 2], d[u]);
          e[u] = fma(q.y, a[u][4 * h + 3], e[u]);
        }
      }
#pragma unroll
      for (int u = s; u < SN; ++u) d[u] += e[u];
      const double sig = __shfl_sync(0xffffffffu, d[s], o, G);
      double f = 0.0, v0 = 0.0, beta = alpha;
      const double n2 = fma(alpha, alpha, sig);
      if (sig > 0.0 && n2 > 1e-290) {  // (a smaller column leaves a zero diagonal, which hands the target off)
        const double nrm = n2 * f64_rsqrt(n2);
        beta = alpha >= 0.0 ? -nrm : nrm;
        v0 = alpha - beta;
        f = f64_rcp(nrm * fabs(v0));  // 2 / (v0^2 + sig)
      }
#pragma unroll
      for (int u = s; u < SN; ++u) {
        const bool act = (u > s || lane > o) && (u < SN - 1 || lane < last);
        double* rp = rrow + (act ? u * G + lane : k);
        const double rk = act ? *rp : 0.0;
        d[u] = act ? fma(v0, rk, d[u]) * -f : 0.0;
        if (act) *rp = fma(d[u], v0, rk);
      }
#pragma unroll
      for (int h = 0; h < P / 4; ++h) {
        if (h >= nch) break;
        const double2 p = reinterpret_cast<const double2*>(vb)[2 * h], q = reinterpret_cast<const double2*>(vb)[2 * h + 1];
#pragma unroll
        for (int u = s; u < SN; ++u) {
          a[u][4 * h] = fma(d[u], p.x, a[u][4 * h]);
          a[u][4 * h + 1] = fma(d[u], p.y, a[u][4 * h + 1]);
          a[u][4 * h + 2] = fma(d[u], q.x, a[u][4 * h + 2]);
          a[u][4 * h + 3] = fma(d[u], q.y, a[u][4 * h + 3]);
        }
      }
      if (lane == o) rrow[k] = beta;
      rrow += N - 1 - k;
    }
  }
}

// w <- R^-1 R^-T w; entry p at lane p % G, slot p / G
template <int N, int G, int SN>
__device__ __forceinline__ void f64_solve(const double* R, const double* ID, double (&w)[SN], int lane) {
  const double* rrow = R + lane;
#pragma unroll
  for (int s = 0; s < SN; ++s) {
#pragma unroll 1
    for (int o = 0; o < (s < SN - 1 ? G : N - (SN - 1) * G); ++o) {
      const int i = s * G + o;
      const double yi = __shfl_sync(0xffffffffu, w[s], o, G) * ID[i];
      if (lane == o) w[s] = yi;
#pragma unroll
      for (int u = s; u < SN; ++u) {
        const bool act = (u > s || lane > o) && u * G + lane < N;
        w[u] = fma(act ? -rrow[u * G] : 0.0, yi, w[u]);
      }
      rrow += N - 1 - i;
    }
  }
  const double* rcol[SN];
#pragma unroll
  for (int u = 0; u < SN; ++u) rcol[u] = R + rpk<N>(u * G + lane < N ? u * G + lane : 0, 0);
#pragma unroll
  for (int s = SN - 1; s >= 0; --s) {
#pragma unroll 1
    for (int o = (s < SN - 1 ? G : N - (SN - 1) * G) - 1; o >= 0; --o) {
      const int i = s * G + o;
      const double yi = __shfl_sync(0xffffffffu, w[s], o, G) * ID[i];
      if (lane == o) w[s] = yi;
#pragma unroll
      for (int u = 0; u <= s; ++u) w[u] = fma((u < s || lane < o) ? -rcol[u][i] : 0.0, yi, w[u]);
    }
  }
}

// Shared memory of one group, in doubles
template <int KIND, int D, int DEG, int G, int P>
struct F64Lay {
  using Dm = SneDims<KIND, D, DEG, false>;
  static constexpr bool DF = Dm::DF;
  static constexpr int Q = Dm::Q, N = Dm::N, LMAX = DF ? D : D + 1, RHS = LMAX * Dm::NC, HI1 = Dm::HI + 1;
  __host__ __device__ static constexpr int up2(int v) { return (v + 1) & ~1; }
  __host__ __device__ static constexpr int max2(int a, int b) { return a > b ? a : b; }
  static constexpr int PS = P + 2;  // column stride of the staged block
  static constexpr int R = 0;
  static constexpr int ID = N * (N + 1) / 2;
  static constexpr int LT = ID + N;  // q, q', q'' at the target [D][HI + 1][3]
  static constexpr int LP = LT + 3 * D * HI1;                                   // divergence-free: Laplacians of the columns
  static constexpr int XC = LP + (DF ? Q : 0);                                  // and the coefficients of the further terms
  static constexpr int RA = XC + (DF ? sne_extras(D, DEG) : 0);                 // and R_A
  static constexpr int DST = up2(RA + (DF ? Q * (Q + 1) / 2 : 0));              // SneDst [RHS][2]
  static constexpr int VB = DST + 4 * RHS;                                      // reflectors, two in turn
  static constexpr int ST = VB + 2 * (P + 2);                                   // staged rows; then u and y
  static constexpr int U = ST, Y = U + RHS * Q;
  static constexpr int X = up2(ST + max2(Q * PS, RHS * Q + N));                 // eta [D][kp], sqrt(W) [kp]
  __host__ __device__ static int stride(int kp) { return X + (D + 1) * kp + 2; }  // kp a multiple of four
};

template <int KIND, int D, int DEG, int G, int P, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) stencil_f64_kernel(StencilJob j, const F64Tab ftab, int kp) {
  using Dm = SneDims<KIND, D, DEG, false>;
  using Lay = F64Lay<KIND, D, DEG, G, P>;
  constexpr bool DF = Dm::DF;
  constexpr int LO = Dm::LO, HI = Dm::HI, Q = Dm::Q, N = Dm::N, NC = Dm::NC, NTOP = Dm::NTOP, RHS = Lay::RHS;
  constexpr int SA = (Q + G - 1) / G, SN = (N + G - 1) / G;
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(N == gmls_gen::basis_size(KIND, D, DEG), "basis size");
  static_assert(P % 4 == 0, "chunks of four rows");
  static_assert(KIND != GMLS_BASIS_STAGGERED, "columns orthogonal to a constant");
  extern __shared__ __align__(16) double smd[];
  const SneTab& tab = ftab.t;
  const int lane = threadIdx.x & (G - 1);
  const int gpb = blockDim.x / G, grp = threadIdx.x / G, gpw = 32 / G;
  double* base = smd + (size_t)grp * Lay::stride(kp);
  double *R = base + Lay::R, *ID = base + Lay::ID, *LT = base + Lay::LT, *LP = base + Lay::LP, *XC = base + Lay::XC;
  double *VB = base + Lay::VB, *STG = base + Lay::ST, *U = base + Lay::U, *Y = base + Lay::Y;
  double *X = base + Lay::X, *SW = X + D * kp, *RA = DF ? base + Lay::RA : R;
  SneDst* dst = reinterpret_cast<SneDst*>(base + Lay::DST);
  const int L = j.L;
  const int64_t n = j.n, n_items = j.items ? (int64_t)(*j.n_items) : j.n_tgt;

  for (int64_t ib = (int64_t)blockIdx.x * gpb + (threadIdx.x / 32) * gpw; ib < n_items; ib += (int64_t)gridDim.x * gpb) {
    const int64_t it = ib + (grp & (gpw - 1));
    const bool have = it < n_items;
    const int64_t pos = have ? it : n_items - 1;
    const int64_t to = j.items ? (int64_t)j.items[pos] : pos;
    const int64_t t = j.tgt[to], o0 = j.off[to];
    const int k = (int)(j.off[to + 1] - o0);
    const uint8_t st = j.nbr_status ? j.nbr_status[to] : 0;
    const double eps = j.eps[to];
    // what the shared-memory kernel takes
    bool hand = have && ((st & GMLS_T_TOO_FEW_NEIGHBOURS) || !(eps > 0.0) || k > kp || k < (DF ? Q : N));
    const int ke = have && !hand ? k : 0;
    const int kw = __reduce_max_sync(FULL, ke);  // the longest list in the warp
    if (kw > 0) {
      // ---- 1. eta = (x_j - x_T) / eps, sqrt(W); centroid and moments (any constants
      // near them do: FP32), coefficients of q_2 .. q_HI
      const double inv_eps = 1.0 / eps, ie2 = inv_eps * inv_eps;
      double xt[D];
      float mw = 0.0f, m1[D];
#pragma unroll
      for (int c = 0; c < D; ++c) {
        xt[c] = j.x[c * n + t];
        m1[c] = 0.0f;
      }
      const int kr = (kw + 3) & ~3;
#pragma unroll 2
      for (int q = lane; q < kr; q += G) {
        const int64_t jj = q < ke ? (int64_t)j.idx[o0 + q] : t;
        double dx[D], r2 = 0.0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          dx[c] = j.x[c * n + jj] - xt[c];
          r2 = fma(dx[c], dx[c], r2);
        }
        const double u = fma(-sqrt(r2), inv_eps, 1.0);
        double sw = u;
        for (int p = 1; p < j.wpow_half; ++p) sw *= u;
        if (!(q < ke && u > 0.0)) sw = 0.0;
        const float wt = (float)sw * (float)sw;
        mw += wt;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const double xi = dx[c] * inv_eps;
          X[c * kp + q] = xi;
          m1[c] = fmaf(wt, (float)xi, m1[c]);
        }
        SW[q] = sw;
      }
      mw = 1.0f / gsum<G>(mw);
      float sh[D], mu[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int c = 0; c < D; ++c) sh[c] = gsum<G>(m1[c]) * mw;
#pragma unroll 2
      for (int q = lane; q < kr; q += G) {  // (the rows this lane wrote)
        const float wt = (float)SW[q] * (float)SW[q];
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const double x = X[c * kp + q] - (double)sh[c];
          X[c * kp + q] = x;
          const float s = (float)x * (float)x;
          float p = wt * s;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (e >= HI) break;
            mu[e] += p;
            p *= s;
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) mu[e] = e < HI ? gsum<G>(mu[e]) * (mw / (float)D) : 0.0f;
      SneCoef cf;
      sne_coefficients<HI, false>(mu, cf);
      // q, q', q'' at the target (eta = -centroid): entry (axis, power, derivative)
      __syncwarp();
      if (lane < D) {
        float s0 = sh[0];
#pragma unroll
        for (int c = 1; c < D; ++c)
          if (lane == c) s0 = sh[c];
        const double x = -(double)s0, tt = x * x, a = cf.a, b = cf.b, cc = cf.c, dd = cf.d;
        double* o = LT + lane * 3 * (HI + 1);
        auto put = [&](int p, double v, double d1, double d2) { o[3 * p] = v, o[3 * p + 1] = d1, o[3 * p + 2] = d2; };
        put(0, 1.0, 0.0, 0.0);
        put(1, x, 1.0, 0.0);
        if constexpr (HI >= 2) put(2, tt - a, 2.0 * x, 2.0);
        if constexpr (HI >= 3) put(3, x * (tt - b), 3.0 * tt - b, 6.0 * x);
        if constexpr (HI >= 4) put(4, tt * (tt - cc) + dd, x * (4.0 * tt - 2.0 * cc), 12.0 * tt - 2.0 * cc);
      }
      for (int r = lane; r < L * NC; r += G) {
        const int l = r / NC, cc = r - l * NC;
        SneDst* d = dst + 2 * r;
        int nd = 0;
        d[0].p = d[1].p = nullptr;
        for (int f = 0; f < j.nout; ++f) {
          const int RW = j.out_rows[f], C = j.out_ncomp[f], rr = l - j.out_src[f];
          const bool div = !DF && j.out_fn[f] == GMLS_F_DIV;  // d/dx_c on component c
          if (j.out_src[f] < 0 || rr < 0 || rr >= (div ? C : RW) || nd == 2) continue;
          double* wo = j.out_w[f] + o0 * (int64_t)RW * C;
          d[nd].p = div ? wo + rr : wo + (int64_t)rr * k * NC + cc;
          d[nd].stride = div ? C : NC;
          d[nd].sgn = (float)j.out_sign[f];
          ++nd;
        }
      }
      for (int e = lane; e < Q * (Q + 1) / 2; e += G) RA[e] = 0.0;
      __syncwarp();
      auto lt = [&](int axis, int col, int der) { return LT[(axis * (HI + 1) + tab.e[axis][col]) * 3 + der]; };
      auto lap_col = [&](int col) {  // Laplacian of column col at the target (unscaled)
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          double p = lt(c, col, 2);
#pragma unroll
          for (int c2 = 0; c2 < D; ++c2)
            if (c2 != c) p *= lt(c2, col, 0);
          s += p;
        }
        return s;
      };
      if constexpr (DF) {
        for (int g = lane; g < Q; g += G) LP[g] = lap_col(g);
        for (int x = lane; x < tab.nx; x += G) {  // further terms, as in stencil_sne.cuh
          const int i = tab.xcol[x], c = 1 + i / Q, g = i % Q, g0 = tab.e[0][g], gc = tab.e[c][g];
          const double a = cf.a, b = cf.b, cc = cf.c;
          XC[x] = gc >= 3 ? (gc == 3 ? 3.0 * a - b : 4.0 * b - 2.0 * cc) / (double)(g0 + 1)
                          : (g0 == 2 ? b / 3.0 - a : 0.25 * cc - 0.5 * b) * (double)gc;
        }
      }

      // ---- 2. A = Q_A R_A: blocks of P rows against the triangle
      int par = 0;
#pragma unroll 1
      for (int r0 = 0; r0 < kr; r0 += P) {
        const int nr = min(P, kr - r0);
        __syncwarp();  // the previous block has been read
#pragma unroll 1
        for (int i = lane; i < nr; i += G) {
          double x[D], m[Q];
#pragma unroll
          for (int c = 0; c < D; ++c) x[c] = X[c * kp + r0 + i];
          sne_columns<D, LO, HI>(x, cf, m);
          const double sw = SW[r0 + i];
#pragma unroll
          for (int c = 0; c < Q; ++c) STG[c * Lay::PS + i] = m[c] * sw;
        }
        __syncwarp();
        double a[SA][P];
#pragma unroll
        for (int s = 0; s < SA; ++s) {
          const int c = s * G + lane;
          const double* col = STG + (c < Q ? c : 0) * Lay::PS;
#pragma unroll
          for (int i = 0; i < P; ++i) a[s][i] = i < nr && (s < SA - 1 || c < Q) ? col[i] : 0.0;
        }
        f64_append<P, SA, Q, G>(a, RA, VB, lane, par, nr / 4);
      }
      __syncwarp();
      if constexpr (DF) {
        // ---- 3. G = (I (x) R_A) C: diag(R_A, ..) above, the component-0 rows eliminated against it
        for (int e = lane; e < N * (N + 1) / 2; e += G) R[e] = 0.0;
        __syncwarp();
#pragma unroll
        for (int s = 0; s < SN; ++s) {
          const int col = s * G + lane;
          if (col < NTOP) {
            const int b0 = col / Q * Q, cg = col - b0;
            for (int r = 0; r <= cg; ++r) R[rpk<N>(b0 + r, col)] = RA[rpk<Q>(r, cg)];
          }
        }
#pragma unroll 1
        for (int r0 = 0; r0 < Q; r0 += P) {
          const int nr = min(P, Q - r0);
          double a[SN][P];
#pragma unroll
          for (int s = 0; s < SN; ++s) {
            const int col = s * G + lane;
            int src = -1, xs = -1;
            double cm = 0.0, cx = 0.0;
            if (col < NTOP) {
              src = tab.src[col];
              cm = -ftab.mc[col];
              if (tab.xslot[col] >= 0) {
                xs = tab.xsrc[(int)tab.xslot[col]];
                cx = -XC[(int)tab.xslot[col]];
              }
            } else if (col < N) {
              src = tab.f0[col - NTOP];
              cm = 1.0;
            }
#pragma unroll
            for (int i = 0; i < P; ++i) {
              const int r = r0 + i;
              double v = src >= r ? cm * RA[rpk<Q>(r, src)] : 0.0;
              if (xs >= r) v = fma(cx, RA[rpk<Q>(r, xs)], v);
              a[s][i] = i < nr ? v : 0.0;
            }
          }
          __syncwarp();
          f64_append<P, SN, N, G>(a, R, VB, lane, par, (nr + 3) / 4);
        }
        __syncwarp();
      }
      // 1 / r_ii and the conditioning of the factor on the Taylor scale (1 / b!)
      float dmx = 0.0f, dmn = 3.0e38f;
#pragma unroll
      for (int s = 0; s < SN; ++s) {
        const int p = s * G + lane;
        if (p < N) {
          const double d = R[rpk<N>(p, p)];
          ID[p] = 1.0 / d;
          const int col = DF ? (p < NTOP ? p % Q : tab.f0[p < NTOP ? 0 : p - NTOP]) : p;
          float sc = (float)fabs(d);
#pragma unroll
          for (int c = 0; c < D; ++c) {
            const int e = tab.e[c][col];
            sc *= e < 2 ? 1.0f : e == 2 ? 0.5f : e == 3 ? 1.0f / 6.0f : e == 4 ? 1.0f / 24.0f : 1.0f / 120.0f;
          }
          dmx = fmaxf(dmx, sc);
          dmn = sc > 0.0f ? fminf(dmn, sc) : 0.0f;  // (zero and NaN)
        }
      }
      dmx = gmax<G>(dmx);
      dmn = -gmax<G>(-dmn);
      hand = hand || (have && !(dmn * 1.0e5f >= dmx && dmn > 0.0f));
      __syncwarp();

      // ---- 4. y = R^-1 R^-T lambda, u = C y
#pragma unroll 1
      for (int l = 0; l < L; ++l) {
        const bool second = !DF && j.lam_fn[l] == 1;  // the Laplacian
        const int ax = j.lam_row[l];
        double w[SN];
#pragma unroll
        for (int s = 0; s < SN; ++s) {
          const int i = s * G + lane < N ? s * G + lane : 0;
          double v = 0.0;
          if constexpr (DF) {
            const int c = i < NTOP ? 1 + i / Q : 0, g = i < NTOP ? i % Q : tab.f0[i - NTOP];
            if (l == c) {
              v = LP[g];
            } else if (l == 0) {
              if (tab.src[i] >= 0) v = -ftab.mc[i] * LP[(int)tab.src[i]];
              if (tab.xslot[i] >= 0) v = fma(-XC[(int)tab.xslot[i]], LP[(int)tab.xsrc[(int)tab.xslot[i]]], v);
            }
            v *= ie2;
          } else if (second) {
            v = lap_col(i) * ie2;
          } else {
            v = inv_eps;
#pragma unroll
            for (int c = 0; c < D; ++c) v *= lt(c, i, c == ax ? 1 : 0);
          }
          w[s] = s * G + lane < N ? v : 0.0;
        }
        f64_solve<N, G, SN>(R, ID, w, lane);
        double* o = DF ? Y : U + l * Q;
#pragma unroll
        for (int s = 0; s < SN; ++s)
          if (s * G + lane < N) o[s * G + lane] = w[s];
        __syncwarp();
        if constexpr (DF) {
          for (int e = lane; e < NC * Q; e += G) {
            const int c = e / Q, g = e - c * Q;
            double v = 0.0;
            if (c >= 1) {
              v = Y[(c - 1) * Q + g];
            } else if (tab.fidx[g] >= 0) {
              v = Y[NTOP + tab.fidx[g]];
            } else {
#pragma unroll
              for (int c2 = 1; c2 < D; ++c2) {
                const int i = tab.inv[c2][g];
                if (i >= 0) v = fma(-ftab.mc[i], Y[i], v);
              }
              for (int x = 0; x < tab.nx; ++x)
                if (tab.xsrc[x] == g) v = fma(-XC[x], Y[(int)tab.xcol[x]], v);
            }
            U[l * NC * Q + e] = v;
          }
          __syncwarp();
        }
      }

      // ---- 5. w = W B y
      const bool live = have && !hand;
      if (live) {
#pragma unroll 1
        for (int q = lane; q < ke; q += G) {
          double x[D], m[Q];
#pragma unroll
          for (int c = 0; c < D; ++c) x[c] = X[c * kp + q];
          sne_columns<D, LO, HI>(x, cf, m);
          const double wt = SW[q] * SW[q];
#pragma unroll 1
          for (int r = 0; r < L * NC; ++r) {
            const double* u = U + r * Q;
            double s0 = 0.0, s1 = 0.0;
#pragma unroll
            for (int g = 0; g < Q; g += 2) {
              s0 = fma(m[g], u[g], s0);
              if (g + 1 < Q) s1 = fma(m[g + 1 < Q ? g + 1 : 0], u[g + 1 < Q ? g + 1 : 0], s1);
            }
            const double v = (s0 + s1) * wt;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const SneDst d = dst[2 * r + e];
              if (d.p) __stcs(d.p + (int64_t)q * d.stride, d.sgn < 0.0f ? -v : v);
            }
          }
        }
        for (int f = 0; f < j.nout; ++f)
          if (j.out_src[f] < 0) {
            const int64_t cnt = (int64_t)j.out_rows[f] * k * j.out_ncomp[f];
            double* wz = j.out_w[f] + o0 * (int64_t)j.out_rows[f] * j.out_ncomp[f];
            for (int64_t e = lane; e < cnt; e += G) wz[e] = 0.0;
          }
        if (j.beta)
          for (int l = lane; l < L; l += G) j.beta[to * L + l] = 0.0;
        if (lane == 0) {
          j.status[to] = st;
          if (j.iters) j.iters[to] = 0;
        }
      }
    }
    if (hand && lane == 0) j.gen_items[atomicAdd(j.gen_count, 1)] = (int32_t)to;
    __syncwarp();
  }
}

struct F64Entry {
  int kind, dim, deg, G, maxt, lmax;
  const void* fn;
  int (*stride)(int kp);  // doubles of shared memory per group
  F64Tab (*tab)();
};
#define GMLS_F64(KIND, D, DEG, G, P)                                                                            \
  F64Entry {                                                                                                    \
    KIND, D, DEG, G, 256, F64Lay<KIND, D, DEG, G, P>::LMAX, (const void*)stencil_f64_kernel<KIND, D, DEG, G, P, 256>, \
        &F64Lay<KIND, D, DEG, G, P>::stride,                                                                    \
        &make_f64_tab<D, SneDims<KIND, D, DEG, false>::LO, SneDims<KIND, D, DEG, false>::HI>                    \
  }

}  // namespace gmls
