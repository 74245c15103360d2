// stencil_sne.cuh -- GMLS stencils by corrected semi-normal equations: FP32 R
// factor, float-float residuals, several targets per warp.
//
// The same systems as stencil_fast.cuh and stencil_dfx.cuh (Sec. 2.1 - 2.5 of
// the paper: B = sqrt(W) P, weights w = sqrt(W) s, s the least-norm solution
// of B^T s = lambda^T), for the scalar, the staggered and the divergence-free
// basis, with or without the Neumann constraint.  What differs:
//
//  * Q is never formed or applied.  Only R (FP32, Householder) is kept:
//      y0 = R^-1 R^-T lambda,   s0 = B y0          (float-float),
//      g  = lambda - B^T s0 (float-float),  dy = R^-1 R^-T g,  s = s0 + B dy.
//    With E the backward error of the factorisation (R = Q^T (B + E)), the
//    error in z = R y contracts per step by |I - (B R^-1)^T (B R^-1)| =
//    O(|E R^-1|) = O(kappa u_32), the same rate as a step that applies Q
//    (Bjorck 1987, corrected semi-normal equations).
//  * Stencils do not depend on the basis within its span, so the columns are
//    products of one-dimensional polynomials q_0 .. q_m, orthogonal under the
//    target's own weighted neighbours (moments about their centroid, averaged
//    over the axes): kappa is some ten times below that of the monomials, the
//    error after one step a hundred times.  In the order of the monomials the
//    change of basis is triangular, so the scaled diagonal of R is that of the
//    Taylor basis.  Averaging needs axes of like extent: an axis along which the
//    neighbours spread at most a quarter as far as along the widest is stretched by
//    a power of two (axis c by 2^s_c; the derivatives at the target and the
//    component-0 parts below carry the factors).  On a 3D cloud flattened 100 times
//    the common coefficients alone cost three digits (4.8e-9).
//  * A group of G lanes (8, 16 or 32) owns a target, 32 / G targets a warp.  For
//    the QR a lane owns whole columns (column c on lane c % G) and the rows
//    stream through its registers P at a time, each block eliminated against
//    the triangle kept in shared memory: one shuffle a step (a shuffle issues at
//    a quarter of the FMA rate), the reflector broadcast through shared memory
//    in 16-byte loads, and any row count in one instantiation.  For the products
//    a lane owns rows.
//  * Both run on packed FP32 pairs (two rows in the QR, two right-hand sides in
//    the products per instruction): the same 128 operations a clock and SM as
//    scalar FP32 at half the issue slots.
//  * The tile is not stored: only eta = (x_j - x_T) / eps - centroid and sqrt(W)
//    are (float-float); the columns are recomputed in each pass.
//  * Products are accumulated against a large constant: h starts at M = 1.5 2^e,
//    2^(e-1) above the sum of the |products|, so that every partial sum stays
//    in one binade and  t = fl(fl(h + a b) - h)  is exact; then
//    fma(a, b, -t) is the rounding error of the step.  Six operations a term
//    instead of the twelve of a compensated product with TwoSum.  The bounds
//    (Cauchy-Schwarz, column norms of R): |p_q / |A e_q|| |u_q |A e_q|| over the
//    columns for a row of B y0, |A e_q| |s| for B^T s.  The roundings of the low
//    parts are about 2^-43 of the bound; the residual's are amplified by the
//    condition number, so the steps after the first (targets whose first
//    correction is above 1e-5) sum B^T s with TwoSum.
//  * Divergence-free basis: B = (I (x) A) C as in stencil_dfx.cuh, with
//    phi_{c,g} = e_c p_g - e_0 int d_c p_g (c >= 1; the antiderivative in x_0 is
//    a combination of at most four p's) and phi_{0,g} = e_0 p_g (g_0 = 0); R_A,
//    then the component-0 rows of (I (x) R_A) C are eliminated by the same
//    routine as a row block.
//  * Neumann targets (Sec. 2.3): B^T s + beta f = lambda^T with f the normal
//    derivative at x_T of the basis, |s| least: s = s_lambda - beta s_f, beta =
//    (s_f . s_lambda) / (s_f . s_f), f one more right-hand side.  A gradient row
//    enters as its tangential part (the normal part n_c f / |n|^2 goes into beta
//    alone), so rows along the normal, whose weights nearly vanish, lose nothing
//    to the difference.  The Laplacian row, on a one-sided target mostly beta s_f, is
//    solved as lambda - beta_0 f with beta_0 from the FP32 factor for the same
//    reason (without it its weights were 4 to 27 times further off than by
//    elimination: 3D degree 2 1.1e-12, degree 3 6.1e-12).
//  * Range: lambda carries eps^-1 or eps^-2 and the bounds above its squares, which
//    leave FP32 already at eps = 1e-9 (a cloud of nanometres).  The systems are
//    solved for lambda 2^(ORDER ee), 2^ee <= eps < 2^(ee + 1), ORDER the highest
//    power of 1 / eps among the rows: everything is homogeneous in lambda, so no
//    other bit changes, and sqrt(W) of the last product carries 2^(-ORDER ee).
#pragma once
#include <cuda_runtime.h>

#include <utility>

#include "stencil_fast.cuh"

namespace gmls {

// ----------------------------------------------------- packed pairs of floats
using f2 = unsigned long long;  // two FP32 values in one 64-bit register pair
__device__ __forceinline__ f2 pk2(float a, float b) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ f2 dup2(float a) { return pk2(a, a); }
__device__ __forceinline__ void unpk2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 neg2(f2 v) {
  float a, b;
  unpk2(v, a, b);
  return pk2(-a, -b);
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float sum2(f2 v) {
  float a, b;
  unpk2(v, a, b);
  return a + b;
}

// float-float values of two rows
struct ffp {
  f2 h, l;
};
// product without the final normalisation (lo up to an ulp of hi)
__device__ __forceinline__ ffp mul_raw(ffp a, ffp b) {
  ffp r;
  r.h = mul2(a.h, b.h);
  r.l = fma2(a.l, b.h, fma2(a.h, b.l, fma2(a.h, b.h, neg2(r.h))));
  return r;
}
__device__ __forceinline__ ff mul_raw(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  return ff(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ float mul_raw(float a, float b) { return a * b; }
__device__ __forceinline__ double mul_raw(double a, double b) { return a * b; }
__device__ __forceinline__ ffp add_c(ffp a, float c) {  // a + c, not normalised
  const f2 cc = dup2(c);
  ffp r;
  r.h = add2(a.h, cc);
  const f2 bb = sub2(r.h, a.h);
  r.l = add2(add2(sub2(a.h, sub2(r.h, bb)), sub2(cc, bb)), a.l);
  return r;
}
__device__ __forceinline__ ff add_c(ff a, float c) {
  const ff s = two_sum(a.h, c);
  return ff(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ float add_c(float a, float c) { return a + c; }
__device__ __forceinline__ double add_c(double a, float c) { return a + (double)c; }
__device__ __forceinline__ ffp quick2(f2 h, f2 l) {  // h + l renormalised, |h| >= |l|
  ffp r;
  r.h = add2(h, l);
  r.l = sub2(l, sub2(r.h, h));
  return r;
}
__device__ __forceinline__ ffp mul_ff(ffp a, ffp b) {
  const ffp r = mul_raw(a, b);
  return quick2(r.h, r.l);
}
__device__ __forceinline__ ffp add_ff(ffp a, ffp b) {
  const f2 h = add2(a.h, b.h), bb = sub2(h, a.h);
  return quick2(h, add2(add2(sub2(a.h, sub2(h, bb)), sub2(b.h, bb)), add2(a.l, b.l)));
}
__device__ __forceinline__ ff row_of(ffp a, int r) {
  float h0, h1, l0, l1;
  unpk2(a.h, h0, h1);
  unpk2(a.l, l0, l1);
  return r ? ff(h1, l1) : ff(h0, l0);
}

// h + l += a b, two right-hand sides b, h kept near the constant it started from
__device__ __forceinline__ void sne_acc(f2& h, f2& l, ff a, ffp b) {
  const f2 ah = dup2(a.h), hn = fma2(ah, b.h, h);
  l = add2(l, fma2(ah, b.h, sub2(h, hn)));
  l = fma2(dup2(a.l), b.h, fma2(ah, b.l, l));
  h = hn;
}
__device__ __forceinline__ void sne_acc(f2& h, f2& l, ff a, f2 b) {
  const f2 ah = dup2(a.h), hn = fma2(ah, b, h);
  l = add2(l, fma2(ah, b, sub2(h, hn)));
  l = fma2(dup2(a.l), b, l);
  h = hn;
}
// the same without a constant (TwoSum): for the steps after the first, which only
// ill-conditioned targets take
__device__ __forceinline__ void sne_acc_twosum(f2& h, f2& l, ff a, ffp b) {
  const f2 ah = dup2(a.h), p = mul2(ah, b.h);
  const f2 e = fma2(dup2(a.l), b.h, fma2(ah, b.l, fma2(ah, b.h, neg2(p))));
  const f2 s = add2(h, p), bb = sub2(s, h);
  l = add2(l, add2(add2(sub2(h, sub2(s, bb)), sub2(p, bb)), e));
  h = s;
}
// 1.5 2^e with 2^(e-1) > bound
__device__ __forceinline__ float sne_magic(float bound) {
  const unsigned e = (__float_as_uint(bound * 1.01f) >> 23) & 0xffu;
  return __uint_as_float(((e < 252u ? e + 2u : 254u) << 23) | 0x400000u);
}
// the power of two above v
__device__ __forceinline__ float sne_pow2(float v) {
  const unsigned e = (__float_as_uint(v) >> 23) & 0xffu;
  return __uint_as_float((e < 253u ? e + 1u : 254u) << 23);
}

// float-float -> double: exponents re-biased with integer operations and one
// FP64 addition; hi near the ends of the exponent range takes the conversions
// (a zero lo becomes 2^-127, far below half an ulp of hi)
__device__ __forceinline__ double sne_to_double(ff a) {
  const unsigned u = __float_as_uint(a.h), v = __float_as_uint(a.l);
  if (((u >> 23) & 0xffu) - 100u >= 150u) return (double)a.h + (double)a.l;
  const double h = __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
  const double l = __hiloint2double((int)((v & 0x80000000u) | (((v & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(v << 29));
  return h + l;
}
// 2^e; zero and infinity beyond the normal range
__device__ __forceinline__ float sne_exp2(int e) { return __int_as_float(e < -126 ? 0 : (min(e, 128) + 127) << 23); }
// where the weights of one right-hand side go: entry q at p + q * stride
struct SneDst {
  double* p;
  int stride;
  float sgn;
};

// --------------------------------------------------------------- the columns
// Products q_a(x) q_b(y) q_c(z) of total degree LO..HI in the order of the
// Taylor monomials (degree ascending; within a degree the power of x descends,
// then that of y).
template <int D, int LO, int HI>
struct SneMono {
  __host__ __device__ static constexpr int count(int m) {
    return m < 0 ? 0 : D == 2 ? (m + 1) * (m + 2) / 2 : (m + 1) * (m + 2) * (m + 3) / 6;
  }
  static constexpr int Q = count(HI) - count(LO - 1);
  // position of exponents (a, b, c)
  __host__ __device__ static constexpr int index(int a, int b, int c) {
    const int s = a + b + c;
    return count(s - 1) + (D == 2 ? b : (s - a) * (s - a + 1) / 2 + c) - count(LO - 1);
  }
  __host__ __device__ static constexpr int exponent(int i, int axis) {
    int j = i + count(LO - 1), s = 0;
    while (count(s) <= j) ++s;
    j -= count(s - 1);
    if (D == 2) return axis == 0 ? s - j : axis == 1 ? j : 0;
    int r = 0;  // s - a
    while ((r + 1) * (r + 2) / 2 <= j) ++r;
    const int c = j - r * (r + 1) / 2;
    return axis == 0 ? s - r : axis == 1 ? r - c : c;
  }
};

// Column tables (a kernel parameter: constant bank, run-time indices).  For the
// divergence-free basis the component-0 part of column i = phi_{c,g}, c >= 1, is
//   -(mc[i] p_{src[i]} + x_i p_{xsrc[i]}),  mc = g_c / (g_0 + 1), src = g - e_c + e_0:
// d q_p = p q_{p-1} + (target's coefficient, p >= 3) q_{p-3} and int q_p =
// q_{p+1} / (p + 1) + (target's coefficient, p >= 2) q_{p-1} give at most one
// further term up to degree 4 (xsrc < 0: none); x_i is formed per target.
constexpr int kSneMaxExtra = 16;
__host__ __device__ constexpr int sne_extras(int d, int m) { return (d - 1) * (m < 3 ? 0 : d == 2 ? (m == 3 ? 2 : 6) : (m == 3 ? 2 : 8)); }
struct SneTab {
  int8_t e[3][40];      // powers of column i of A
  int8_t f0[16];        // phi_{0,.}: its column of A
  int8_t fidx[40];      // g_0 = 0: position among the phi_0 columns, else -1
  int8_t src[72], xslot[72];            // phi_{c,g}: main source; slot of its further term, or -1
  int8_t inv[3][40];                    // c, p: the column phi_{c,.} whose main source is p, or -1
  int8_t xcol[kSneMaxExtra], xsrc[kSneMaxExtra], nx;  // further terms: column, source
  float mch[72], mcl[72];               // main coefficient, float-float
};
template <int D, int LO, int HI>
SneTab make_sne_tab() {
  using Mo = SneMono<D, LO, HI>;
  constexpr int Q = Mo::Q;
  SneTab t{};
  int f = 0;
  for (int i = 0; i < Q && i < 40; ++i) {
    for (int c = 0; c < 3; ++c) t.e[c][i] = (int8_t)Mo::exponent(i, c);
    t.fidx[i] = -1;
    if (LO == 0 && Mo::exponent(i, 0) == 0 && f < 16) {
      t.f0[f] = (int8_t)i;
      t.fidx[i] = (int8_t)f++;
    }
  }
  for (auto& r : t.inv)
    for (auto& v : r) v = -1;
  for (auto& v : t.src) v = -1;
  for (auto& v : t.xslot) v = -1;
  if (LO == 0)
    for (int c = 1; c < D; ++c)
      for (int g = 0; g < Q; ++g) {
        const int i = (c - 1) * Q + g, g0 = t.e[0][g], gc = t.e[c][g];
        if (i >= 72 || gc == 0) continue;
        int h[3] = {g0 + 1, t.e[1][g], t.e[2][g]};
        h[c] -= 1;
        t.src[i] = (int8_t)Mo::index(h[0], h[1], h[2]);
        t.inv[c][(int)t.src[i]] = (int8_t)i;
        const double mc = (double)gc / (g0 + 1);
        t.mch[i] = (float)mc;
        t.mcl[i] = (float)(mc - (double)t.mch[i]);
        if (gc >= 3 || g0 >= 2) {
          if (gc >= 3)
            h[c] -= 2;
          else
            h[0] -= 2;
          t.xslot[i] = t.nx;
          t.xcol[(int)t.nx] = (int8_t)i;
          t.xsrc[(int)t.nx] = (int8_t)Mo::index(h[0], h[1], h[2]);
          ++t.nx;
        }
      }
  return t;
}

// coefficients of q_2 = x^2 - a, q_3 = x^3 - b x, q_4 = x^4 - c x^2 + d, q_5 = x^5 - e x^3 + f x
struct SneCoef {
  float a, b, c, d, e, f;
};

// from the moments 2, 4, 6, 8 averaged over the axes
template <int HI, bool ST>
__device__ __forceinline__ void sne_coefficients(const float (&mu)[4], SneCoef& cf) {
  const float i2 = 1.0f / mu[0], den = mu[1] - mu[0] * mu[0], d4 = mu[2] * mu[0] - mu[1] * mu[1];
  cf.a = ST ? 0.0f : mu[0];
  cf.b = HI >= 3 ? mu[1] * i2 : 0.0f;
  const bool full4 = !ST && den > 1e-4f * mu[1];
  cf.c = HI >= 4 ? (full4 ? (mu[2] - mu[0] * mu[1]) / den : mu[2] / mu[1]) : 0.0f;
  cf.d = full4 ? cf.c * mu[0] - mu[1] : 0.0f;
  const bool full5 = d4 > 1e-4f * mu[1] * mu[1];
  cf.e = HI >= 5 ? (full5 ? (mu[3] * mu[0] - mu[2] * mu[1]) / d4 : mu[3] / mu[2]) : 0.0f;
  cf.f = HI >= 5 && full5 ? (cf.e * mu[1] - mu[2]) * i2 : 0.0f;
}

// q_0 .. q_HI of one axis (q[0] unused)
template <int HI, typename T>
__device__ __forceinline__ void sne_axis(T x, const SneCoef& k, T (&q)[HI + 1]) {
  q[1] = x;
  if constexpr (HI >= 2) {
    const T t = mul_raw(x, x);
    q[2] = add_c(t, -k.a);
    if constexpr (HI >= 3) q[3] = mul_raw(x, add_c(t, -k.b));
    if constexpr (HI >= 4) q[4] = add_c(mul_raw(t, add_c(t, -k.c)), k.d);
    if constexpr (HI >= 5) q[5] = mul_raw(x, add_c(mul_raw(t, add_c(t, -k.e)), k.f));
  }
}
__device__ __forceinline__ ffp sne_one(ffp) { return ffp{dup2(1.0f), dup2(0.0f)}; }
__device__ __forceinline__ ff sne_one(ff) { return ff(1.0f, 0.0f); }
__device__ __forceinline__ float sne_one(float) { return 1.0f; }
__device__ __forceinline__ double sne_one(double) { return 1.0; }

// column I from the axis values (products that columns share are left to the
// compiler)
template <int D, int LO, int HI, int I, typename T>
__device__ __forceinline__ T sne_column(const T (&q)[D][HI + 1]) {
  using Mo = SneMono<D, LO, HI>;
  constexpr int a = Mo::exponent(I, 0), b = Mo::exponent(I, 1), c = Mo::exponent(I, 2);
  if constexpr (a + b + c == 0) {
    return sne_one(q[0][1]);
  } else if constexpr (c == 0 || D == 2) {
    if constexpr (b == 0) return q[0][a];
    if constexpr (a == 0) return q[1][b];
    return mul_raw(q[0][a], q[1][b]);
  } else {
    if constexpr (a == 0 && b == 0) return q[2][c];
    return mul_raw(sne_column<D, LO, HI, Mo::index(a, b, 0)>(q), q[2][c]);
  }
}
template <int D, int LO, int HI, typename T, int Q, int... I>
__device__ __forceinline__ void sne_columns_all(const T (&q)[D][HI + 1], T (&m)[Q], std::integer_sequence<int, I...>) {
  ((m[I] = sne_column<D, LO, HI, I>(q)), ...);
}
template <int D, int LO, int HI, typename T, int Q>
__device__ __forceinline__ void sne_columns(const T (&x)[D], const SneCoef& k, T (&m)[Q]) {
  T q[D][HI + 1];
#pragma unroll
  for (int c = 0; c < D; ++c) sne_axis<HI>(x[c], k, q[c]);
  sne_columns_all<D, LO, HI>(q, m, std::make_integer_sequence<int, Q>{});
}

template <int G>
__device__ __forceinline__ float gsum(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, G);
  return v;
}
template <int G>
__device__ __forceinline__ float gmax(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o, G));
  return v;
}
template <int G>
__device__ __forceinline__ ff gsum(ff v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1)
    v = v + ff(__shfl_xor_sync(0xffffffffu, v.h, o, G), __shfl_xor_sync(0xffffffffu, v.l, o, G));
  return v;
}

// sum of v[0..C) over the G lanes of a group; the totals of entries
// lane C / G .. (lane + 1) C / G - 1 end in v[0..C / G) of that lane
template <int G, int C>
__device__ __forceinline__ void sne_reduce_scatter(float (&v)[C], int lane) {
  static_assert(C % G == 0, "whole shares");
#pragma unroll
  for (int st = 0; (G >> st) > 1; ++st) {
    const int o = (G / 2) >> st, h = C >> (st + 1);
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i)
      if (i < h) {
        const float send = up ? v[i] : v[i + h];
        const float keep = up ? v[i + h] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o, G);
      }
  }
}

// the same for float-float values
template <int G, int C>
__device__ __forceinline__ void sne_reduce_scatter(float (&h)[C], float (&l)[C], int lane) {
#pragma unroll
  for (int st = 0; (G >> st) > 1; ++st) {
    const int o = (G / 2) >> st, n = C >> (st + 1);
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i)
      if (i < n) {
        const float sh = up ? h[i] : h[i + n], sl = up ? l[i] : l[i + n];
        const ff s = two_sum(up ? h[i + n] : h[i], __shfl_xor_sync(0xffffffffu, sh, o, G));
        h[i] = s.h;
        l[i] = ((up ? l[i + n] : l[i]) + __shfl_xor_sync(0xffffffffu, sl, o, G)) + s.l;
      }
  }
}

// Householder elimination of a block of P rows against the packed upper
// triangle R (N columns): column c of the block (row pairs) in slot c / G of
// lane c % G.  Reflector k acts on (row k of R, the block): v = (alpha - beta,
// block column k), H = I - f v v^T, f = 2 / v^T v.  The owner of column k
// publishes it in vbuf (two buffers in turn: one barrier a step); its own dot
// product with it is |block column k|^2.
template <int P, int SN, int N, int G>
__device__ __forceinline__ void sne_append(f2 (&a)[SN][P / 2], float* R, float* vbuf, int lane, int& par) {
  constexpr int PV = P + 4;
  static_assert(P % 4 == 0, "16-byte rows");
#pragma unroll
  for (int s = 0; s < SN; ++s) {
    constexpr int last = N - (SN - 1) * G;  // columns of the last slot
    float* rrow = R + rpk<N>(s * G, 0);     // row k of R: entry c at rrow[c]
#pragma unroll 1
    for (int o = 0; o < (s < SN - 1 ? G : last); ++o) {
      const int k = s * G + o;
      float* vb = vbuf + par * PV;
      par ^= 1;
      if (lane == o) {
        ulonglong2* v4 = reinterpret_cast<ulonglong2*>(vb);
#pragma unroll
        for (int i = 0; i < P / 4; ++i) v4[i] = make_ulonglong2(a[s][2 * i], a[s][2 * i + 1]);
        vb[P] = rrow[k];
      }
      __syncwarp();
      f2 v[P / 2];
      {
        const ulonglong2* v4 = reinterpret_cast<const ulonglong2*>(vb);
#pragma unroll
        for (int i = 0; i < P / 4; ++i) {
          const ulonglong2 q = v4[i];
          v[2 * i] = q.x;
          v[2 * i + 1] = q.y;
        }
      }
      const float alpha = vb[P];
      float d[SN];
#pragma unroll
      for (int u = s; u < SN; ++u) {
        f2 d0 = mul2(v[0], a[u][0]), d1 = mul2(v[1], a[u][1]);
#pragma unroll
        for (int i = 2; i < P / 2; ++i) {
          if (i & 1)
            d1 = fma2(v[i], a[u][i], d1);
          else
            d0 = fma2(v[i], a[u][i], d0);
        }
        d[u] = sum2(add2(d0, d1));
      }
      const float sig = __shfl_sync(0xffffffffu, d[s], o, G);
      float f = 0.0f, v0 = 0.0f, beta = alpha;
      if (sig > 0.0f) {
        const float n2 = fmaf(alpha, alpha, sig), nrm = n2 * rsqrtf(n2);  // a few ulp, as the products around it
        beta = alpha >= 0.0f ? -nrm : nrm;
        v0 = alpha - beta;
        f = __fdividef(2.0f, fmaf(v0, v0, sig));
      }
#pragma unroll
      for (int u = s; u < SN; ++u) {
        const bool act = (u > s || lane > o) && (u < SN - 1 || lane < last);
        float* rp = rrow + (act ? u * G + lane : k);
        const float rk = act ? *rp : 0.0f;
        const float td = act ? fmaf(v0, rk, d[u]) * f : 0.0f;
        if (act) *rp = fmaf(-td, v0, rk);
        const f2 nt = dup2(-td);
#pragma unroll
        for (int i = 0; i < P / 2; ++i) a[u][i] = fma2(nt, v[i], a[u][i]);
      }
      if (lane == o) rrow[k] = beta;
      rrow += N - 1 - k;
    }
  }
}

// w <- R^-T w (TRANS) or R^-1 w; entry p of a vector at lane p % G, slot p / G
// (entries past N hold anything: no entry before N reads them)
template <int N, int L, int G, int SN, bool TRANS>
__device__ __forceinline__ void sne_solve(const float* R, const float* ID, float (&w)[L][SN], int lane) {
  if constexpr (TRANS) {
    const float* rrow = R + lane;  // row i of R: entry p = u G + lane at rrow[u G]
#pragma unroll
    for (int s = 0; s < SN; ++s) {
#pragma unroll 1
      for (int o = 0; o < (s < SN - 1 ? G : N - (SN - 1) * G); ++o) {
        const int i = s * G + o;
        const float inv = ID[i];
        float yi[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
          yi[l] = __shfl_sync(0xffffffffu, w[l][s], o, G) * inv;
          if (lane == o) w[l][s] = yi[l];
        }
#pragma unroll
        for (int u = s; u < SN; ++u) {
          const float r = (u > s || lane > o) ? rrow[u * G] : 0.0f;
#pragma unroll
          for (int l = 0; l < L; ++l) w[l][u] = fmaf(-r, yi[l], w[l][u]);
        }
        rrow += N - 1 - i;
      }
    }
  } else {
    const float* rcol[SN];  // entry (p, i), p = u G + lane <= i, at rcol[u][i]
#pragma unroll
    for (int u = 0; u < SN; ++u) rcol[u] = R + rpk<N>(u * G + lane < N ? u * G + lane : 0, 0);
#pragma unroll
    for (int s = SN - 1; s >= 0; --s) {
#pragma unroll 1
      for (int o = (s < SN - 1 ? G : N - (SN - 1) * G) - 1; o >= 0; --o) {
        const int i = s * G + o;
        const float inv = ID[i];
        float yi[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
          yi[l] = __shfl_sync(0xffffffffu, w[l][s], o, G) * inv;
          if (lane == o) w[l][s] = yi[l];
        }
#pragma unroll
        for (int u = 0; u <= s; ++u) {
          const float r = (u < s || lane < o) ? rcol[u][i] : 0.0f;
#pragma unroll
          for (int l = 0; l < L; ++l) w[l][u] = fmaf(-r, yi[l], w[l][u]);
        }
      }
    }
  }
}

template <int KIND, int D, int DEG, bool NEU>
struct SneDims {
  static constexpr int DIM = D, DEGREE = DEG;
  static constexpr bool DF = KIND == GMLS_BASIS_DIVFREE, ST = KIND == GMLS_BASIS_STAGGERED;
  static constexpr int LO = ST ? 1 : 0;
  static constexpr int HI = ST ? DEG + 1 : DEG;
  static constexpr int Q = SneMono<D, LO, HI>::Q;  // columns of A
  static constexpr int NC = DF ? D : 1;
  static constexpr int NTOP = DF ? (D - 1) * Q : 0;                              // phi_{c,g}, c >= 1
  static constexpr int N0 = DF ? (D == 2 ? DEG + 1 : (DEG + 1) * (DEG + 2) / 2) : 0;  // phi_{0,g}
  static constexpr int N = DF ? NTOP + N0 : Q;                                   // unknowns
};

// Shared memory of one group, in floats
template <int KIND, int D, int DEG, int L, int G, int P, int LS, bool NEU>
struct SneLay {
  using Dm = SneDims<KIND, D, DEG, NEU>;
  static constexpr bool DF = Dm::DF;
  static constexpr int Q = Dm::Q, N = Dm::N, LR = L + (NEU ? 1 : 0);
  static constexpr int RHS = (LR * Dm::NC + LS - 1) / LS * LS;  // right-hand sides of the products, whole passes
  static_assert(LS % 2 == 0, "pairs of right-hand sides");
  __host__ __device__ static constexpr int up4(int v) { return (v + 3) & ~3; }
  static constexpr int QP = up4(Q);
  static constexpr int PS = (P / 4) % 2 ? P : P + 4;  // column stride of the staged block: 8 columns' 16-byte loads in distinct banks
  static constexpr int PG = up4(Q);                   // rows of the component-0 block
  static constexpr int NR = N * (N + 1) / 2;
  static constexpr bool ST_IN_R = DF && Q * PS <= NR;  // R is not in use yet while A is factored
  static constexpr int R = 0;                          // packed triangle of the solve
  static constexpr int ID = up4(NR);                   // 1 / r_ii
  static constexpr int HI1 = Dm::HI + 1;
  static constexpr int LT = up4(ID + N);                           // q, q', q'' at the target: ff [D][HI + 1][3]
  static constexpr int LP = LT + (DF ? 0 : up4(6 * D * HI1));  // divergence-free instead: Laplacians of the columns
  static constexpr int XC = up4(LP + (DF ? 2 * Q : 0));        // and the coefficients of the further terms
  static constexpr int X = up4(XC + (DF ? 2 * sne_extras(Dm::DIM, Dm::DEGREE) : 0));  // the rest takes turns
  // QR: staged rows, reflector buffers, R_A
  static constexpr int VB = X;
  static constexpr int VBN = 2 * ((P > PG || !DF ? P : PG) + 4);
  static constexpr int RA = up4(VB + VBN);
  static constexpr int ST = ST_IN_R ? R : up4(RA + (DF ? Q * (Q + 1) / 2 : 0));
  static constexpr int E1 = ST_IN_R ? RA + Q * (Q + 1) / 2 : ST + Q * PS;
  // solve: u (then v, then du), accumulator constants, y
  static constexpr int UH = X;
  static constexpr int UL = UH + RHS * QP;
  static constexpr int MG = UL + RHS * QP;
  static constexpr int MS = MG + LR * QP;
  static constexpr int IC = up4(MS + RHS);  // 1 / |A e_q|
  // (divergence-free) the unknowns, before they are spread into u; the 3D
  // degree-3 basis keeps them in u's place (eleven instead of ten warps per SM)
  static constexpr bool Y_IN_U = DF && D == 3 && DEG == 3;
  static constexpr int Y = Y_IN_U ? UH : IC + QP;
  static constexpr int E2 = Y_IN_U || !DF ? IC + QP : Y + L * N;
  static constexpr int DST = UL;  // SneDst [L NC][2], in the last section
  static_assert(!Y_IN_U || L * N <= RHS * QP, "y fits in u's place");
  static_assert(8 * L * Dm::NC <= RHS * QP, "the destinations fit in the low parts' place");
  // targets' tables of the divergence-free basis (needed before UH .. only)
  static constexpr int E3 = DF ? X + 6 * D * HI1 : X;
  static constexpr int emax(int a, int b) { return a > b ? a : b; }
  // eta and sqrt(W): float [2 (D + 1)][kp]; root of sum_q (p_q / |A e_q|)^2: float [kp];
  // the axes' s_c, eight bits each: int
  static constexpr int XI = up4(emax(emax(E1, E2), E3));
  // group stride: the 32 / G groups of a warp start G banks apart
  __host__ __device__ static int stride(int kp) {
    const int need = XI + (2 * (D + 1) + 1) * kp + 1;
    return G == 32 ? ((need + 3) & ~3) : ((need + 31 - G) / 32 * 32 + G);
  }
};

// MAXT bounds the registers (65536 / MAXT a thread): the launcher fills an SM
// with one block of up to MAXT threads.  LS: right-hand sides per product pass
// (their 2 Q LS accumulators, high and low parts, live in registers).
template <int KIND, int D, int DEG, int L, int G, int P, int LS, bool NEU, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) stencil_sne_kernel(StencilJob j, const SneTab tab, int kp) {
  using Dm = SneDims<KIND, D, DEG, NEU>;
  using Lay = SneLay<KIND, D, DEG, L, G, P, LS, NEU>;
  using Mo = SneMono<D, Dm::LO, Dm::HI>;
  constexpr bool DF = Dm::DF, ST = Dm::ST;
  constexpr int LO = Dm::LO, HI = Dm::HI, Q = Dm::Q, N = Dm::N, NC = Dm::NC, QP = Lay::QP, NTOP = Dm::NTOP;
  constexpr int LR = Lay::LR, LC = LR * NC, RHS = Lay::RHS;
  constexpr int SA = (Q + G - 1) / G, SN = (N + G - 1) / G;  // column slots of A and of the solve
  static_assert(N == gmls_gen::basis_size(KIND, D, DEG), "basis size");
  static_assert(!NEU || KIND == GMLS_BASIS_SCALAR, "the Neumann constraint is for the scalar basis");
  // margin on the estimated error: the contraction measured against 64-bit
  // weights is up to four times the size of the first correction for the
  // divergence-free and the staggered columns (the latter have no constant to be
  // orthogonal to)
  constexpr float kSafe = DF ? 4.0f : ST ? 16.0f : 1.0f;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(16) float smf[];
  const int lane = threadIdx.x & (G - 1);
  const int gpb = blockDim.x / G, grp = threadIdx.x / G, gpw = 32 / G;
  float* base = smf + (size_t)grp * Lay::stride(kp);
  float* R = base + Lay::R;
  float* ID = base + Lay::ID;
  float* XH = base + Lay::XI;
  float* XL = XH + D * kp;
  float* SWH = XL + D * kp;
  float* SWL = SWH + kp;
  float* RN = SWL + kp;
  int* AX = reinterpret_cast<int*>(RN + kp);
  float* UH = base + Lay::UH;
  float* UL = base + Lay::UL;
  float* MG = base + Lay::MG;
  float* MS = base + Lay::MS;
  float* IC = base + Lay::IC;
  float* Y = base + Lay::Y;
  // s of row q, right-hand sides 2 i and 2 i + 1: (hi, hi, lo, lo) at S0[i kp + q]
  ulonglong2* S0 = reinterpret_cast<ulonglong2*>(j.dscratch) + ((size_t)blockIdx.x * gpb + grp) * (size_t)(RHS / 2 * kp);
  const int64_t n = j.n;
  // work list: everything, a list with its length, or one bucket of a sorted list
  const int64_t first = j.item_range ? (int64_t)j.item_range[0] : 0;
  const int64_t n_items = j.item_range ? (int64_t)j.item_range[1] - first : j.items ? (int64_t)(*j.n_items) : j.n_tgt;
  const float tolf = (float)j.tol;
  // u / v / du of right-hand side r, column g
  auto ux = [](int r, int g) { return ((r >> 1) * QP + g) * 2 + (r & 1); };
  auto row_pair = [](const float* p, int i) { return *reinterpret_cast<const f2*>(p + 2 * i); };

  for (int64_t ib = ((int64_t)blockIdx.x * gpb) + (threadIdx.x / 32) * gpw; ib < n_items; ib += (int64_t)gridDim.x * gpb) {
    const int64_t it = ib + (grp & (gpw - 1));
    const bool have = it < n_items;
    const int64_t pos = first + (have ? it : n_items - 1);
    const int64_t to = j.items ? (int64_t)j.items[pos] : pos;
    const int64_t t = j.tgt[to];
    const int64_t o0 = j.off[to];
    const int k = (int)(j.off[to + 1] - o0);
    const uint8_t st = j.nbr_status ? j.nbr_status[to] : 0;
    const bool neu = KIND == GMLS_BASIS_SCALAR && j.neumann && j.bflag && j.bflag[t] && j.normals;
    const bool too_few = (st & GMLS_T_TOO_FEW_NEIGHBOURS) || k <= 0 || !(j.eps[to] > 0.0);
    int self = -1;  // staggered: the target's own entry
    if constexpr (ST) {
      int f1 = 0x7fffffff;
      if (have && !too_few)
        for (int q = lane; q < k; q += G)
          if (j.idx[o0 + q] == (int32_t)t) f1 = min(f1, q);
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) f1 = min(f1, __shfl_xor_sync(FULL, f1, o, G));
      self = f1 == 0x7fffffff ? -1 : f1;
    }
    // tiles this path does not take (the shared-memory FP32 kernel does)
    const bool misfit = neu != NEU || k > kp || k < (DF ? Q : N) || (ST && self < 0);
    const bool active = have && !too_few && !misfit;
    if (have && too_few) {
      for (int f = 0; f < j.nout; ++f) {
        const int64_t cnt = (int64_t)j.out_rows[f] * k * j.out_ncomp[f];
        double* w = j.out_w[f] + o0 * (int64_t)j.out_rows[f] * j.out_ncomp[f];
        for (int64_t e = lane; e < cnt; e += G) w[e] = 0.0;
      }
      if (j.beta)
        for (int l = lane; l < L; l += G) j.beta[to * L + l] = 0.0;
      if (lane == 0) {
        j.status[to] = st;
        if (j.iters) j.iters[to] = 0;
      }
    } else if (have && misfit && lane == 0) {
      if (!NEU && neu && j.neu_items)
        j.neu_items[atomicAdd(j.neu_count, 1)] = (int32_t)to;
      else
        j.gen_items[atomicAdd(j.gen_count, 1)] = (int32_t)to;
      j.status[to] = 0;
    }
    const int ke = active ? k : 0;
    const int pw = (__reduce_max_sync(FULL, ke) + 1) >> 1;  // row pairs of the longest list in the warp
    if (pw == 0) continue;
    __syncwarp();

    // ---- 1. xi = (x_j - x_T) / eps and sqrt(W) (float-float from the FP64 offsets)
    // 2^ee / eps (of eps / 2^ee), 1 / eps and 1 / eps^2 times 2^(ORDER ee)
    constexpr int ORDER = !DF && L == D ? 1 : 2;  // (L == D: the gradient alone)
    auto eps_exponent = [&]() { return min(126, max(-126, ((__double2hiint(j.eps[to]) >> 20) & 0x7ff) - 1023)); };
    const float pe = sne_exp2(eps_exponent()), pi = sne_exp2(-eps_exponent());
    const ff inv_eps = recip(ff(j.eps[to] * (double)pi));
    const ff ie2 = inv_eps * inv_eps;
    [[maybe_unused]] const ff ie1 = ORDER == 1 ? inv_eps : ff(inv_eps.h * pe, inv_eps.l * pe);
    double xt[D];
#pragma unroll
    for (int c = 0; c < D; ++c) xt[c] = j.x[c * n + t];
    float mw = 0.0f, m1[D], m2[D];
#pragma unroll
    for (int c = 0; c < D; ++c) m1[c] = m2[c] = 0.0f;
    // (the gathers of four rows in flight together)
#pragma unroll 1
    for (int q0 = 0; q0 < 2 * pw; q0 += 4 * G) {
      int32_t jj[4];
      double xv[4][D];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int q = q0 + 2 * G * (e >> 1) + 2 * lane + (e & 1);
        jj[e] = q < ke ? j.idx[o0 + q] : (int32_t)t;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int c = 0; c < D; ++c) xv[e][c] = j.x[c * n + jj[e]];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = q0 + 2 * G * h + 2 * lane;  // rows q and q + 1
        if (q >= 2 * pw) continue;
        const ffp ie{dup2(inv_eps.h), dup2(inv_eps.l)};
        ffp xi[D], r2{0, 0};
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const ff d0 = diff_ff(xv[2 * h][c], xt[c]), d1 = diff_ff(xv[2 * h + 1][c], xt[c]);
          const ffp dx{mul2(pk2(d0.h, d1.h), dup2(pi)), mul2(pk2(d0.l, d1.l), dup2(pi))};
          xi[c] = mul_ff(dx, ie);
          r2 = add_ff(r2, mul_ff(dx, dx));
        }
        ffp u;
        {
          const ff a = sqrt_ff(row_of(r2, 0)), b = sqrt_ff(row_of(r2, 1));
          u = mul_ff(ffp{pk2(a.h, b.h), pk2(a.l, b.l)}, ie);
          u = add_ff(ffp{dup2(1.0f), 0}, ffp{neg2(u.h), neg2(u.l)});
        }
        ffp sw = u;
        for (int p = 1; p < j.wpow_half; ++p) sw = mul_ff(sw, u);
        float uh[2], sv[4];
        unpk2(u.h, uh[0], uh[1]);
        unpk2(sw.h, sv[0], sv[1]);
        unpk2(sw.l, sv[2], sv[3]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const bool in = q + e < ke && uh[e] > 0.0f;
          if (!in) sv[e] = sv[2 + e] = 0.0f;
          const float wt = sv[e] * sv[e];
          mw += wt;
#pragma unroll
          for (int c = 0; c < D; ++c) {
            const float x = row_of(xi[c], e).h;
            m1[c] = fmaf(wt, x, m1[c]);
            m2[c] = fmaf(wt * x, x, m2[c]);
          }
        }
#pragma unroll
        for (int c = 0; c < D; ++c) {
          *reinterpret_cast<f2*>(XH + c * kp + q) = xi[c].h;
          *reinterpret_cast<f2*>(XL + c * kp + q) = xi[c].l;
        }
        *reinterpret_cast<f2*>(SWH + q) = pk2(sv[0], sv[1]);
        *reinterpret_cast<f2*>(SWL + q) = pk2(sv[2], sv[3]);
      }
    }
    // centroid (the staggered columns vanish at the target: no shift there) and
    // the moments about it, then the coefficients of q_2 .. q_HI
    mw = 1.0f / gsum<G>(mw);
    float sh[D];
#pragma unroll
    for (int c = 0; c < D; ++c) sh[c] = ST ? 0.0f : gsum<G>(m1[c]) * mw;
    // axes to stretch (variances; a flat axis below 2^-40 of the widest is left)
    int ax = 0;
    {
      float vmax = 0.0f;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        m2[c] = fmaf(-sh[c], sh[c], gsum<G>(m2[c]) * mw);
        vmax = fmaxf(vmax, m2[c]);
      }
#pragma unroll
      for (int c = 0; c < D; ++c)
        if (m2[c] * 16.0f <= vmax && m2[c] > vmax * 0x1p-40f)
          ax |= (int)((__float_as_uint(__fdividef(vmax, m2[c])) >> 23) - 127u) >> 1 << (8 * c);
    }
    if (lane == 0) *AX = ax;
    __syncwarp();
    float mu[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // moments 2, 4, 6, 8
#pragma unroll 1
    for (int i = lane; i < pw; i += G) {
      float w0, w1;
      unpk2(row_pair(SWH, i), w0, w1);
      const f2 wt = pk2(w0 * w0, w1 * w1);
      f2 acc[4] = {0, 0, 0, 0};
#pragma unroll
      for (int c = 0; c < D; ++c) {
        ffp x{row_pair(XH + c * kp, i), row_pair(XL + c * kp, i)};
        if constexpr (!ST) {
          x = add_c(x, -sh[c]);
          x = quick2(x.h, x.l);
        }
        if (ax != 0) {
          const f2 f = dup2(sne_exp2((ax >> (8 * c)) & 255));
          x = ffp{mul2(x.h, f), mul2(x.l, f)};
        }
        if (!ST || ax != 0) {
          *reinterpret_cast<f2*>(XH + c * kp + 2 * i) = x.h;
          *reinterpret_cast<f2*>(XL + c * kp + 2 * i) = x.l;
        }
        const f2 s = mul2(x.h, x.h);
        f2 p = mul2(wt, s);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (e >= HI) break;
          acc[e] = add2(acc[e], p);
          p = mul2(p, s);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) mu[e] += sum2(acc[e]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) mu[e] = (e < HI) ? gsum<G>(mu[e]) * (mw / (float)D) : 0.0f;
    SneCoef cf;
    sne_coefficients<HI, ST>(mu, cf);
    // q, q', q'' at the target (eta = -centroid), float-float: entry (axis, power, derivative)
    float* LT = base + (DF ? Lay::X : Lay::LT);
    if (lane < D) {
      float s0 = sh[0];
#pragma unroll
      for (int c = 1; c < D; ++c)
        if (lane == c) s0 = sh[c];
      const float f = sne_exp2((ax >> (8 * lane)) & 255), f2nd = f * f;  // of the axis and its derivatives
      const ff x(-s0 * f, 0.0f), tt = x * x;
      float* o = LT + lane * 6 * (HI + 1);
      auto put = [&](int p, ff v, ff d1, ff d2) {
        o[6 * p] = v.h, o[6 * p + 1] = v.l, o[6 * p + 2] = d1.h * f, o[6 * p + 3] = d1.l * f;
        o[6 * p + 4] = d2.h * f2nd, o[6 * p + 5] = d2.l * f2nd;
      };
      const ff zero(0.f, 0.f), one(1.f, 0.f);
      put(0, one, zero, zero);
      put(1, x, one, zero);
      if constexpr (HI >= 2) put(2, add_f(tt, -cf.a), ff(2.f * x.h, 0.f), ff(2.f, 0.f));
      if constexpr (HI >= 3) put(3, x * add_f(tt, -cf.b), add_f(mul_f(tt, 3.f), -cf.b), mul_f(x, 6.f));
      if constexpr (HI >= 4)
        put(4, add_f(tt * add_f(tt, -cf.c), cf.d), x * add_f(mul_f(tt, 4.f), -2.f * cf.c), add_f(mul_f(tt, 12.f), -2.f * cf.c));
      if constexpr (HI >= 5) {
        const ff e3 = mul_f(ff(cf.e, 0.f), 3.f);
        put(5, x * add_f(tt * add_f(tt, -cf.e), cf.f), add_f(tt * (mul_f(tt, 5.f) - e3), cf.f),
            x * (mul_f(tt, 20.f) - mul_f(e3, 2.f)));
      }
    }
    __syncwarp();
    auto lt = [&](int axis, int col, int der) {
      const float* o = LT + (axis * (HI + 1) + tab.e[axis][col]) * 6 + 2 * der;
      return ff(o[0], o[1]);
    };
    auto lap_col = [&](int col) {  // Laplacian of column col at the target (unscaled)
      ff s(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < D; ++c) {
        ff p = lt(c, col, 2);
#pragma unroll
        for (int c2 = 0; c2 < D; ++c2)
          if (c2 != c) p = p * lt(c2, col, 0);
        s = s + p;
      }
      return s;
    };
    // int d_c: times 2^(s_c - s_0)
    [[maybe_unused]] const float st1 = sne_exp2(((ax >> 8) & 255) - (ax & 255)), st2 = sne_exp2(((ax >> 16) & 255) - (ax & 255));
    [[maybe_unused]] auto stretch = [&](int c) { return D == 2 || c == 1 ? st1 : st2; };
    // component-0 part of column i < NTOP over values ff v[.] (float-float): main + further term
    [[maybe_unused]] auto comp0 = [&](int i, const float* vh, const float* vl, int stride) {
      const int src = tab.src[i], xs = tab.xslot[i];
      ff r(0.f, 0.f);
      if (src >= 0) {
        const float f = stretch(1 + i / Q);
        r = ff(tab.mch[i] * f, tab.mcl[i] * f) * ff(vh[src * stride], vl[src * stride]);
      }
      if (xs >= 0) {
        const float* xc = base + Lay::XC + 2 * xs;
        const int x = tab.xsrc[xs] * stride;
        r = r + ff(xc[0], xc[1]) * ff(vh[x], vl[x]);
      }
      return r;
    };
    if constexpr (DF) {
      float* LP = base + Lay::LP;
      for (int g = lane; g < Q; g += G) {
        const ff v = lap_col(g);
        LP[2 * g] = v.h;
        LP[2 * g + 1] = v.l;
      }
      // further terms: q_3' = 3 q_2 + (3 a - b) q_0, q_4' = 4 q_3 + (4 b - 2 c) q_1;
      // int q_2 = q_3 / 3 + (b / 3 - a) q_1, int q_3 = q_4 / 4 + (c / 4 - b / 2) q_2
      for (int x = lane; x < tab.nx; x += G) {
        const int i = tab.xcol[x], c = 1 + i / Q, g = i % Q, g0 = tab.e[0][g], gc = tab.e[c][g];
        const ff a(cf.a, 0.f), b(cf.b, 0.f), cc(cf.c, 0.f);
        ff v;
        if (gc >= 3)
          v = (gc == 3 ? mul_f(a, 3.f) - b : mul_f(b, 4.f) - mul_f(cc, 2.f)) * recip(ff((float)(g0 + 1), 0.f));
        else
          v = mul_f(g0 == 2 ? b * recip(ff(3.f, 0.f)) - a : mul_f(cc, 0.25f) - mul_f(b, 0.5f), (float)gc);
        const float f = stretch(c);
        base[Lay::XC + 2 * x] = v.h * f;
        base[Lay::XC + 2 * x + 1] = v.l * f;
      }
      __syncwarp();
    }

    // ---- 2. A = Q_A R_A: blocks of P rows against the triangle
    float* RA = DF ? base + Lay::RA : R;
    for (int e = lane; e < Q * (Q + 1) / 2; e += G) RA[e] = 0.0f;
    int par = 0;
#pragma unroll 1
    for (int r0 = 0; r0 < pw; r0 += P / 2) {
      float* STG = base + Lay::ST;
#pragma unroll 1
      for (int i = lane; i < P / 2; i += G) {
        const int r = r0 + i;
        ffp x[D], m[Q], sw{0, 0};
#pragma unroll
        for (int c = 0; c < D; ++c) x[c] = ffp{0, 0};
        if (r < pw) {
#pragma unroll
          for (int c = 0; c < D; ++c) x[c] = ffp{row_pair(XH + c * kp, r), row_pair(XL + c * kp, r)};
          sw = ffp{row_pair(SWH, r), row_pair(SWL, r)};
        }
        sne_columns<D, LO, HI>(x, cf, m);
#pragma unroll
        for (int c = 0; c < Q; ++c)
          *reinterpret_cast<f2*>(STG + c * Lay::PS + 2 * i) = fma2(m[c].h, sw.h, fma2(m[c].h, sw.l, mul2(m[c].l, sw.h)));
      }
      __syncwarp();
      f2 a[SA][P / 2];
#pragma unroll
      for (int s = 0; s < SA; ++s) {
        const int c = s * G + lane;
        const ulonglong2* col = reinterpret_cast<const ulonglong2*>(STG + (c < Q ? c : 0) * Lay::PS);
#pragma unroll
        for (int i = 0; i < P / 4; ++i) {
          ulonglong2 v = col[i];
          if (s == SA - 1 && c >= Q) v = make_ulonglong2(0, 0);
          a[s][2 * i] = v.x;
          a[s][2 * i + 1] = v.y;
        }
      }
      sne_append<P, SA, Q, G>(a, RA, base + Lay::VB, lane, par);
    }
    __syncwarp();
    float cn[SA];  // column norms of A
#pragma unroll
    for (int s = 0; s < SA; ++s) {
      const int c = s * G + lane;
      float v = 0.0f;
      if (c < Q)
        for (int r = 0; r <= c; ++r) v = fmaf(RA[rpk<Q>(r, c)], RA[rpk<Q>(r, c)], v);
      cn[s] = sqrtf(v);
    }
    if constexpr (DF) {
      // ---- 3. G = (I (x) R_A) C: diag(R_A, ..) above, the component-0 rows eliminated against it
      constexpr int PG = Lay::PG;
      for (int e = lane; e < Lay::NR; e += G) R[e] = 0.0f;
      __syncwarp();
      f2 a[SN][PG / 2];
#pragma unroll
      for (int s = 0; s < SN; ++s) {
        const int col = s * G + lane;
        float v[PG];
#pragma unroll
        for (int r = 0; r < PG; ++r) v[r] = 0.0f;
        auto add_column = [&](int src, float co) {
#pragma unroll
          for (int r = 0; r < Q; ++r)
            if (src >= r) v[r] = fmaf(co, RA[rpk<Q>(r, src)], v[r]);
        };
        if (col < NTOP) {
          const int b0 = col / Q * Q, cg = col - b0, xs = tab.xslot[col];
          if (tab.src[col] >= 0) add_column(tab.src[col], -tab.mch[col] * stretch(1 + col / Q));
          if (xs >= 0) add_column(tab.xsrc[xs], -base[Lay::XC + 2 * xs]);
          for (int r = 0; r <= cg; ++r) R[rpk<N>(b0 + r, col)] = RA[rpk<Q>(r, cg)];
        } else if (col < N) {
          add_column(tab.f0[col - NTOP], 1.0f);
        }
#pragma unroll
        for (int r = 0; r < PG / 2; ++r) a[s][r] = pk2(v[2 * r], v[2 * r + 1]);
      }
      __syncwarp();
      sne_append<PG, SN, N, G>(a, R, base + Lay::VB, lane, par);
      __syncwarp();
    }
    // 1 / r_ii and the conditioning of the factor on the Taylor scale (1 / b!, axes as they are)
    float dmx = 0.0f, dmn = 3.0e38f;
#pragma unroll
    for (int s = 0; s < SN; ++s) {
      const int p = s * G + lane;
      if (p < N) {
        const float d = R[rpk<N>(p, p)];
        ID[p] = 1.0f / d;
        const int col = DF ? (p < NTOP ? p % Q : tab.f0[p < NTOP ? 0 : p - NTOP]) : p;
        float sc = fabsf(d);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const int e = tab.e[c][col];
          sc *= e < 2 ? 1.0f : e == 2 ? 0.5f : e == 3 ? 1.0f / 6.0f : e == 4 ? 1.0f / 24.0f : 1.0f / 120.0f;
          if (ax != 0) sc *= sne_exp2(-e * ((ax >> (8 * c)) & 255));
        }
        dmx = fmaxf(dmx, sc);
        dmn = sc > 0.0f ? fminf(dmn, sc) : 0.0f;  // (zero and NaN)
      }
    }
    dmx = gmax<G>(dmx);
    dmn = -gmax<G>(-dmn);
    const bool ill = !(dmn * 1.0e6f >= dmx) || !(dmn > 0.0f);
    // no estimate from one step (which left up to 1e-8) where the columns are far from
    // orthogonal -- some r_ii below 1/20 of its column, on flattened and rotated
    // clouds; 99 % of the targets of jittered ones stay above 1/8 -- or few
    // neighbours carry the weight (powers from 10 on)
    bool second = j.wpow_half >= 5;
    [[maybe_unused]] bool skewed = false;
    if constexpr (!DF) {
      float off = 0.0f;
#pragma unroll
      for (int s = 0; s < SA; ++s)
        if (s * G + lane < Q) off = fmaxf(off, cn[s] * fabsf(ID[s * G + lane]));
      off = gmax<G>(off);
      second |= off > 20.0f;
      // (the staggered columns then carry roundings of their own, 3e-9 after two steps)
      skewed = ST && off > 40.0f;
    }
    second = second && j.max_refine > 1;
    __syncwarp();

    // functional rows at unknown i (float-float): rows of the gradient, then the
    // Laplacian (L = 1: the Laplacian alone; Neumann: then the normal derivative);
    // divergence-free: the vector Laplacian
    [[maybe_unused]] ff nv[D], in2;
    [[maybe_unused]] float b0 = 0.0f;  // beta_0 of the Laplacian row, once known
    [[maybe_unused]] float fs = 1.0f;  // power of two that brings s_f (about |n| / eps, scaled) to order one
    if constexpr (NEU) {
      ff n2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < D; ++c) {
        nv[c] = ff(j.normals[c * n + t]);
        n2 = n2 + nv[c] * nv[c];
      }
      in2 = recip(n2);
      fs = sne_exp2(-eps_exponent() - (((int)((__float_as_uint(n2.h) >> 23) & 0xffu) - 127) >> 1));
    }
    auto lam = [&](int i, ff (&v)[LR]) {
      if constexpr (DF) {
        const float* LP = base + Lay::LP;
        const int c = i < NTOP ? 1 + i / Q : 0, g = i < NTOP ? i % Q : tab.f0[i - NTOP];
        const ff own = ff(LP[2 * g], LP[2 * g + 1]) * ie2;
#pragma unroll
        for (int l = 0; l < L; ++l) v[l] = l == c ? own : ff(0.f, 0.f);
        if (c > 0) v[0] = -comp0(i, LP, LP + 1, 2) * ie2;
      } else {
        ff p[D];  // products of the other axes' values
        if constexpr (D == 2) {
          p[0] = lt(1, i, 0);
          p[1] = lt(0, i, 0);
        } else {
          const ff a = lt(0, i, 0), b = lt(1, i, 0), c = lt(2, i, 0);
          p[0] = b * c;
          p[1] = a * c;
          p[2] = a * b;
        }
        ff lap(0.f, 0.f), nd(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          if (L != D) lap = lap + p[c] * lt(c, i, 2);
          if (L >= D) {
            v[c < LR ? c : 0] = p[c] * lt(c, i, 1) * ie1;
          }
        }
        if constexpr (NEU) {
          static_assert(!NEU || L > D, "gradient and Laplacian rows");
#pragma unroll
          for (int c = 0; c < D; ++c) nd = nd + nv[c] * v[c];
          ff tg[D];  // tangential parts: sum_b n_b (n_b g_c - n_c g_b) / |n|^2
#pragma unroll
          for (int c = 0; c < D; ++c) tg[c] = ff(0.f, 0.f);
#pragma unroll
          for (int b = 0; b < D; ++b)
#pragma unroll
            for (int c = b + 1; c < D; ++c) {
              const ff x = (nv[b] * v[c] - nv[c] * v[b]) * in2;
              tg[c] = tg[c] + nv[b] * x;
              tg[b] = tg[b] - nv[c] * x;
            }
#pragma unroll
          for (int c = 0; c < D; ++c) v[c] = tg[c];
        }
        if (L != D) v[L == 1 ? 0 : D < LR ? D : 0] = lap * ie2;
        if constexpr (NEU) {
          v[D] = v[D] - mul_f(nd, b0);
          v[L] = nd;
        }
      }
    };
    float w[LR][SN];
#pragma unroll
    for (int s = 0; s < SN; ++s) {
      ff v[LR];
      lam(s * G + lane < N ? s * G + lane : 0, v);
#pragma unroll
      for (int l = 0; l < LR; ++l) w[l][s] = s * G + lane < N ? v[l].h : 0.0f;
    }
    // C y for the unknowns in Y (divergence-free basis) into u: component c of (l, c), column g
    [[maybe_unused]] auto spread = [&]() {
      auto entry = [&](int e) {
        const int lc = e / Q, g = e - lc * Q, l = lc / D, c = lc - l * D;
        const float* y = Y + l * N;
        if (c >= 1) return ff(y[(c - 1) * Q + g], 0.f);
        if (tab.fidx[g] >= 0) return ff(y[NTOP + tab.fidx[g]], 0.f);
        ff uv(0.f, 0.f);
#pragma unroll
        for (int c2 = 1; c2 < D; ++c2) {
          const int i = tab.inv[c2][g];
          if (i >= 0) {
            const float f = stretch(c2);
            uv = uv - mul_f(ff(tab.mch[i] * f, tab.mcl[i] * f), y[i]);
          }
        }
        if constexpr (Lay::Y_IN_U) {
#pragma unroll 1
          for (int x = 0; x < tab.nx; ++x)
            if (tab.xsrc[x] == g) uv = uv - mul_f(ff(base[Lay::XC + 2 * x], base[Lay::XC + 2 * x + 1]), y[tab.xcol[x]]);
        }
        return uv;
      };
      auto put = [&](int e, ff v) {
        UH[ux(e / Q, e % Q)] = v.h;
        UL[ux(e / Q, e % Q)] = v.l;
      };
      if constexpr (Lay::Y_IN_U) {
        constexpr int IT = (LC * Q + G - 1) / G;
        ff u[IT];
#pragma unroll
        for (int i = 0; i < IT; ++i) u[i] = i * G + lane < LC * Q ? entry(i * G + lane) : ff(0.f, 0.f);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < IT; ++i)
          if (i * G + lane < LC * Q) put(i * G + lane, u[i]);
      } else {
        for (int e = lane; e < LC * Q; e += G) put(e, entry(e));
        __syncwarp();
        if (lane < L)
          for (int x = 0; x < tab.nx; ++x) {
            const int a = ux(lane * D, tab.xsrc[x]);
            const ff uv = ff(UH[a], UL[a]) - mul_f(ff(base[Lay::XC + 2 * x], base[Lay::XC + 2 * x + 1]), Y[lane * N + tab.xcol[x]]);
            UH[a] = uv.h;
            UL[a] = uv.l;
          }
      }
    };
    bool conv = false, hand = false;
    int used = 0;
    float prev = 0.0f;
    [[maybe_unused]] bool beta_ok = true;
#pragma unroll 1
    for (int step = 0; step <= j.max_refine; ++step) {
      const bool pending = active && !ill && !conv && !hand;
      if (!__any_sync(FULL, pending)) break;
      if (step > 0) {
        // ---- 5. s0 = B y0 (first step; later ones take s as stored) and B^T s
#pragma unroll 1
        for (int r0 = 0; r0 < RHS; r0 += LS) {
          constexpr int NP = LS / 2;  // pairs of right-hand sides
          auto mg = [&](int i, int g) {
            const int ra = r0 + 2 * i, rb = ra + 1;
            return pk2(MG[(ra < LC ? ra / NC : 0) * QP + g], MG[(rb < LC ? rb / NC : 0) * QP + g]);
          };
          f2 ah[NP][Q], al[NP][Q];
#pragma unroll
          for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int g = 0; g < Q; ++g) {
              ah[i][g] = step == 1 ? mg(i, g) : 0;
              al[i][g] = 0;
            }
#pragma unroll 1
          for (int q = lane; q < 2 * pw; q += G) {
            ff x[D], m[Q];
#pragma unroll
            for (int d = 0; d < D; ++d) x[d] = ff(XH[d * kp + q], XL[d * kp + q]);
            sne_columns<D, LO, HI>(x, cf, m);
            const ffp sw{dup2(SWH[q]), dup2(SWL[q])};
            ffp tv[NP];
            if (step == 1) {
              if (r0 == 0) {
                float rn[2] = {0.0f, 0.0f};
#pragma unroll
                for (int g = 0; g < Q; ++g) {
                  const float v = m[g].h * IC[g];
                  rn[g & 1] = fmaf(v, v, rn[g & 1]);
                }
                const float nn = fmaxf(rn[0] + rn[1], 1e-30f);  // (the staggered columns vanish at the target)
                RN[q] = sne_magic(nn * rsqrtf(nn));
              }
              const float rn = RN[q];
#pragma unroll
              for (int i = 0; i < NP; ++i) {
                // (Cauchy-Schwarz over the columns, each scaled to unit length)
                const int ri = r0 + 2 * i;
                const f2 ms = mul2(dup2(rn), *reinterpret_cast<const f2*>(MS + ri));
                constexpr int CH = 2;  // independent chains
                f2 sh2[CH], sl2[CH];
#pragma unroll
                for (int e = 0; e < CH; ++e) {
                  sh2[e] = ms;
                  sl2[e] = 0;
                }
#pragma unroll
                for (int g = 0; g < Q; g += 2) {
                  const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(UH + ux(ri, g));
                  if constexpr (DF) {
                    const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(UL + ux(ri, g));
                    sne_acc(sh2[0], sl2[0], m[g], ffp{b.x, c.x});
                    if (g + 1 < Q) sne_acc(sh2[1], sl2[1], m[g + 1 < Q ? g + 1 : 0], ffp{b.y, c.y});
                  } else {
                    sne_acc(sh2[0], sl2[0], m[g], b.x);
                    if (g + 1 < Q) sne_acc(sh2[1], sl2[1], m[g + 1 < Q ? g + 1 : 0], b.y);
                  }
                }
                // exact: each chain's sum is a multiple of the same ulp, their total below the constant
                const f2 th = add2(sub2(sh2[0], ms), sub2(sh2[1], ms)), tl = add2(sl2[0], sl2[1]);
                const ffp s = mul_ff(quick2(th, tl), sw);
                S0[(ri >> 1) * kp + q] = make_ulonglong2(s.h, s.l);
                tv[i] = mul_ff(s, sw);
              }
            } else {
#pragma unroll
              for (int i = 0; i < NP; ++i) {
                const ulonglong2 s = S0[((r0 >> 1) + i) * kp + q];
                tv[i] = mul_ff(ffp{s.x, s.y}, sw);
              }
            }
            if (step == 1) {
#pragma unroll
              for (int i = 0; i < NP; ++i)
#pragma unroll
                for (int g = 0; g < Q; ++g) sne_acc(ah[i][g], al[i][g], m[g], tv[i]);
            } else {
#pragma unroll
              for (int i = 0; i < NP; ++i)
#pragma unroll
                for (int g = 0; g < Q; ++g) sne_acc_twosum(ah[i][g], al[i][g], m[g], tv[i]);
            }
          }
          constexpr int C = (LS * Q + G - 1) / G * G, SH = C / G;
          float vh[C], vl[C];
#pragma unroll
          for (int e = LS * Q; e < C; ++e) vh[e] = vl[e] = 0.0f;
#pragma unroll
          for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int g = 0; g < Q; ++g) {
              if (step == 1) ah[i][g] = sub2(ah[i][g], mg(i, g));
              unpk2(ah[i][g], vh[2 * i * Q + g], vh[(2 * i + 1) * Q + g]);
              unpk2(al[i][g], vl[2 * i * Q + g], vl[(2 * i + 1) * Q + g]);
            }
          if (step == 1) {  // exact in the high parts: multiples of one ulp below the constant
            sne_reduce_scatter<G>(vh, lane);
            sne_reduce_scatter<G>(vl, lane);
          } else {
            sne_reduce_scatter<G>(vh, vl, lane);
          }
          __syncwarp();  // u of these right-hand sides has been read: v takes its place
#pragma unroll
          for (int i = 0; i < SH; ++i) {
            const int e = lane * SH + i, ri = e / Q, g = e - ri * Q;
            if (e < LS * Q) {
              const ff v = quick_two_sum(vh[i], vl[i]);
              UH[ux(r0 + ri, g)] = v.h;
              UL[ux(r0 + ri, g)] = v.l;
            }
          }
        }
        __syncwarp();
        // g = lambda - B^T s
#pragma unroll
        for (int s = 0; s < SN; ++s) {
          const int i = s * G + lane;
          ff v[LR];
          lam(i < N ? i : 0, v);
#pragma unroll
          for (int l = 0; l < LR; ++l) {
            float gv = 0.0f;
            if (i < N) {
              ff ct;
              if constexpr (DF) {
                const int c = i < NTOP ? 1 + i / Q : 0, g = i < NTOP ? i % Q : tab.f0[i < NTOP ? 0 : i - NTOP];
                ct = ff(UH[ux(l * D + c, g)], UL[ux(l * D + c, g)]);
                if (c >= 1) ct = ct - comp0(i, UH + ux(l * D, 0), UL + ux(l * D, 0), 2);
              } else {
                ct = ff(UH[ux(l, i)], UL[ux(l, i)]);
              }
              const ff gg = v[l] - ct;
              gv = __fadd_rn(gg.h, gg.l);
            }
            w[l][s] = gv;
          }
        }
        __syncwarp();
      }
      // ---- 4. y = R^-1 R^-T w
      sne_solve<N, LR, G, SN, true>(R, ID, w, lane);
      if constexpr (NEU)
        if (step == 0) {  // s . s' = (R^-T lambda) . (R^-T lambda')
          float num = 0.0f, den = 0.0f;
#pragma unroll
          for (int s = 0; s < SN; ++s)
            if (s * G + lane < N) {
              num = fmaf(w[D][s], w[L][s], num);
              den = fmaf(w[L][s], w[L][s], den);
            }
          b0 = gsum<G>(num) / gsum<G>(den);
          if (!(fabsf(b0) < 1e30f)) b0 = 0.0f;
#pragma unroll
          for (int s = 0; s < SN; ++s) w[D][s] = fmaf(-b0, w[L][s], w[D][s]);
        }
      if (step == 0) {
        // accumulator constants of B^T s: |A e_q| |s|, |s| = |R^-T lambda|
#pragma unroll
        for (int l = 0; l < LR; ++l) {
          float v = 0.0f;
#pragma unroll
          for (int s = 0; s < SN; ++s)
            if (s * G + lane < N) v = fmaf(w[l][s], w[l][s], v);
          v = sqrtf(gsum<G>(v));
#pragma unroll
          for (int s = 0; s < SA; ++s)
            if (s * G + lane < Q) MG[l * QP + s * G + lane] = sne_magic(v * cn[s]);
        }
#pragma unroll
        for (int s = 0; s < SA; ++s)
          if (s * G + lane < Q) IC[s * G + lane] = 1.0f / cn[s];
      }
      sne_solve<N, LR, G, SN, false>(R, ID, w, lane);
      if constexpr (DF) {
#pragma unroll
        for (int l = 0; l < LR; ++l)
#pragma unroll
          for (int s = 0; s < SN; ++s)
            if (s * G + lane < N) Y[l * N + s * G + lane] = w[l][s];
        __syncwarp();
        spread();
      } else {
#pragma unroll
        for (int l = 0; l < LR; ++l)
#pragma unroll
          for (int s = 0; s < SN; ++s)
            if (s * G + lane < N) UH[ux(l, s * G + lane)] = w[l][s];
      }
#pragma unroll
      for (int r = LC; r < RHS; ++r)  // the last pass's spare right-hand sides
        for (int g = lane; g < Q; g += G) UH[ux(r, g)] = UL[ux(r, g)] = 0.0f;
      __syncwarp();
      if (step == 0) {
        // root of sum_q (u_q |A e_q|)^2, for the accumulator constants of B y0
#pragma unroll 1
        for (int r = 0; r < RHS; ++r) {
          float v = 0.0f;
#pragma unroll
          for (int s = 0; s < SA; ++s) {
            const int c = s * G + lane;
            if (c < Q) v = fmaf(UH[ux(r, c)] * cn[s], UH[ux(r, c)] * cn[s], v);
          }
          v = sqrtf(gsum<G>(v));
          if (lane == 0) MS[r] = sne_pow2(v);
        }
        __syncwarp();
        continue;
      }
      // ---- 6. s += B dy, w = sqrt(W) s (stored by targets still in the loop)
      // the weights' destinations: row l of the solve serves at most two functionals
      for (int r = lane; r < L * NC; r += G) {
        const int l = r / NC, cc = r - l * NC;
        SneDst* d = reinterpret_cast<SneDst*>(base + Lay::DST) + 2 * r;
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
      __syncwarp();
      float dmax = 0.0f, smax = 0.0f;
      // a correction that is not finite (the maxima below drop NaN) hands the target on
#pragma unroll
      for (int l = 0; l < LR; ++l)
#pragma unroll
        for (int s = 0; s < SN; ++s)
          if (s * G + lane < N && !(fabsf(w[l][s]) < 3e38f)) dmax = 3e38f;
      [[maybe_unused]] double others[L];
      [[maybe_unused]] Dot2 pb[LR];
      [[maybe_unused]] auto scale = [&](ff v) { return ff(v.h * fs, v.l * fs); };
      if constexpr (ST) {
#pragma unroll
        for (int l = 0; l < L; ++l) others[l] = 0.0;
      }
      // the weights of row q, right-hand side r
      const SneDst* dst = reinterpret_cast<const SneDst*>(base + Lay::DST);
      const float so = sne_exp2(-ORDER * eps_exponent());
      auto store = [&](int q, int r, ff wv) {
        const double val = sne_to_double(wv);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const SneDst d = dst[2 * r + e];
          if (d.p && !(ST && q == self)) __stcs(d.p + (int64_t)q * d.stride, d.sgn < 0.0f ? -val : val);
        }
        return val;
      };
#pragma unroll 1
      for (int q = lane; q < ke; q += G) {
        if (!pending) break;
        float x[D], m[Q];
#pragma unroll
        for (int d = 0; d < D; ++d) x[d] = XH[d * kp + q];
        sne_columns<D, LO, HI>(x, cf, m);
        const ffp sw{dup2(SWH[q]), dup2(SWL[q])}, swo{dup2(SWH[q] * so), dup2(SWL[q] * so)};
        [[maybe_unused]] ff sf;  // Neumann: the constraint's right-hand side, taken first
        constexpr int PR = (LC + 1) / 2, PF = NEU ? L / 2 : 0;  // pairs; the first one taken
        ulonglong2 sn = S0[PF * kp + q];
#pragma unroll 1
        for (int i = 0; i < PR; ++i) {
          const int pr = NEU ? (i == 0 ? PF : i - (i <= PF ? 1 : 0)) : i;
          const ulonglong2 s0 = sn;
          if (i + 1 < PR) sn = S0[(NEU ? i + 1 - (i + 1 <= PF ? 1 : 0) : i + 1) * kp + q];  // the next one's load in flight
          f2 d0 = 0, d1 = 0;
#pragma unroll
          for (int g = 0; g < Q; g += 2) {
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(UH + 2 * (pr * QP + g));
            d0 = fma2(dup2(m[g]), b.x, d0);
            if (g + 1 < Q) d1 = fma2(dup2(m[g + 1 < Q ? g + 1 : 0]), b.y, d1);
          }
          const f2 ds = mul2(add2(d0, d1), sw.h);
          // s0 + ds
          ffp s1;
          {
            const f2 h = add2(s0.x, ds), bb = sub2(h, s0.x);
            s1 = quick2(h, add2(add2(sub2(s0.x, sub2(h, bb)), sub2(ds, bb)), s0.y));
          }
          S0[pr * kp + q] = make_ulonglong2(s1.h, s1.l);
          const bool two = 2 * pr + 1 < LC;
          float a0, a1, b0, b1;
          unpk2(ds, a0, a1);
          unpk2(s1.h, b0, b1);
          dmax = fmaxf(dmax, fabsf(a0));
          smax = fmaxf(smax, fabsf(b0));
          if (two) {
            dmax = fmaxf(dmax, fabsf(a1));
            smax = fmaxf(smax, fabsf(b1));
          }
          if constexpr (NEU) {
            if (i == 0) sf = scale(row_of(s1, L & 1));
#pragma unroll
            for (int l = 0; l < LR; ++l)
              if (l >> 1 == pr) pb[l].add_prod(l == L ? sf : row_of(s1, l & 1), sf);
          } else {
            const ffp wv = mul_ff(s1, swo);
            const double v0 = store(q, 2 * pr, row_of(wv, 0));
            double v1 = 0.0;
            if (two) v1 = store(q, 2 * pr + 1, row_of(wv, 1));
            if constexpr (ST) {
              if (q != self)
#pragma unroll
                for (int l = 0; l < L; ++l)
                  if (l >> 1 == pr) others[l] += (l & 1) ? v1 : v0;
            }
          }
        }
      }
      dmax = gmax<G>(dmax);
      smax = gmax<G>(smax);
      if constexpr (ST) {
        // the target's own entry: minus the sum of the others
#pragma unroll
        for (int l = 0; l < L; ++l)
#pragma unroll
          for (int o = G / 2; o > 0; o >>= 1) others[l] += __shfl_xor_sync(FULL, others[l], o, G);
        if (pending && lane == 0)
          for (int f = 0; f < j.nout; ++f)
#pragma unroll
            for (int l = 0; l < L; ++l) {
              const int rr = l - j.out_src[f];
              if (j.out_src[f] >= 0 && rr >= 0 && rr < j.out_rows[f])
                j.out_w[f][(o0 * j.out_rows[f] + (int64_t)rr * k) + self] = -others[l];
            }
      }
      if constexpr (NEU) {
        ff bt[L];
        beta_ok = true;
        const ff ff2 = recip(gsum<G>(pb[L].value()));
#pragma unroll
        for (int l = 0; l < L; ++l) {
          bt[l] = gsum<G>(pb[l].value()) * ff2;
          beta_ok = beta_ok && fabsf(bt[l].h) < 1e30f;  // (false for NaN)
          // (s = s_lambda - bt (fs s_f): beta = fs bt)
          if (pending && lane == 0 && j.beta) j.beta[to * L + l] = to_double(l < D ? scale(bt[l]) + nv[l < D ? l : 0] * in2 : add_f(scale(bt[l]), b0));
        }
#pragma unroll 1
        for (int q = lane; q < ke; q += G) {
          if (!pending) break;
          ffp sp[(LR + 1) / 2];
#pragma unroll
          for (int i = 0; i < (LR + 1) / 2; ++i) {
            const ulonglong2 v = S0[i * kp + q];
            sp[i] = ffp{v.x, v.y};
          }
          const ff sf = scale(row_of(sp[L / 2], L & 1)), sw(SWH[q] * so, SWL[q] * so);
#pragma unroll
          for (int l = 0; l < L; ++l) store(q, l, (row_of(sp[l / 2], l & 1) - bt[l] * sf) * sw);
        }
      }
      if (pending) {
        // error left ~ |ds| times the contraction, estimated by the correction's
        // relative size (first step) or the ratio of successive corrections
        const float rho = step == 1 ? dmax / fmaxf(smax, 1e-37f) : dmax / fmaxf(prev, 1e-37f);
        conv = kSafe * dmax * fminf(1.0f, rho) <= tolf * smax && (step > 1 || !second);
        prev = dmax;
        used = step;
        // kappa above about 300: u's cancelling entries leave their roundings in
        // s0, where no further step reaches them; the shared-memory FP32 kernel,
        // which starts from Q, takes the target
        hand = step == 1 && rho > 5e-5f && j.max_refine > 1;
        // no finite beta (a zero normal): its weights are that kernel's too
        if (NEU && !beta_ok) hand = true;
        if (ST && skewed && j.max_refine > 1) hand = true;
        conv = conv && !hand;
      }
      __syncwarp();
    }
    if (active && !conv) {
      if (lane == 0 && hand) {
        j.gen_items[atomicAdd(j.gen_count, 1)] = (int32_t)to;
        j.status[to] = 0;
      } else if (lane == 0) {
        j.fb_items[atomicAdd(j.fb_count, 1)] = (int32_t)to;
        j.status[to] = ill ? GMLS_T_ILL_CONDITIONED : GMLS_T_REFINE_NOT_CONVERGED;
      }
    } else if (active) {
      for (int f = 0; f < j.nout; ++f)
        if (j.out_src[f] < 0) {
          const int64_t cnt = (int64_t)j.out_rows[f] * k * j.out_ncomp[f];
          double* wz = j.out_w[f] + o0 * (int64_t)j.out_rows[f] * j.out_ncomp[f];
          for (int64_t e = lane; e < cnt; e += G) wz[e] = 0.0;
        }
      if (j.beta && !NEU)
        for (int l = lane; l < L; l += G) j.beta[to * L + l] = 0.0;
      if (lane == 0) {
        j.status[to] = st;
        if (j.iters) j.iters[to] = (uint8_t)used;
      }
    }
    __syncwarp();
  }
}

// ----------------------------------------------------------------- dispatch
struct SneEntry {
  int kind, dim, deg, L, neu, G, maxt, rhs;
  const void* fn;
  int (*stride)(int kp);  // floats of shared memory per group
  SneTab (*tab)();
};

// What the tables' G, P, LS and MAXT follow:
//  * G: eight lanes up to 26 unknowns, 16 for 35 to 50, a warp for 85 -- the
//    triangle and the right-hand sides of 32 / G targets have to leave room for 8 to
//    12 warps in 227 KB;
//  * P: rows a lane keeps per block, whole blocks for the library's default lists
//    (12, 20 and 36 neighbours in one; 40 in two of 20; 84 in three of 28); any
//    other list runs ceil(k / P) blocks, 37 neighbours at degree 4 two of 36;
//  * LS: four right-hand sides a pass where their 2 Q LS accumulators fit beside the
//    columns (most bases of up to ten columns), else two;
//  * MAXT: 384 threads (168 registers), 512 (128) for the smallest scalar bases, 256
//    (255) for 35 columns and 85 unknowns; spills of up to about 300 bytes remain.
// Neumann rows have the gradient-and-Laplacian set only: the Laplacian alone goes to
// the shared-memory kernel.
#define GMLS_SNE(KIND, D, DEG, L, G, P, LS, NEU, MAXT)                                                              \
  SneEntry {                                                                                                        \
    KIND, D, DEG, L, NEU, G, MAXT, SneLay<KIND, D, DEG, L, G, P, LS, NEU>::RHS,                                     \
        (const void*)stencil_sne_kernel<KIND, D, DEG, L, G, P, LS, NEU, MAXT>,                                      \
        &SneLay<KIND, D, DEG, L, G, P, LS, NEU>::stride,                                                            \
        &make_sne_tab<D, SneDims<KIND, D, DEG, NEU>::LO, SneDims<KIND, D, DEG, NEU>::HI>                            \
  }

}  // namespace gmls
