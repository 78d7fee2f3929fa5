// Device helpers shared by the spreading, interpolation, direct-sum and
// solve kernels.
#pragma once

#include <cuda_runtime.h>

#include "checked.cuh"
#include "internal.h"

namespace fk {

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

template <typename T>
__device__ __forceinline__ T inv_h_of(const GeoDev& g, int j);
template <>
__device__ __forceinline__ float inv_h_of<float>(const GeoDev& g, int j) { return g.inv_h_f[j]; }
template <>
__device__ __forceinline__ double inv_h_of<double>(const GeoDev& g, int j) { return g.inv_h[j]; }

// Spreading kernel phi at offset z (fine cells): exponential of semicircle
// exp(beta (sqrt(1 - (2z/w)^2) - 1)) on |z| <= w/2, or the truncated Gaussian
// exp(-beta z^2) of eq. 17.
template <typename T>
__device__ __forceinline__ T phi(int kind, int w, T beta, T z) {
  if (kind == FKREG_SPREAD_ES) {
    const T t = z * (T(2) / T(w));
    const T a = T(1) - t * t;
    return a > T(0) ? exp(beta * (sqrt(a) - T(1))) : T(0);
  }
  return (fabs(z) <= T(0.5) * T(w)) ? exp(-beta * z * z) : T(0);
}

// FP32: the same kernels from the hardware reciprocal square root and base-2
// exponential (rsqrtf, exp2f), with exp(x) = 2^(x log2 e).  sqrt(a) is taken
// as s = a rsqrt(a) plus one Newton step on the exact residual a - s^2
// (fmaf), which brings s to within about one unit in the last place, as a
// correctly rounded square root would be; the exponent beta log2e (s - 1) is
// one fused multiply-add.  The error of the value, relative, stays near
// beta 2^-23 at the centre (the amplification of the rounding of s that the
// formula itself has) and far below the FP32 tolerance of the transform.
template <>
__device__ __forceinline__ float phi<float>(int kind, int w, float beta, float z) {
  constexpr float kLog2e = 1.4426950408889634f;
  const float bl = beta * kLog2e;
  if (kind == FKREG_SPREAD_ES) {
    const float t = z * (2.f / float(w));
    const float a = fmaf(-t, t, 1.f);
    if (!(a > 0.f)) return 0.f;
    const float r = rsqrtf(a);
    float s = a * r;
    s = fmaf(0.5f * r, fmaf(-s, s, a), s);
    return exp2f(fmaf(s, bl, -bl));
  }
  return (fabsf(z) <= 0.5f * float(w)) ? exp2f(-bl * z * z) : 0.f;
}

// All W kernel values phi(off + t), t = 0 .. W-1, of one axis (off is the first
// cell's offset, in [-w/2, -w/2 + 1)).  FP32: phi at each.  FP64: with
// x = off + (W - 1)/2 in [-1/2, 1/2) the taps lie at x +- c, and each pair is
// phi(x +- c) = E_c(x^2) +- x O_c(x^2) with polynomials of eight coefficients
// fitted when the plan is made (PhiPoly), right to 2e-16 of the peak; the two
// outermost taps, where the square root ends, are evaluated.  A pair costs 16
// instructions on the FP64 pipe (one warp instruction per SM and 16 clocks)
// where two square roots and exponentials take some 90.
template <typename T>
struct PhiTab {};  // FP32 needs no table
template <>
struct PhiTab<double> {
  PhiPoly p;
};
template <int W>
__device__ __forceinline__ void phi_row(const PhiTab<float>&, int skind, float beta, float off,
                                        float (&v)[W]) {
#pragma unroll
  for (int t = 0; t < W; ++t) v[t] = phi<float>(skind, W, beta, off + float(t));
}
template <typename T>
__device__ __noinline__ T phi_call(int skind, int w, T beta, T z) {
  return phi<T>(skind, w, beta, z);
}
template <int W>
__device__ __forceinline__ void phi_row(const PhiTab<double>& tab, int skind, double beta,
                                        double off, double (&v)[W]) {
  const double x = off + 0.5 * (W - 1), y = x * x;
  v[0] = phi_call<double>(skind, W, beta, off);
  v[W - 1] = phi_call<double>(skind, W, beta, off + (W - 1));
#pragma unroll
  for (int k = 1; k < (W + 1) / 2; ++k) {
    double e = tab.p.e[k][kPhiTerms - 1], o = tab.p.o[k][kPhiTerms - 1];
#pragma unroll
    for (int j = kPhiTerms - 2; j >= 0; --j) {
      e = fma(e, y, tab.p.e[k][j]);
      if (2 * k != W - 1) o = fma(o, y, tab.p.o[k][j]);
    }
    if (2 * k == W - 1) {
      v[k] = e;
    } else {  // tap k lies at x - c, its mirror at x + c
      v[k] = fma(-x, o, e);
      v[W - 1 - k] = fma(x, o, e);
    }
  }
}

// Compile-time chain of the monomials of degree <= DEG in d = D variables, in
// the graded order the plan's monomial table uses (degree by degree, index
// multisets in lexicographic order): monomial f > 0 is monomial parent[f]
// times coordinate axis[f].  The monomials of degree <= l are a prefix.
struct MonoChain {
  int n;
  int parent[kMaxMono];
  int axis[kMaxMono];
};

__host__ __device__ constexpr MonoChain make_mono_chain(int D, int DEG) {
  MonoChain c{0, {}, {}};
  int e[kMaxMono][3] = {};
  for (int k = 0; k <= DEG; ++k) {
    int idx[4] = {0, 0, 0, 0};
    for (;;) {
      const int m = c.n;
      for (int j = 0; j < 3; ++j) e[m][j] = 0;
      for (int j = 0; j < k; ++j) e[m][idx[j]] += 1;
      c.parent[m] = 0;
      c.axis[m] = 0;
      if (k > 0) {
        const int ax = idx[k - 1];
        c.axis[m] = ax;
        for (int r = 0; r < m; ++r) {
          bool same = true;
          for (int j = 0; j < 3; ++j)
            if (e[r][j] != e[m][j] - (j == ax ? 1 : 0)) same = false;
          if (same) {
            c.parent[m] = r;
            break;
          }
        }
      }
      c.n = m + 1;
      int p = k - 1;
      while (p >= 0 && idx[p] == D - 1) --p;
      if (p < 0) break;
      idx[p] += 1;
      for (int j = p + 1; j < k; ++j) idx[j] = idx[p];
    }
  }
  return c;
}

__host__ __device__ constexpr int mono_count(int D, int DEG) { return make_mono_chain(D, DEG).n; }

template <typename T, int D, int DEG, int F = 0>
__device__ __forceinline__ void mono_build(T* mo, const T* z) {
  if constexpr (F < mono_count(D, DEG)) {
    if constexpr (F == 0) {
      mo[0] = T(1);
    } else {
      constexpr int pf = make_mono_chain(D, DEG).parent[F];
      constexpr int af = make_mono_chain(D, DEG).axis[F];
      mo[F] = mo[pf] * z[af];
    }
    mono_build<T, D, DEG, F + 1>(mo, z);
  }
}

// Candidate bins of a support query for points whose coordinates (relative
// to lo) span [mn_j, mx_j] on each axis.  box(): the bins of the leading axes
// and the full range of the last axis; row(): one row of leading-axis bins,
// i.e. a run of bins adjacent along the last axis (one contiguous range of
// the sort).  With a diagonal H the row's last-axis range is cut to the
// section of the support ellipsoid nearest to the points: a sample whose
// leading coordinates lie at distances dx_j from [mn_j, mx_j] can be inside
// the support only within sigma_d sqrt(1 - sum (dx_j / sigma_j)^2) of
// [mn_d, mx_d].  The bin arithmetic is FP32 (floor(floor(u) / t) =
// floor(u / t) for the tile t); every range is widened by 1e-3 sigma and by
// a rounding margin in bins, so that no sample inside a support is dropped.
template <int D>
struct DirectRows {
  int blo[3], bhi[3];
  float mn[3], mx[3], sg[3], isg[3], ibw[3], wb[3], mb[3];
  bool diag;

  __device__ __forceinline__ void box(const GeoDev& g, const BwDev& B) {
    diag = true;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int c = 0; c < D; ++c)
        if (a != c && B.Hinv[a * 3 + c] != 0.0) diag = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      blo[j] = 0;
      bhi[j] = 0;
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
      sg[j] = float(B.sigma[j]);
      isg[j] = float(1.0 / B.sigma[j]);
      ibw[j] = float(g.inv_h[j] / double(g.tile[j]));
      wb[j] = float(double(g.tile[j]) / g.inv_h[j]);
      mb[j] = 1e-3f + 2e-7f * float(g.nbins[j]);
      const float hw = sg[j] * 1.001f;
      const int nb = int(g.nbins[j]);
      int b0 = int(floorf((mn[j] - hw) * ibw[j] - mb[j]));
      int b1 = int(floorf((mx[j] + hw) * ibw[j] + mb[j]));
      blo[j] = b0 < 0 ? 0 : (b0 > nb - 1 ? nb - 1 : b0);
      bhi[j] = b1 < 0 ? 0 : (b1 > nb - 1 ? nb - 1 : b1);
    }
  }
  __device__ __forceinline__ int rows0() const { return D > 1 ? bhi[0] - blo[0] + 1 : 1; }
  __device__ __forceinline__ int rows1() const { return D > 2 ? bhi[1] - blo[1] + 1 : 1; }

  // bins [first, last] of row (r0, r1); false when the row is empty
  __device__ __forceinline__ bool row(const GeoDev& g, int r0, int r1, int64_t& first,
                                      int64_t& last) const {
    int lo = blo[D - 1], hi = bhi[D - 1];
    if (D > 1 && diag) {
      const int b[2] = {blo[0] + r0, blo[1] + r1};
      float rem = 1.f;
#pragma unroll
      for (int j = 0; j < D - 1; ++j) {
        const float a = float(b[j]) * wb[j], e = a + wb[j];
        float dx = fmaxf(a - mx[j], mn[j] - e) - 1e-3f * sg[j];
        dx = dx > 0.f ? dx : 0.f;
        const float t = dx * isg[j];
        rem -= t * t;
      }
      if (rem < 0.f) return false;
      const float hw = sg[D - 1] * (sqrtf(rem) + 1e-3f);
      const int c0 = int(floorf((mn[D - 1] - hw) * ibw[D - 1] - mb[D - 1]));
      const int c1 = int(floorf((mx[D - 1] + hw) * ibw[D - 1] + mb[D - 1]));
      lo = c0 > lo ? c0 : lo;
      hi = c1 < hi ? c1 : hi;
      if (lo > hi) return false;
    }
    if (D == 1) {
      first = lo;
      last = hi;
    } else if (D == 2) {
      first = int64_t(blo[0] + r0) * g.nbins[1] + lo;
      last = first + (hi - lo);
    } else {
      first = (int64_t(blo[0] + r0) * g.nbins[1] + blo[1] + r1) * g.nbins[2] + lo;
      last = first + (hi - lo);
    }
    return true;
  }
};

template <typename T>
__device__ __forceinline__ T sel3(int ax, T a, T b, T c) {
  return ax == 0 ? a : (ax == 1 ? b : c);
}

__device__ __forceinline__ int64_t wrap_idx(int64_t m, int64_t nf) {
  return m < 0 ? m + nf : (m >= nf ? m - nf : m);
}

template <typename T>
__device__ __forceinline__ T warp_sum_t(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int mono_index(const MonoTab& m, int nm, int e0, int e1, int e2) {
  for (int k = 0; k < nm; ++k)
    if (m.e[k][0] == e0 && m.e[k][1] == e1 && m.e[k][2] == e2) return k;
  return 0;
}

// The normal matrix of a D-variate system of order ORD at compile time: s[i][j]
// is the s-field of the product of the t-monomials i and j (the graded order
// of make_mono_chain), ax[i] the axes of t-monomial i (-1 past its degree).
template <int D, int ORD>
struct LprTab {
  int s[mono_count(D, ORD)][mono_count(D, ORD)];
  int ax[mono_count(D, ORD)][2];
};
template <int D, int ORD>
__host__ __device__ constexpr LprTab<D, ORD> make_lpr_tab() {
  constexpr int P = mono_count(D, ORD);
  const MonoChain c = make_mono_chain(D, 2 * ORD);
  int e[kMaxMono][3] = {};
  for (int f = 1; f < c.n; ++f) {
    for (int j = 0; j < 3; ++j) e[f][j] = e[c.parent[f]][j];
    e[f][c.axis[f]] += 1;
  }
  LprTab<D, ORD> t{};
  for (int i = 0; i < P; ++i) {
    int n = 0;
    t.ax[i][0] = t.ax[i][1] = -1;
    for (int j = 0; j < 3; ++j)
      for (int r = 0; r < e[i][j]; ++r) t.ax[i][n++] = j;
    for (int j = 0; j < P; ++j)
      for (int f = 0; f < c.n; ++f)
        if (e[f][0] == e[i][0] + e[j][0] && e[f][1] == e[i][1] + e[j][1] &&
            e[f][2] == e[i][2] + e[j][2])
          t.s[i][j] = f;
  }
  return t;
}

// S a = e_1 (P x P, FP64) by elimination with partial pivoting, every index
// known at compile time (the columns are unrolled by recursion) so that S stays
// in registers: the largest entry of a column is brought up by conditional
// swaps (integer selects, next to nothing on the 2-lane FP64 pipe of an SM)
// and each pivot costs one division.  With S in local memory and runtime
// indices the 6 x 6 systems of 300,007 samples took most of a 0.77 ms kernel.
// solve_e1 returns false if S is singular.
template <int P, int C>
__device__ __forceinline__ bool eliminate(double (&S)[P][P], double (&r)[P], double* a) {
  if constexpr (C == P) {
    return true;
  } else {
#pragma unroll
    for (int i = C + 1; i < P; ++i) {
      const bool up = fabs(S[i][C]) > fabs(S[C][C]);
#pragma unroll
      for (int j = C; j < P; ++j) {
        const double t = S[C][j];
        S[C][j] = up ? S[i][j] : t;
        S[i][j] = up ? t : S[i][j];
      }
      const double t = r[C];
      r[C] = up ? r[i] : t;
      r[i] = up ? t : r[i];
    }
    const bool ok = fabs(S[C][C]) > 0.0;
    const double inv = 1.0 / S[C][C];
#pragma unroll
    for (int i = C + 1; i < P; ++i) {
      const double f = S[i][C] * inv;
#pragma unroll
      for (int j = C + 1; j < P; ++j) S[i][j] -= f * S[C][j];
      r[i] -= f * r[C];
    }
    const bool rest = eliminate<P, C + 1>(S, r, a);
    double v = r[C];
#pragma unroll
    for (int j = C + 1; j < P; ++j) v -= S[C][j] * a[j];
    a[C] = v * inv;
    return ok && rest;
  }
}
template <int P>
__device__ __forceinline__ bool solve_e1(double (&S)[P][P], double* a) {
  double r[P];
#pragma unroll
  for (int i = 0; i < P; ++i) r[i] = (i == 0) ? 1.0 : 0.0;
  return eliminate<P, 0>(S, r, a) && isfinite(a[0]);
}

// sigma^g for the t-field monomial a
__device__ __forceinline__ double tscale(const MonoTab& mono, int a, const double* sigma) {
  double sc = 1.0;
  for (int j = 0; j < 3; ++j)
    for (int r = 0; r < mono.e[a][j]; ++r) sc *= sigma[j];
  return sc;
}

// its[i] = 1 / sigma^g of t-monomial i from isg = 1 / sigma.
template <int D, int ORD>
__device__ __forceinline__ void lpr_iscale(const double* isg, double* its) {
  constexpr auto tab = make_lpr_tab<D, ORD>();
#pragma unroll
  for (int i = 0; i < mono_count(D, ORD); ++i) {
    double sc = 1.0;
#pragma unroll
    for (int w = 0; w < 2; ++w)
      if (tab.ax[i][w] >= 0) sc *= isg[tab.ax[i][w]];
    its[i] = sc;
  }
}

// a = S~^-1 e_1 of the scaled normal matrix S~_ab = s_(a+b) / sigma^(a+b)
// (the intercept is unchanged by the scaling), isg = 1 / sigma: closed forms
// for Nadaraya-Watson and local linear in 1-D and 2-D (one division),
// elimination for local linear in 3-D and local quadratic.
template <int D, int ORD>
__device__ __forceinline__ bool lpr_weights(const double* s, const double* isg, double* a) {
  if constexpr (ORD == 0) {
    a[0] = 1.0 / s[0];
    return s[0] > 0.0;
  } else if constexpr (D == 1 && ORD == 1) {
    const double s01 = s[1] * isg[0], s11 = s[2] * (isg[0] * isg[0]);
    const double det = s[0] * s11 - s01 * s01;
    if (!(det > 0.0)) return false;
    const double inv = 1.0 / det;
    a[0] = s11 * inv;
    a[1] = -s01 * inv;
    return isfinite(a[0]);
  } else if constexpr (D == 2 && ORD == 1) {
    const double h0 = isg[0], h1 = isg[1];
    const double s00 = s[0], s01 = s[1] * h0, s02 = s[2] * h1;
    const double s11 = s[3] * (h0 * h0), s12 = s[4] * (h0 * h1), s22 = s[5] * (h1 * h1);
    const double c0 = s11 * s22 - s12 * s12;
    const double c1 = s12 * s02 - s01 * s22;
    const double c2 = s01 * s12 - s11 * s02;
    const double det = s00 * c0 + s01 * c1 + s02 * c2;
    if (!(det > 0.0)) return false;
    const double inv = 1.0 / det;
    a[0] = c0 * inv;
    a[1] = c1 * inv;
    a[2] = c2 * inv;
    return isfinite(a[0]);
  } else {
    constexpr int P = mono_count(D, ORD);
    constexpr auto tab = make_lpr_tab<D, ORD>();
    double S[P][P], its[P];
    lpr_iscale<D, ORD>(isg, its);
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
      for (int j = i; j < P; ++j) S[i][j] = S[j][i] = s[tab.s[i][j]] * (its[i] * its[j]);
    return solve_e1<P>(S, a);
  }
}

// The same for an order known at run time (3-D plans have orders 0 and 1).
// Eliminations are a call: inlined, their registers spilled the gathers of the
// 512-thread kernels that hold this (3-D local linear 3.8 -> 6.2 ms).
template <int D, int ORD>
__device__ __noinline__ bool lpr_weights_call(const double* s, const double* isg, double* a) {
  return lpr_weights<D, ORD>(s, isg, a);
}
template <int D>
__device__ __forceinline__ bool lpr_weights_order(int order, const double* s, const double* isg,
                                                  double* a) {
  if (order == 0) return lpr_weights<D, 0>(s, isg, a);
  if constexpr (D < 3) {
    if (order == 2) return lpr_weights_call<D, 2>(s, isg, a);
    return lpr_weights<D, 1>(s, isg, a);
  } else {
    return lpr_weights_call<D, 1>(s, isg, a);
  }
}

// ---- compensated FP32 arithmetic for the at-sample solves ------------------
// two_sum: s + e == a + b exactly (Knuth's branch-free sum).
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// a b - c d by Kahan's algorithm: the rounding error of c d is recovered
// exactly with an FMA, so the result is within two units of rounding of the
// exact value even under cancellation (Jeannerod, Louvet, Muller 2013).
__device__ __forceinline__ float dop(float a, float b, float c, float d) {
  const float w = __fmul_rn(c, d);
  const float e = fmaf(-c, d, w);
  const float f = fmaf(a, b, -w);
  return __fadd_rn(f, e);
}

// a = S~^-1 e_1 for p <= 3 from FP32 s-fields, S~_jk = D_j D_k s_(j+k) with
// D = (1, dsc[1], dsc[2]) the scaling the t-fields get.  Cofactors come from
// dop and the determinant from a compensated dot product (Ogita, Rump, Oishi
// 2005), so the solve adds rounding errors of a few units of FP32 whatever
// the cancellation in the cofactor expansion; the FP32 field values carry
// the NUFFT tolerance, which dominates.
__device__ __forceinline__ bool lpr_weights_f32(int p, const float* s, const float* dsc,
                                                float a[kMaxP]) {
  if (p == 1) {
    a[0] = 1.0f / s[0];
    return s[0] > 0.f;
  }
  if (p == 2) {  // 1-D local linear
    const float h0 = dsc[1];
    const float s01 = s[1] * h0, s11 = s[2] * (h0 * h0);
    const float det = dop(s[0], s11, s01, s01);
    if (!(det > 0.f)) return false;
    const float inv = 1.0f / det;
    a[0] = s11 * inv;
    a[1] = -s01 * inv;
    return isfinite(a[0]);
  }
  // 2-D local linear, s-fields 1, z1, z2, z1z1, z1z2, z2z2
  const float h0 = dsc[1], h1 = dsc[2];
  const float s00 = s[0], s01 = s[1] * h0, s02 = s[2] * h1;
  const float s11 = s[3] * (h0 * h0), s12 = s[4] * (h0 * h1), s22 = s[5] * (h1 * h1);
  const float c0 = dop(s11, s22, s12, s12);
  const float c1 = dop(s12, s02, s01, s22);
  const float c2 = dop(s01, s12, s11, s02);
  const float p0 = __fmul_rn(s00, c0), r0 = fmaf(s00, c0, -p0);
  const float m1 = __fmul_rn(s01, c1), r1 = fmaf(s01, c1, -m1);
  const float m2 = __fmul_rn(s02, c2), r2 = fmaf(s02, c2, -m2);
  float q1, q2;
  const float p1 = two_sum(p0, m1, q1);
  const float p2 = two_sum(p1, m2, q2);
  const float det = __fadd_rn(p2, __fadd_rn(__fadd_rn(r0, r1), __fadd_rn(__fadd_rn(q1, r2), q2)));
  if (!(det > 0.f)) return false;
  const float inv = 1.0f / det;
  a[0] = c0 * inv;
  a[1] = c1 * inv;
  a[2] = c2 * inv;
  return isfinite(a[0]);
}

}  // namespace fk
