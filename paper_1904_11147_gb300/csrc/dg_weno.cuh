// WENO reconstruction of the limiters on the differences of the stencil averages, and the
// arithmetic form that GB300's FP64 pipe runs fastest.
//
// The FP64 pipe issues a DFMA whose three operands are vector registers at 1.89 lanes per
// clock and SM, but a DADD, a DMUL, or a DFMA with a constant-bank, uniform or immediate
// operand at 1.60 (measured with one to eight independent chains on 4 to 32 warps per SM).
// So sums and products are written as fma(x, one, y) and fma(x, y, -0.0) with `one` and
// `-0.0` in registers the compiler cannot see through -- the same IEEE results, signed zeros
// included -- and tables are read from shared memory into registers.
#pragma once

#include "dg_common.cuh"
#include "tables.h"

namespace dg {

struct Reg64 {  // the opaque constants 1.0 and -0.0
  double one, nz;
  __device__ __forceinline__ double add(double x, double y) const { return fma(x, one, y); }
  __device__ __forceinline__ double sub(double x, double y) const { return fma(x, one, -y); }
  __device__ __forceinline__ double mul(double x, double y) const { return fma(x, y, nz); }
};

// rcp_d with its constant in a register
__device__ __forceinline__ double rcp_k(double x, const Reg64& K) {
  if (((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x00100000u >= 0x7fc00000u) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, K.one);
  return fma(y, fma(e, e, e), y);
}

// what the kernels need of gamma
struct Gamma {
  double gm1, hgm1, sg;  // gamma - 1, -(gamma - 1) / 2, sqrt(gamma)
};

// sqrt(x) for the wave speed: the hardware's ~20-bit 1/sqrt(x) = y, t = x y = sqrt(x) (1-e)^(1/2)
// with e = 1 - x y^2, and t (1 + e/2 + 3 e^2 / 8) (see sqrt_d; here without its final product).
__device__ __forceinline__ double sqrt_t(double x, const Reg64& K, double c38, double half) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  if (b - 0x0010000000000000ull >= 0x7fe0000000000000ull) return sqrt(x);  // not a positive normal
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = K.mul(x, y), e = fma(-t, y, K.one);
  return fma(t, K.mul(e, fma(c38, e, half)), t);
}

// larger of |a| and |b|, a NaN (a state without a real sound speed) if either is one: on the
// bit patterns, where non-negative doubles order as integers and a NaN is largest (word by
// word: a 64-bit mask would become an FP64 |x| instruction)
__device__ __forceinline__ double max_speed(double a, double b) {
  const unsigned ah = (unsigned)__double2hiint(a) & 0x7fffffffu, bh = (unsigned)__double2hiint(b) & 0x7fffffffu;
  const unsigned al = (unsigned)__double2loint(a), bl = (unsigned)__double2loint(b);
  const bool first = ah > bh || (ah == bh && al >= bl);
  return __hiloint2double((int)(first ? ah : bh), (int)(first ? al : bl));
}

// Doubled values at the Q Gauss points of sum_t e_t psi_t / psi_0 (KQ: sqrt(2) psi_t).
template <int N>
__device__ __forceinline__ void eval_gauss2(const double (&e)[N + 1], const double* __restrict__ kq, const Reg64& K,
                                            double (&out)[N + 1]) {
  constexpr int Q = N + 1;
#pragma unroll
  for (int q = 0; q < Q / 2; ++q) {
    const double* c = kq + q * (N + 1);
    double ev = e[0];
    if constexpr (N >= 2) ev = fma(c[2], e[2], ev);
    if constexpr (N == 3) {
      const double od = fma(c[3], e[3], K.mul(c[1], e[1]));
      out[q] = K.add(ev, od);
      out[Q - 1 - q] = K.sub(ev, od);
    } else {
      out[q] = fma(c[1], e[1], ev);
      out[Q - 1 - q] = fma(-c[1], e[1], ev);
    }
  }
  if constexpr (N == 2) out[1] = fma(kq[(N + 1) + 2], e[2], e[0]);
}

// Tables of one limiter (degree N, CSWENO or parent) as the kernels keep them in shared memory.
template <int N>
struct LimTab {
  static constexpr int N1 = N + 1, NG = N == 1 ? 2 : 4;
  static constexpr int ONE = 0, NZ = 1;
  static constexpr int BF = 2;                  // [2][6] bform
  static constexpr int WH = BF + 12;            // [NG][N1]
  static constexpr int WC = WH + NG * N1;       // [NG][N1][N]
  static constexpr int QS = WC + NG * N1 * N;   // [2] qsp
  static constexpr int PG = QS + 2;             // [NG][N1] w_g psi_n(r_g)
  static constexpr int PG0 = PG + NG * N1;      // sum_g w_g psi_0
  static constexpr int CA = PG0 + 1;            // x part of the subcell averages times psi_0: [4] SA[last][n] psi_0
  static constexpr int CR = CA + 4;             // y part over psi_0: [4] SA[last][n] / psi_0
  static constexpr int P0 = CR + 4;             // psi_0
  static constexpr int CS = P0 + 1;             // 1D subcell averages: [4] SA[last][n]
  static constexpr int SIZE = (CS + 4 + 1) / 2 * 2;
};

// the largest of them, one row per degree
constexpr int kLimTab = LimTab<3>::SIZE;
static_assert(LimTab<1>::SIZE <= kLimTab && LimTab<2>::SIZE <= kLimTab, "row length");

template <int N>
inline void pack_lim(const dgt::Tabs& t, double* h) {
  using L = LimTab<N>;
  h[L::ONE] = 1.0;
  h[L::NZ] = -0.0;
  for (int r = 0; r < 2; ++r)
    for (int k = 0; k < 6; ++k) h[L::BF + 6 * r + k] = t.bform[r][k];
  h[L::QS] = t.qsp[0];
  h[L::QS + 1] = t.qsp[1];
  h[L::PG0] = 0.0;
  for (int g = 0; g < L::NG; ++g) {
    for (int i = 0; i <= N; ++i) {
      h[L::WH + g * L::N1 + i] = t.wh[g][i];
      for (int j = 0; j < N; ++j) h[L::WC + (g * L::N1 + i) * N + j] = t.wc[g][i][j];
      h[L::PG + g * L::N1 + i] = t.rw[g] * t.psiG[g][i];
    }
    h[L::PG0] += t.rw[g] * t.psiG[g][0];
  }
  const double p0 = t.psi_0[0];
  for (int n = 0; n < 4; ++n) {
    const double v = n <= N ? t.SA[2 * N][n] : 0.0;
    h[L::CA + n] = v * p0;
    h[L::CR + n] = v / p0;
    h[L::CS + n] = v;
  }
  h[L::P0] = p0;
}

// Steps 2-5: u_g - avg[N] at the Step 1 points from the 2N differences d (see Tabs::bform,
// wc, wh).  Per call 20 / 71 / 142 FP64 instructions for N = 1, 2, 3.
//
// The weights need 1 / D_i^2-like ratios only up to a common factor, so instead of a
// reciprocal per stencil P_i is the product of the other stencils' D.  That overflows for
// extreme data, so where any D reaches 2^150 (or is not a number) the reciprocals are
// taken, scaled by the power of two that brings the largest into [1, 2).
// SPLIT: the CSWENO P3 rule with one negative weight at each inner point.  With T and S the
// sums of wc P d and wh P over the positive (+) and the negative (-) weights, the difference
// of the two normalised parts of the split is
//   [T+ (den1 + q0 S-) - T- (q1 S+ - den2)] / (den1 den2), den1 = 2 S+ + S-, den2 = S+ + 2 S-.
template <int N, bool SPLIT>
__device__ __forceinline__ void weno_diff(const double (&d)[2 * N], const double* __restrict__ tab, const Reg64& K,
                                          double (&out)[N == 1 ? 2 : 4]) {
  using L = LimTab<N>;
  constexpr int N1 = N + 1, NG = L::NG;
  double D[N1];
#pragma unroll
  for (int i = 0; i < N1; ++i) {
    const bool mir = 2 * i > N;
    const double* f = tab + L::BF + 6 * (mir ? N - i : i);
    double b;
    if constexpr (N == 1) {
      b = fma(d[i], d[i], f[0]);
    } else if constexpr (N == 2) {
      const double e0 = mir ? d[i + 1] : d[i], e1 = mir ? d[i] : d[i + 1];
      const double v = fma(f[3], e1, e0);
      b = fma(v, v, fma(f[1], K.mul(e1, e1), f[0]));
    } else {
      const double e0 = mir ? d[i + 2] : d[i], e1 = d[i + 1], e2 = mir ? d[i] : d[i + 2];
      const double v = fma(f[3], e1, fma(f[4], e2, e0)), w = fma(f[5], e2, e1);
      b = fma(v, v, fma(K.mul(f[2], w), w, fma(f[1], K.mul(e2, e2), f[0])));
    }
    D[i] = K.mul(b, b);
  }
  int hi = __double2hiint(D[0]);
#pragma unroll
  for (int i = 1; i < N1; ++i) hi = max(hi, __double2hiint(D[i]));
  double P[N1];
  if (hi < (1023 + 150) << 20) {  // D >= eps^2 / M^2 > 0, so the bit patterns order as integers
    if constexpr (N == 1) {
      P[0] = D[1];
      P[1] = D[0];
    } else if constexpr (N == 2) {
      P[0] = K.mul(D[1], D[2]);
      P[1] = K.mul(D[0], D[2]);
      P[2] = K.mul(D[0], D[1]);
    } else {
      const double a = K.mul(D[0], D[1]), b = K.mul(D[2], D[3]);
      P[0] = K.mul(D[1], b);
      P[1] = K.mul(D[0], b);
      P[2] = K.mul(D[3], a);
      P[3] = K.mul(D[2], a);
    }
  } else {
    int top = 0;
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      P[i] = 1.0 / D[i];
      top = max(top, __double2hiint(P[i]) & 0x7fffffff);
    }
    top = (top >> 20) < 2047 ? (top >> 20) : 1023;
    const double s = __hiloint2double((2046 - top) << 20, 0);  // 2^(1023 - top)
#pragma unroll
    for (int i = 0; i < N1; ++i) P[i] *= s;
  }
  double X[N1][N];
#pragma unroll
  for (int i = 0; i < N1; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) X[i][j] = K.mul(P[i], d[i + j]);
  double num[NG], den[NG];
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    constexpr int kNone = -1;
    const int neg = SPLIT ? dgt::weno_neg(N, g, false) : kNone;
    const int ref = dgt::weno_ref(N, g);
    const double* wc = tab + L::WC + g * N1 * N;
    const double* wh = tab + L::WH + g * N1;
    double T = 0.0, S = P[ref];
    bool first = true;
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      if (i == neg) continue;
      if (i != ref) S = fma(wh[i], P[i], S);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        T = first ? K.mul(wc[i * N + j], X[i][j]) : fma(wc[i * N + j], X[i][j], T);
        first = false;
      }
    }
    if (neg < 0) {
      num[g] = T;
      den[g] = S;
    } else {
      const double Sm = K.mul(wh[neg], P[neg]);
      double Tm = K.mul(wc[neg * N], X[neg][0]);
#pragma unroll
      for (int j = 1; j < N; ++j) Tm = fma(wc[neg * N + j], X[neg][j], Tm);
      const double den1 = K.add(S, K.add(S, Sm)), den2 = K.add(Sm, K.add(S, Sm));
      num[g] = fma(T, fma(tab[L::QS], Sm, den1), -K.mul(Tm, fma(tab[L::QS + 1], S, -den2)));
      den[g] = K.mul(den1, den2);
    }
  }
  // one range check for all points (see rcp_d)
  bool ok = true;
#pragma unroll
  for (int g = 0; g < NG; ++g)
    ok = ok && ((unsigned)__double2hiint(den[g]) & 0x7fffffffu) - 0x00100000u < 0x7fc00000u;
  if (ok) {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      double y;
      asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(den[g]));
      const double e = fma(-den[g], y, K.one);
      out[g] = K.mul(num[g], fma(y, fma(e, e, e), y));
    }
  } else {
#pragma unroll
    for (int g = 0; g < NG; ++g) out[g] = num[g] / den[g];
  }
}

}  // namespace dg
