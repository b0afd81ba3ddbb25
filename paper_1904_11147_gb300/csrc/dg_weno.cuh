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

#include <cmath>
#include <cstring>

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

// ----------------------------------------------------------------------------- fixed point
// Sums of modes times constants in 64-bit fixed point.  In the time of one FP64 instruction (67
// clocks per warp and SM sub-partition) the integer pipes do several 64-bit products, and
// they are idle otherwise.  The modes of a variable are aligned to the largest one; products are
// rounded to nearest and the modes taken without a product are truncated on the magnitude, so
// the sums are odd in the modes (a mirror image gives the mirrored result) and without bias.
// Error of a trace before its final rounding, against 128-bit values over random modes, relative
// to the largest mode: rms 7e-19 (P1), 2.4e-18 (P2), 6.5e-18 (P3), at most 2.7e-18, 1.4e-17, 4.3e-17;
// FP64 sums of the same terms are off by 6e-17, 9e-17 and 1.0e-16 (rms).

// t 2^q as a double, rounded to nearest, ties away or (EVEN) to even; out of range: 0 or infinity.  The
// traces, one in 32 of which is a tie for P3, take ties to even: away would lengthen them by 3e-18.
template <bool EVEN = false>
__device__ __forceinline__ double pack_s64(long long t, int q) {
  const unsigned long long a = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int z = __clzll((long long)a), e = 1086 - z + q;
  const unsigned long long m = a << (z & 63);
  const unsigned lo = (unsigned)m, up = EVEN ? (lo & 0x7ffu) + ((lo >> 11) & 1u) > 0x400u : (lo >> 10) & 1u;
  unsigned long long bits = ((unsigned long long)(unsigned)(e - 1) << 52) + (m >> 11) + up;
  if (e < 1 || a == 0) bits = 0ull;
  if (e > 2046 && a != 0) bits = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(bits | ((unsigned long long)t & 0x8000000000000000ull)));
}

// X[m] 2^(E - 1075 - F) = u[m], |X| < 2^(53 + F); values 2^-(53 + F) below the largest are dropped.  The
// low LOW bits of the modes of degree 0 in the first direction are cleared: those enter the
// sums shifted by LOW.  E >= 2047: a mode is not finite.
template <int M, int F, int LOW>
__device__ __forceinline__ int align_modes(const double (&u)[M], long long (&X)[M]) {
  unsigned top = 1u << 20;
#pragma unroll
  for (int m = 0; m < M; ++m) top = max(top, (unsigned)__double2hiint(u[m]) & 0x7fffffffu);
  const int E = (int)(top >> 20);
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const unsigned hi = (unsigned)__double2hiint(u[m]), lo = (unsigned)__double2loint(u[m]), ex = (hi >> 20) & 0x7ffu;
    const unsigned sig = (hi & 0xfffffu) | (min(ex, 1u) << 20);  // (no leading 1 below the normal range)
    const unsigned long long w = ((unsigned long long)__funnelshift_l(lo, sig, F) << 32) | (lo << F);
    const unsigned long long keep = mode_a(m) == 0 ? ~((1ull << LOW) - 1) : ~0ull;
    const long long x = (long long)((w >> min(E - (int)max(ex, 1u), 63)) & keep), s = (long long)((int)hi >> 31);
    X[m] = (x ^ s) - s;
  }
  return E;
}

// c x / 2^64 rounded to nearest
__device__ __forceinline__ long long mul_rn(long long c, long long x) {
  return __mul64hi(c, x) + (long long)(((unsigned long long)c * (unsigned long long)x) >> 63);
}

// sum_t e_t KQ_qt at the Q Gauss points (KQ_q0 = 1); kq: KQ 2^62, rows of the points <= 0; |e_t| < 2^61
// for t > 0.
template <int N>
__device__ __forceinline__ void eval_fix(const long long (&e)[N + 1], const long long* __restrict__ kq,
                                         long long (&out)[N + 1]) {
  constexpr int Q = N + 1;
#pragma unroll
  for (int q = 0; q < Q / 2; ++q) {
    const long long* c = kq + q * (N + 1);
    long long ev = e[0], od = mul_rn(c[1], e[1] << 2);
    if constexpr (N >= 2) ev += mul_rn(c[2], e[2] << 2);
    if constexpr (N == 3) od += mul_rn(c[3], e[3] << 2);
    out[q] = ev + od;
    out[Q - 1 - q] = ev - od;
  }
  if constexpr (N == 2) out[1] = e[0] + mul_rn(kq[(N + 1) + 2], e[2] << 2);
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
  static constexpr int BR = BF + 12;            // brel as U64f (integers): significand, exponent
  static constexpr int WH = BR + 2;             // [NG][N1] wh 2^63 (integers)
  static constexpr int WC = WH + NG * N1;       // [NG][N1][N] wc 2^62 (signed integers)
  static constexpr int QS = WC + NG * N1 * N;   // [2] qsp 2^59 (integers; qsp is 12.2 and 9.3)
  static constexpr int QD = QS + 2;             // [2] qsp in FP64
  static constexpr int PG = QD + 2;             // [NG][N1] w_g psi_n(r_g)
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
  auto put = [&](int k, unsigned long long v) { std::memcpy(h + k, &v, sizeof(v)); };
  int be;
  const double bf = std::frexp(t.brel, &be);  // in [1/2, 1): significand 2^64 bf, brel = m 2^(be - 64)
  put(L::BR, (unsigned long long)std::ldexp(bf, 64));
  put(L::BR + 1, (unsigned long long)(long long)be);
  for (int r = 0; r < 2; ++r) h[L::QD + r] = t.qsp[r];
  for (int r = 0; r < 2; ++r) put(L::QS + r, (unsigned long long)(long long)std::llrint(std::ldexp(t.qsp[r], 59)));
  h[L::PG0] = 0.0;
  for (int g = 0; g < L::NG; ++g) {
    for (int i = 0; i <= N; ++i) {
      put(L::WH + g * L::N1 + i, (unsigned long long)std::ldexp(t.wh[g][i], 63));
      for (int j = 0; j < N; ++j)
        put(L::WC + (g * L::N1 + i) * N + j, (unsigned long long)(long long)std::llrint(std::ldexp(t.wc[g][i][j], 62)));
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

// ----------------------------------------------------------------------------- reconstruction
// Integer arithmetic of the reconstruction.  In the time of one FP64 instruction (67 clocks
// per warp and SM sub-partition) the integer pipes do a 64-bit product and more, so everything
// behind the smoothness indicators runs there, on positive floating-point numbers m 2^e with a
// 64-bit significand (products and weights: 11 bits more than a double) and on fixed-point sums.
struct U64f {
  unsigned long long m;  // in [2^63, 2^64), or 0
  int e;
};
__device__ __forceinline__ U64f unpack_pos(double x) {  // of a positive normal number; e is biased
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  return U64f{((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11), (int)(hi >> 20)};
}
// a b / 2^64; relative error below 2^-62
__device__ __forceinline__ U64f mul_n(U64f a, U64f b) {
  const unsigned long long m = __umul64hi(a.m, b.m);
  const int up = (long long)m >= 0;  // in [2^62, 2^63)
  return U64f{m << up, a.e + b.e - up};
}
// t / s 2^q as a double; the quotient before its rounding is within 2^-60 (relative).  1/s from
// FP32's reciprocal Y (23 bits) and one third-order step, Y (1 + e + e^2) with e = 1 - s Y.
__device__ __forceinline__ double quot_s64(long long t, unsigned long long s, int q) {
  unsigned long long a = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int zt = __clzll((long long)a), zs = __clzll((long long)s);
  a <<= zt & 63;
  s <<= zs & 63;
  const unsigned hi = (unsigned)(s >> 32), lo = (unsigned)s;
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(0x3f800000u | ((hi >> 8) & 0x7fffffu))));
  const unsigned yb = __float_as_uint(y), Y = yb >= 0x3f800000u ? 0xffffffffu : (yb << 8) | 0x80000000u;  // 2^95 / s
  // e 2^63, rounded down: the reciprocal does not pass 2^64
  const long long e = (long long)(0x7fffffffffffffffull - ((unsigned long long)hi * Y + __umulhi(lo, Y)));
  const int eh = (int)(e >> 11);
  const long long g = e + (((long long)eh * eh) >> 41);
  const long long d = (((long long)(int)(g >> 12) * (long long)Y) >> 19) + (long long)__umulhi(((unsigned)g & 0xfffu) << 1, Y);
  const unsigned long long h = __umul64hi(a, ((unsigned long long)Y << 32) + (unsigned long long)d);  // >= 2^62
  const int up = (long long)h >= 0, b = 1023 + q - zt + zs - up;
  const unsigned long long m = h << up;
  unsigned long long bits = ((unsigned long long)(unsigned)(b - 1) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  if (b < 1 || t == 0) bits = 0ull;
  if (b > 2046 && t != 0) bits = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(bits | ((unsigned long long)t & 0x8000000000000000ull)));
}

// Steps 2-5: u_g - avg[N] at the Step 1 points from the 2N differences d (see Tabs::bform,
// wc, wh).
//
//   b_i   (eps + beta_i) / M_i, a sum of squares, in FP64
//   P_i   the weights' 1 / (eps + beta_i)^2 up to a common factor: the product of the other
//         stencils' squares, as U64f (any magnitude of the data)
//   X_ij  P_i d_{i+j}, sign apart
//   T_g, S_g   sum wc X and sum wh P in 64-bit fixed point: all X are shifted to the largest
//         one's exponent (below 2^62), all P to theirs.  With sum |wc| <= 4.7 (below 8) and sum wh <=
//         3.7 (below 4) per point both stay below 2^63 (dgt::sums_fit).  A term loses at most 2^-62
//         of the largest one, and every product at most one unit of the sum, half of it on
//         average (added back at the start).
//   u_g - avg[N] = T_g / S_g, in integers rounded once, or in FP64
// Out of FP64's normal range: subnormal differences enter with their leading zeros; a quotient in
// integers below 2^-1022 is 0 (see kSmall in dg_limit2.cu).
// FP64 instructions per call: 2 / 12 / 32 for N = 1, 2, 3 (10 / 27 / 64 with the quotient in
// FP64, 20 / 71 / 142 with all of it), next to some 250 / 800 / 1,700 integer ones.  From all of it
// in FP64 to FP64 quotients: limiter of 130k P2 cells 974 -> 730 us, of 140k P3 cells 2,200 ->
// 1,950 us.  Integer quotients besides: 1024^2 P2 step 12.3 -> 11.1 ms, P3 batch of 8 x 128 x
// 512 cells 31.8 -> 30.0 ms.
//
// INTQ: the quotient in integers (2D).  1D keeps it in FP64: its steps gain little (64 x 800 P3
// cells 180 -> 171 us, 160 Burgers cells nothing), and long P3 shock-tube runs without
// the positivity scaling depend on the last bit (of six FP64 runs of one of them, perturbed by
// 1e-16 to 5e-16 each step, one lost positivity).
//
// SPLIT: the CSWENO P3 rule with one negative weight at each inner point.  With T and S the
// sums over the positive (+) and the negative (-) weights, the difference of the two
// normalised parts of the split is
//   [T+ (den1 + q0 S-) - T- (q1 S+ - den2)] / (den1 den2), den1 = 2 S+ + S-, den2 = S+ + 2 S-.
template <int N, bool SPLIT, bool INTQ = true>
__device__ __forceinline__ void weno_diff(const double (&d)[2 * N], const double* __restrict__ tab, const Reg64& K,
                                          double (&out)[N == 1 ? 2 : 4]) {
  using L = LimTab<N>;
  constexpr int N1 = N + 1, NG = L::NG;
  const unsigned long long* itab = reinterpret_cast<const unsigned long long*>(tab);
  bool bad = false;  // a difference that is not finite
  U64f D[N1];
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
    bad = bad || ((unsigned)__double2hiint(b) & 0x7fffffffu) > 0x7ff00000u;
    D[i] = unpack_pos(b);
    // the outer stencils' M over the inner ones'
    if (N > 1 && (i == 0 || i == N)) D[i] = mul_n(D[i], U64f{itab[L::BR], (int)itab[L::BR + 1]});
    D[i] = mul_n(D[i], D[i]);
  }
  U64f P[N1];
  if constexpr (N == 1) {
    P[0] = D[1];
    P[1] = D[0];
  } else if constexpr (N == 2) {
    P[0] = mul_n(D[1], D[2]);
    P[1] = mul_n(D[0], D[2]);
    P[2] = mul_n(D[0], D[1]);
  } else {
    const U64f a = mul_n(D[0], D[1]), b = mul_n(D[2], D[3]);
    P[0] = mul_n(D[1], b);
    P[1] = mul_n(D[0], b);
    P[2] = mul_n(D[3], a);
    P[3] = mul_n(D[2], a);
  }
  U64f dm[2 * N];
  unsigned neg = 0;  // bit k: d_k < 0
#pragma unroll
  for (int k = 0; k < 2 * N; ++k) {
    const unsigned hi = (unsigned)__double2hiint(d[k]), ab = hi & 0x7fffffffu;
    bad = bad || ab >= 0x7ff00000u;
    neg |= (hi >> 31) << k;
    const unsigned lo = (unsigned)__double2loint(d[k]), one = ab >= 0x00100000u ? 0x80000000u : 0u;
    dm[k] = U64f{((unsigned long long)(__funnelshift_l(lo, ab, 11) | one) << 32) | (lo << 11), (int)max(ab >> 20, 1u)};
  }
  U64f X[N1][N];
  int ex = -(1 << 20), ep = P[0].e;
#pragma unroll
  for (int i = 0; i < N1; ++i) {
    ep = max(ep, P[i].e);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      X[i][j] = mul_n(P[i], dm[i + j]);
      if (dm[i + j].m != 0ull) ex = max(ex, X[i][j].e);
    }
  }
  long long Xf[N1][N];
  unsigned long long Pf[N1];
#pragma unroll
  for (int i = 0; i < N1; ++i) {
    Pf[i] = P[i].m >> min(ep - P[i].e + 2, 63);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const long long x = (long long)(X[i][j].m >> min(max(ex - X[i][j].e + 2, 0), 63));
      Xf[i][j] = (neg >> (i + j)) & 1u ? -x : x;
    }
  }
  // T_g 2^64 = sum Xf (wc 2^62), S_g 2^64 = sum Pf (wh 2^63); X = Xf 2^(ex + 2 + 64 - 1086) and
  // P = Pf 2^(ep + 2) up to P's common factor: u_g - avg[N] = T_g / S_g 2^(ex - ep - 1021)
  const int q = min(max(ex - ep - 1021, -8000), 8000);
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int ng = SPLIT ? dgt::weno_neg(N, g, false) : -1, ref = dgt::weno_ref(N, g);
    const long long* wc = reinterpret_cast<const long long*>(itab) + L::WC + g * N1 * N;
    const unsigned long long* wh = itab + L::WH + g * N1;
    long long Tp = ng < 0 ? N1 * N / 2 : N * N / 2, Tm = N / 2;
    unsigned long long Sp = Pf[ref] >> 1, Sm = 0;
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      if (i == ng) Sm = __umul64hi(wh[i], Pf[i]);
      else if (i != ref) Sp += __umul64hi(wh[i], Pf[i]);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const long long t = __mul64hi(wc[i * N + j], Xf[i][j]);
        if (i == ng) Tm += t;
        else Tp += t;
      }
    }
    if constexpr (!INTQ) {
      double num, den;
      if (ng < 0) {
        num = pack_s64(Tp, q);
        den = pack_s64((long long)Sp, 0);
      } else {
        const double T = pack_s64(Tp, q), Tn = pack_s64(Tm, q), S = pack_s64((long long)Sp, 0), Sn = pack_s64((long long)Sm, 0);
        const double den1 = K.add(S, K.add(S, Sn)), den2 = K.add(Sn, K.add(S, Sn));
        num = fma(T, fma(tab[L::QD], Sn, den1), -K.mul(Tn, fma(tab[L::QD + 1], S, -den2)));
        den = K.mul(den1, den2);
      }
      double y;  // S_g lies in [2^50, 2^63): no range check (see rcp_d)
      asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(den));
      const double e = fma(-den, y, K.one);
      out[g] = K.mul(num, fma(y, fma(e, e, e), y));
    } else if (ng < 0) {
      out[g] = quot_s64(Tp, Sp, q);
    } else {
      // S+ and S- below 2^59 (the larger one from 2^58 on), T+ and T- below 2^63: a factor of T is
      // below (2 + 1 + 12.3) 2^59 < 2^63
      const long long* qs = reinterpret_cast<const long long*>(itab) + L::QS;
      const int c = __clzll((long long)(Sp | Sm));
      const long long A = (long long)((Sp << (c & 63)) >> 5), B = (long long)((Sm << (c & 63)) >> 5);
      const long long den1 = A + A + B, den2 = A + B + B;
      const long long ta = Tp ^ (Tp >> 63), tb = Tm ^ (Tm >> 63);
      const int z = (__clzll(ta | tb) - 1) & 63;
      const long long num = __mul64hi(Tp << z, den1 + 2 * __mul64hi(qs[0], B << 4)) +
                            __mul64hi(Tm << z, den2 - 2 * __mul64hi(qs[1], A << 4));
      out[g] = quot_s64(num, __umul64hi((unsigned long long)den1 << 3, (unsigned long long)den2 << 3), q + 1 + c - z);
    }
    if (bad) out[g] = __longlong_as_double(0x7ff8000000000000LL);
  }
}

}  // namespace dg
