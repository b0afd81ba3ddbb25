// 1D stage, indicator and limiter (P^N, N = 1..3; Burgers V = 1, Euler V = 3).
//
//   k_step1     one whole SSP-RK3 step with the TVB indicator and CSWENO in one kernel
//   k_stage1    one stage;  k_flag1: TVB flags;  k_limit1: CSWENO on the troubled cells
//
// 1D meshes are small (hundreds to thousands of cells per instance), so as separate kernels
// a step is bound by its 15 launches and by single warps that wait for memory.  k_step1 keeps
// a tile of cells in shared memory through all three stages; a tile reads kHalo cells more
// on each side (a stage reaches one cell, its limiter one more) and advances them
// redundantly, so blocks need not exchange anything.  The kernels share every formula, so a
// step equals the stage calls bit for bit.
//
// Arithmetic in the three-register form of dg_weno.cuh; the volume's point values are formed
// over psi_0 (sqrt(2) u) as in the split 2D stage.
#include <cmath>

#include "dg_shared.cuh"
#include "dg_weno.cuh"

namespace dg {
namespace s1 {

template <int N>
struct STab {
  static constexpr int N1 = N + 1, Q = N + 1, NX = (Q + 1) / 2;
  static constexpr int ONE = 0, NZ = 1, C38 = 2, HALF = 3;
  static constexpr int GM1 = 4, SG = 5;            // gamma - 1, sqrt(gamma) (set by the block)
  static constexpr int RA = 6, RB = 9;             // [3] weights of u^n and of the stage's input
  static constexpr int P0 = 12;                    // psi_0
  static constexpr int PP1 = 13;                   // [N1] psi_n(1)
  static constexpr int KQ = PP1 + N1;              // [NX][N1] sqrt(2) psi_n(x_q), x_q <= 0
  // times (2/h) dt
  static constexpr int XF = KQ + NX * N1;
  static constexpr int CX = XF;                    // [NX][N1] w psi_n'(x_p) over the homogeneity factor
  static constexpr int LX = CX + NX * N1;          // [N1] -psi_n(1) / 2
  static constexpr int DX = LX + N1;               // [4] density: integrals psi_1' psi_0, psi_2' psi_1, psi_3' psi_2, psi_3' psi_0
  static constexpr int SIZE = (DX + 4 + 1) / 2 * 2;
};
constexpr int kSTab = STab<3>::SIZE;

__device__ double g_stab[2][3][kSTab];  // [pde][N - 1]
__device__ double g_lim[3][kLimTab];

template <int N>
void pack(const dgt::Tabs& t, int pde, double* h) {
  using S = STab<N>;
  constexpr int N1 = S::N1, Q = S::Q, NX = S::NX;
  h[S::ONE] = 1.0;
  h[S::NZ] = -0.0;
  h[S::C38] = 0.375;
  h[S::HALF] = 0.5;
  const double ra[3] = {0.0, 0.75, 1.0 / 3.0}, rb[3] = {1.0, 0.25, 2.0 / 3.0};
  for (int k = 0; k < 3; ++k) {
    h[S::RA + k] = ra[k];
    h[S::RB + k] = rb[k];
  }
  h[S::P0] = t.psi_0[0];
  // f(sqrt(2) u) = sqrt(2) f(u) (Euler), 2 f(u) (Burgers)
  const double hom = pde == 1 ? std::sqrt(0.5) : 0.5;
  for (int n = 0; n < N1; ++n) {
    h[S::PP1 + n] = t.psi_p1[n];
    for (int q = 0; q < NX; ++q) {
      h[S::KQ + q * N1 + n] = t.kq[q][n];
      h[S::CX + q * N1 + n] = hom * t.gw[q] * t.dpsi_q[q][n];
    }
    h[S::LX + n] = -0.5 * t.psi_p1[n];
  }
  auto dpk = [&](int a, int k) {  // integral of psi_a' psi_k (exact with the Gauss rule)
    double s = 0.0;
    for (int q = 0; q < Q; ++q) s += t.gw[q] * t.dpsi_q[q][a] * t.psi_q[q][k];
    return s;
  };
  h[S::DX] = dpk(1, 0);
  if (N >= 2) h[S::DX + 1] = dpk(2, N >= 2 ? 1 : 0);
  if (N >= 3) {
    h[S::DX + 2] = dpk(N >= 3 ? 3 : 0, N >= 3 ? 2 : 0);
    h[S::DX + 3] = dpk(N >= 3 ? 3 : 0, 0);
  }
}

// Fills a block's stage table: tab[k] for the constants, tab[XF ...] times (2/h) dt (which the
// caller multiplies by the stage's weight, RB, when it uses them).
template <int PDE, int N>
__device__ __forceinline__ void fill_tab(double* tab, const Inst& I, double dt, const Gamma& gm) {
  using T = STab<N>;
  for (int k = threadIdx.x; k < T::SIZE; k += blockDim.x) {
    double x = g_stab[PDE][N - 1][k];
    if (k == T::GM1) x = gm.gm1;
    if (k == T::SG) x = gm.sg;
    if (k >= T::XF) x *= I.sx * dt;
    tab[k] = x;
  }
}

// ----------------------------------------------------------------------------- stage
// Traces at r = +1 and r = -1, plain sums from the mean on: near vacuum the trace is the
// difference of far larger terms, and its rounding the stage's error.
template <int N>
__device__ __forceinline__ void traces(const double (&u)[N + 1], const double* __restrict__ tab, const Reg64& K,
                                       double& tE, double& tW) {
  const double* c = tab + STab<N>::PP1;
  tE = tW = K.mul(u[0], c[0]);
#pragma unroll
  for (int n = 1; n < N + 1; ++n) {  // psi_n(-1) = (-1)^n psi_n(1)
    tE = fma(u[n], c[n], tE);
    tW = fma(u[n], (n & 1) ? -c[n] : c[n], tW);
  }
}

__device__ __forceinline__ void euler_state1(const double* u, const double* __restrict__ c, int gm1, int half,
                                             const Reg64& K, double& r, double& v, double& p) {
  r = rcp_k(u[0], K);
  v = K.mul(u[1], r);
  p = K.mul(c[gm1], fma(K.mul(-c[half], u[1]), v, u[2]));  // one rounding of E - m v / 2, which cancels near vacuum
}

// f(uL) + f(uR) - alpha (uR - uL)
template <int PDE, int N>
__device__ __forceinline__ void flux1(const double* L, const double* R, const double* __restrict__ tab, const Reg64& K,
                                      double* G) {
  using T = STab<N>;
  if constexpr (PDE == 0) {
    const double a = max_speed(L[0], R[0]), d = K.sub(L[0], R[0]);
    G[0] = fma(K.mul(tab[T::HALF], L[0]), L[0], fma(K.mul(tab[T::HALF], R[0]), R[0], K.mul(a, d)));
  } else {
    double rL, vL, pL, rR, vR, pR;
    euler_state1(L, tab, T::GM1, T::HALF, K, rL, vL, pL);
    euler_state1(R, tab, T::GM1, T::HALF, K, rR, vR, pR);
    const double c38 = tab[T::C38], half = tab[T::HALF], sg = tab[T::SG];
    const double a = max_speed(fma(sg, sqrt_t(K.mul(pL, rL), K, c38, half), fabs(vL)),
                               fma(sg, sqrt_t(K.mul(pR, rR), K, c38, half), fabs(vR)));
    G[0] = fma(a, K.sub(L[0], R[0]), K.add(L[1], R[1]));
    G[1] = fma(a, K.sub(L[1], R[1]), fma(L[1], vL, fma(R[1], vR, K.add(pL, pR))));
    G[2] = fma(a, K.sub(L[2], R[2]), fma(K.add(L[2], pL), vL, K.mul(K.add(R[2], pR), vR)));
  }
}

// dt times the right-hand side: volume quadrature over symmetric pairs of points, then the
// lifting of the two face fluxes
template <int PDE, int N>
__device__ __forceinline__ void rhs1(const double (&u)[nv_of(1, PDE)][N + 1], const double* FW, const double* FE,
                                     const double* __restrict__ tab, const Reg64& K,
                                     double (&acc)[nv_of(1, PDE)][N + 1]) {
  using T = STab<N>;
  constexpr int V = nv_of(1, PDE), Q = N + 1, N1 = N + 1;
  double uq[V][Q], F[V][Q];
#pragma unroll
  for (int v = 0; v < V; ++v) eval_gauss2<N>(u[v], tab + T::KQ, K, uq[v]);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if constexpr (PDE == 0) {
      F[0][q] = K.mul(K.mul(tab[T::HALF], uq[0][q]), uq[0][q]);
    } else {
      const double w[3] = {uq[0][q], uq[1][q], uq[2][q]};
      double r, vel, p;
      euler_state1(w, tab, T::GM1, T::HALF, K, r, vel, p);
      F[1][q] = fma(w[1], vel, p);
      F[2][q] = K.mul(K.add(w[2], p), vel);
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const double D = K.sub(FE[v], FW[v]), S = K.add(FE[v], FW[v]);
#pragma unroll
    for (int n = 0; n < N1; ++n) {
      double x = K.mul(tab[T::LX + n], (n & 1) ? S : D);
      if (PDE == 1 && v == 0) {  // the density's flux is the momentum, a polynomial
        if (n) x = fma(tab[T::DX + (n ? n - 1 : 0)], u[PDE == 1 ? 1 : 0][n ? n - 1 : 0], x);
        if (n == 3) x = fma(tab[T::DX + 3], u[PDE == 1 ? 1 : 0][0], x);
      } else if (n) {
#pragma unroll
        for (int p = 0; p < Q / 2; ++p)  // psi_n' has the parity of n + 1
          x = fma(tab[T::CX + p * N1 + n], (n & 1) ? K.add(F[v][p], F[v][Q - 1 - p]) : K.sub(F[v][p], F[v][Q - 1 - p]), x);
        if ((Q & 1) && (n & 1)) x = fma(tab[T::CX + (Q / 2) * N1 + n], F[v][Q / 2], x);
      }
      acc[v][n] = x;
    }
  }
}

// stage combination: s = 0, 1, 2
template <int N>
__device__ __forceinline__ double combine(int s, double un, double us, double acc, const double* __restrict__ tab,
                                          const Reg64& K) {
  using T = STab<N>;
  if (s == 0) return K.add(us, acc);
  return fma(tab[T::RA + s], un, K.mul(tab[T::RB + s], K.add(us, acc)));
}

// ----------------------------------------------------------------------------- indicator
// TVB minmod test of one variable; bit-identical to a plain serial sum without fused
// multiply-adds (products and sums as fma(x, y, -0.0) and fma(x, 1, y) round the same).
template <int N>
__device__ __forceinline__ bool tvb1(const double (&u)[N + 1], double u0L, double u0R, long long mh2,
                                     const double* __restrict__ tab, const Reg64& K, bool& near) {
  using T = STab<N>;
  const double p0 = tab[T::P0];
  const double mean = K.mul(u[0], p0), mL = K.mul(u0L, p0), mR = K.mul(u0R, p0);
  double up = K.mul(u[0], tab[T::PP1]), um = up;
#pragma unroll
  for (int n = 1; n < N + 1; ++n) {  // psi_n(-1) = (-1)^n psi_n(1): one product per mode
    const double pc = K.mul(u[n], tab[T::PP1 + n]);
    up = K.add(up, pc);
    um = (n & 1) ? K.sub(um, pc) : K.add(um, pc);
  }
  const double dp = K.sub(mR, mean), dm = K.sub(mean, mL);
  bool f = tvb_changes_bits(K.sub(up, mean), dp, dm, mh2, near);
  f |= tvb_changes_bits(K.sub(mean, um), dp, dm, mh2, near);
  return f;
}

// ----------------------------------------------------------------------------- limiter
// The 2N differences of neighbouring averages over the stencil of Fig. 1: l and r the modes
// of the left and the right neighbour, c0 the troubled cell's U_0.
template <int N>
__device__ __forceinline__ void diffs1(const double (&l)[N + 1], double c0, const double (&r)[N + 1],
                                       const double* __restrict__ lt, const Reg64& K, double (&d)[2 * N]) {
  const double* cs = lt + LimTab<N>::CS;
  const double c = K.mul(cs[0], c0);
#pragma unroll
  for (int side = 0; side < 2; ++side) {  // the right neighbour is read mirrored
    const double* u = side ? r : l;
    const double t = K.mul(cs[0], u[0]);
    double in[2], next;
    if constexpr (N == 1) {
      next = t;
    } else if constexpr (N == 2) {
      const double s = side ? -K.mul(cs[1], u[1]) : K.mul(cs[1], u[1]);
      in[0] = K.add(s, s);
      next = K.add(t, s);
    } else {
      const double o = fma(cs[3], u[3], K.mul(cs[1], u[1])), od = side ? -o : o;
      const double e = K.mul(cs[2], u[2]), e3 = K.add(e, K.add(e, e));
      in[0] = K.sub(od, e3);
      in[1] = K.add(od, e3);
      next = K.add(t, K.add(e, od));
    }
#pragma unroll
    for (int j = 0; j < N - 1; ++j) {
      if (side == 0) d[j] = in[j];
      else d[2 * N - 1 - j] = -in[j];
    }
    if (side == 0) d[N - 1] = K.sub(c, next);
    else d[N] = K.sub(next, c);
  }
}

struct Eig1 {
  double v, hq2, c, ic, H, b1;  // hq2 = v^2 / 2, b1 = (gamma - 1) / c^2
};
__device__ __forceinline__ Eig1 eig1(double rho, double m, double E, double gam, const Reg64& K) {
  Eig1 e;
  const double gm1 = gam - 1.0, r = rcp_k(rho, K);
  e.v = K.mul(m, r);
  e.hq2 = K.mul(0.5 * e.v, e.v);
  const double p = K.mul(gm1, fma(-rho, e.hq2, E));
  e.c = sqrt_d(K.mul(K.mul(gam, p), r));
  e.ic = rcp_k(e.c, K);
  e.H = K.mul(K.add(E, p), r);
  e.b1 = K.mul(K.mul(gm1, e.ic), e.ic);
  return e;
}
__device__ __forceinline__ void to_char1(const Eig1& e, double rho, double m, double E, const Reg64& K, double& w0,
                                         double& w1, double& w2) {
  const double s = fma(-e.v, m, fma(e.hq2, rho, E));  // (gamma-1) s = pressure difference
  const double a = K.mul(0.5 * e.b1, s), d = fma(-e.v, rho, m), hic = 0.5 * e.ic;
  w0 = fma(-hic, d, a);
  w1 = fma(-e.b1, s, rho);
  w2 = fma(hic, d, a);
}
__device__ __forceinline__ void from_char1(const Eig1& e, double w0, double w1, double w2, const Reg64& K, double& rho,
                                           double& m, double& E) {
  const double s = K.add(w0, w2), t = K.mul(e.c, K.sub(w2, w0));
  rho = K.add(s, w1);
  m = fma(e.v, rho, t);
  E = fma(e.H, s, fma(e.v, t, K.mul(e.hq2, w1)));
}

// reconstruction of one (characteristic) field and its modes 1..N (the constant it is
// relative to has none): t[b - 1] = sum_g w_g psi_b(r_g) u(r_g)
template <int N>
__device__ __forceinline__ void field1(const double (&d)[2 * N], const double* __restrict__ lt, const Reg64& K,
                                       double (&t)[N]) {
  using L = LimTab<N>;
  constexpr int NG = L::NG, N1 = N + 1;
  double r[NG];
  weno_diff<N, N == 3, false>(d, lt, K, r);
#pragma unroll
  for (int b = 1; b <= N; ++b) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NG / 2; ++k) {
      const double x = (b & 1) ? K.sub(r[k], r[NG - 1 - k]) : K.add(r[k], r[NG - 1 - k]);
      s = k == 0 ? K.mul(lt[L::PG + b], x) : fma(lt[L::PG + k * N1 + b], x, s);
    }
    t[b - 1] = s;
  }
}

// ----------------------------------------------------------------------------- kernels
// modes of cell ix with the boundary condition (periodic wrap / outflow mirror)
template <int V, int N1>
__device__ __forceinline__ void load_cell(const double* __restrict__ U, long long ctot, const Inst& I, int ix, int bc,
                                          double (&u)[V][N1]) {
  bool flip = false;
  if (bc == 0) {
    ix = ix < 0 ? ix + I.nx : (ix >= I.nx ? ix - I.nx : ix);
  } else {
    if (ix < 0) { ix = 0; flip = true; }
    if (ix >= I.nx) { ix = I.nx - 1; flip = true; }
  }
  const long long g = I.off + ix;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int n = 0; n < N1; ++n) u[v][n] = neg_if(__ldg(U + (long long)(v * N1 + n) * ctot + g), flip && (n & 1));
}

constexpr int kBlock = 256;  // cells per tile of the single-stage kernels

template <int PDE, int N>
__global__ void __launch_bounds__(kBlock)
    k_stage1(const double* __restrict__ un, const double* __restrict__ us, double* __restrict__ out,
             const Inst* __restrict__ insts, const Tile* __restrict__ tiles, long long ctot, int bc, int stage,
             double dt_all, Gamma gm) {
  using T = STab<N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1;
  __shared__ __align__(16) double tab[T::SIZE];
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  fill_tab<PDE, N>(tab, I, dt_all > 0.0 ? dt_all : I.dt, gm);
  __syncthreads();
  const int ix = tile.x0 + threadIdx.x;
  if (ix >= I.nx) return;
  const Reg64 K{tab[T::ONE], tab[T::NZ]};
  double u[V][N1], ul[V][N1], ur[V][N1];
  load_cell<V, N1>(us, ctot, I, ix, bc, u);
  load_cell<V, N1>(us, ctot, I, ix - 1, bc, ul);
  load_cell<V, N1>(us, ctot, I, ix + 1, bc, ur);
  double a[V], b[V], c[V], d[V], x, FW[V], FE[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    traces<N>(ul[v], tab, K, a[v], x);
    traces<N>(u[v], tab, K, c[v], b[v]);
    traces<N>(ur[v], tab, K, x, d[v]);
  }
  flux1<PDE, N>(a, b, tab, K, FW);
  flux1<PDE, N>(c, d, tab, K, FE);
  double acc[V][N1];
  rhs1<PDE, N>(u, FW, FE, tab, K, acc);
  const long long g = I.off + ix;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int n = 0; n < N1; ++n) {
      const long long idx = (long long)(v * N1 + n) * ctot + g;
      out[idx] = combine<N>(stage - 1, stage == 1 ? 0.0 : un[idx], u[v][n], acc[v][n], tab, K);
    }
}

template <int PDE, int N>
__global__ void __launch_bounds__(kBlock)
    k_flag1(const double* __restrict__ U, const Inst* __restrict__ insts, const Tile* __restrict__ tiles,
            long long ctot, int bc, double M, unsigned char* __restrict__ flags, Counters* cnt,
            int* __restrict__ list_cell, int* __restrict__ list_inst) {
  using T = STab<N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1;
  __shared__ __align__(16) double tab[T::XF];
  for (int k = threadIdx.x; k < T::XF; k += kBlock) tab[k] = g_stab[PDE][N - 1][k];
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  __syncthreads();
  const Reg64 K{tab[T::ONE], tab[T::NZ]};
  const int ix = tile.x0 + threadIdx.x;
  int fl = 0;
  bool near = false;
  long long g = 0;
  if (ix < I.nx) {
    g = I.off + ix;
    int jl = ix - 1, jr = ix + 1;
    if (bc == 0) {
      jl = jl < 0 ? jl + I.nx : jl;
      jr = jr >= I.nx ? jr - I.nx : jr;
    } else {
      jl = jl < 0 ? 0 : jl;
      jr = jr >= I.nx ? I.nx - 1 : jr;
    }
    const long long mh2 = __double_as_longlong(M * I.hx * I.hx);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const double* P = U + (long long)(v * N1) * ctot;
      double u[N1];
#pragma unroll
      for (int n = 0; n < N1; ++n) u[n] = __ldg(P + (long long)n * ctot + g);
      fl |= tvb1<N>(u, __ldg(P + I.off + jl), __ldg(P + I.off + jr), mh2, tab, K, near);
    }
    flags[g] = (unsigned char)(fl | (near ? 2 : 0));  // bit 0 troubled, bit 1 near threshold
  }
  block_compact(fl, near ? 1 : 0, g, tile.inst, cnt, list_cell, list_inst);
}

// CSWENO in 1D (Sec. 3) on the listed cells, one thread per cell.
template <int PDE, int N>
__global__ void __launch_bounds__(128)
    k_limit1(const double* __restrict__ U, const Inst* __restrict__ insts, long long ctot, int bc,
             const int* __restrict__ list_cell, const int* __restrict__ list_inst, const Counters* __restrict__ cnt,
             double* __restrict__ lim, long long cap, double gam) {
  using L = LimTab<N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1;
  __shared__ __align__(16) double lt[L::SIZE];
  const unsigned int n = cnt->n_flag;
  if (blockIdx.x * blockDim.x >= n) return;  // whole blocks without a cell leave at once
  for (int k = threadIdx.x; k < L::SIZE; k += 128) lt[k] = g_lim[N - 1][k];
  __syncthreads();
  const Reg64 K{lt[L::ONE], lt[L::NZ]};
  for (unsigned int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const long long g = list_cell[i];
    const Inst I = insts[list_inst[i]];
    const int ix = (int)(g - I.off);
    double d[V][2 * N], t[V][N];
    double ul[V][N1], ur[V][N1], u0[V];
    load_cell<V, N1>(U, ctot, I, ix - 1, bc, ul);
    load_cell<V, N1>(U, ctot, I, ix + 1, bc, ur);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      u0[v] = __ldg(U + (long long)(v * N1) * ctot + g);
      diffs1<N>(ul[v], u0[v], ur[v], lt, K, d[v]);
    }
    if constexpr (PDE == 1) {
      const double p0 = lt[L::P0];
      const Eig1 e = eig1(K.mul(u0[0], p0), K.mul(u0[V > 1 ? 1 : 0], p0), K.mul(u0[V > 1 ? 2 : 0], p0), gam, K);
#pragma unroll
      for (int k = 0; k < 2 * N; ++k)
        to_char1(e, d[0][k], d[V > 1 ? 1 : 0][k], d[V > 1 ? 2 : 0][k], K, d[0][k], d[V > 1 ? 1 : 0][k], d[V > 1 ? 2 : 0][k]);
#pragma unroll
      for (int f = 0; f < V; ++f) field1<N>(d[f], lt, K, t[f]);
#pragma unroll
      for (int b = 0; b < N; ++b)
        from_char1(e, t[0][b], t[V > 1 ? 1 : 0][b], t[V > 1 ? 2 : 0][b], K, t[0][b], t[V > 1 ? 1 : 0][b], t[V > 1 ? 2 : 0][b]);
    } else {
      field1<N>(d[0], lt, K, t[0]);
    }
    // the cell's own higher modes enter no average: a non-finite one stays
    unsigned top = 0;
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int m = 1; m < N1; ++m)
        top = max(top, (unsigned)__double2hiint(__ldg(U + (long long)(v * N1 + m) * ctot + g)) & 0x7fffffffu);
    if constexpr (N == 2) {  // a half has no part of mode 2
#pragma unroll
      for (int v = 0; v < V; ++v)
        top = max(top, max((unsigned)__double2hiint(ul[v][2]) & 0x7fffffffu, (unsigned)__double2hiint(ur[v][2]) & 0x7fffffffu));
    }
    if constexpr (N == 1) {  // whole cells: only the averages enter
#pragma unroll
      for (int v = 0; v < V; ++v)
        top = max(top, max((unsigned)__double2hiint(ul[v][1]) & 0x7fffffffu, (unsigned)__double2hiint(ur[v][1]) & 0x7fffffffu));
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int b = 1; b <= N; ++b)
        lim[(long long)(v * N1 + b) * cap + i] = top >= 0x7ff00000u ? __longlong_as_double(0x7ff8000000000000LL) : t[v][b - 1];
  }
}

// One SSP-RK3 step (three times stage, TVB indicator, CSWENO) of a tile of kStepTile cells.
// Thread i holds cell x0 - kHalo + i (wrapped for periodic instances; for outflow ones the
// threads beyond the boundary idle and the ghost is the boundary cell's mirror image).  The
// values of stage s are right for threads 2s .. kStepThreads - 1 - 2s.  The troubled cells of
// a stage are listed in shared memory and their work spread over the block by (cell,
// variable), (cell, difference) and (cell, field), so that a few troubled cells do not leave
// most of the block's warps idle.
// Measured per step, with five kernels per stage in parentheses: 160 Burgers P2 cells 21 us
// (80), 64 x 800 Euler P3 cells 180 us (468).  Three blocks per SM (448 tiles of the latter on
// 152 SMs) bound the registers to 168; tiles of 84 cells would need a second wave.  (Other batches were
// not measured for the tile's size.)  P3 spills some 350 B per thread at that bound.
constexpr int kStepThreads = 128, kHalo = 6, kStepTile = kStepThreads - 2 * kHalo;

template <int PDE, int N>
struct StepMem {  // doubles of dynamic shared memory
  static constexpr int V = nv_of(1, PDE), N1 = N + 1, ST = V * N1 * kStepThreads;
  static constexpr int OLD = 0, CUR = ST, NEW = 2 * ST, TR = 3 * ST, FL = TR + V * kStepThreads;
  static constexpr int DIF = FL + V * kStepThreads;                           // [2N][V][cell]
  static constexpr int EIG = DIF + 2 * N * V * kStepThreads;                  // [6][cell], Euler
  static constexpr int SIZE = EIG + (PDE == 1 ? 6 : 0) * kStepThreads;
};

template <int PDE, int N>
__global__ void __launch_bounds__(kStepThreads, 3)
    k_step1(const double* __restrict__ un, double* __restrict__ out, const Inst* __restrict__ insts,
            const Tile* __restrict__ tiles, long long ctot, int bc, double M, double gam, Gamma gm,
            unsigned long long* __restrict__ totals) {
  using T = STab<N>;
  using L = LimTab<N>;
  using S = StepMem<PDE, N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1, B = kStepThreads;
  extern __shared__ __align__(16) double sm[];
  __shared__ __align__(16) double tab[T::SIZE];
  __shared__ __align__(16) double lt[L::SIZE];
  __shared__ unsigned s_warp[B / 32], s_count;
  __shared__ unsigned char s_list[B];
  double *const old = sm + S::OLD, *const cur = sm + S::CUR, *const nw = sm + S::NEW, *const sE = sm + S::TR, *const sF = sm + S::FL;
  double *const sd = sm + S::DIF, *const se = sm + S::EIG;
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  fill_tab<PDE, N>(tab, I, I.dt, gm);
  for (int k = threadIdx.x; k < L::SIZE; k += B) lt[k] = g_lim[N - 1][k];
  const int i = threadIdx.x, lane = i & 31, w = i >> 5;
  if (i == 0) s_count = 0;
  const int ix = tile.x0 * kStepTile - kHalo + i;  // (x0 counts tiles)
  const bool active = bc == 0 || (ix >= 0 && ix < I.nx);
  int jx = ix % I.nx;  // the cell this thread loads
  jx = jx < 0 ? jx + I.nx : jx;
  if (bc != 0) jx = ix < 0 ? 0 : (ix >= I.nx ? I.nx - 1 : ix);
  const bool mine = i >= kHalo && i < kHalo + kStepTile && ix < I.nx;  // a cell of this tile
  const bool ghL = bc != 0 && ix <= 0, ghR = bc != 0 && ix >= I.nx - 1;  // neighbour beyond the boundary
  const int il = ghL || i == 0 ? i : i - 1, ir = ghR || i == B - 1 ? i : i + 1;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int n = 0; n < N1; ++n)
      nw[(v * N1 + n) * B + i] = old[(v * N1 + n) * B + i] = un[(long long)(v * N1 + n) * ctot + I.off + jx];
  bool fl = false;  // this cell was limited: its modes 1..N are in cur, the rest of the state in nw
  __syncthreads();
  const Reg64 K{tab[T::ONE], tab[T::NZ]};
  const long long mh2 = __double_as_longlong(M * I.hx * I.hx);
#pragma unroll 1
  for (int s = 0; s < 3; ++s) {
    // stage
    double u[V][N1], tE[V], tW[V], G[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
      for (int n = 0; n < N1; ++n) u[v][n] = (n && fl ? cur : nw)[(v * N1 + n) * B + i];
      traces<N>(u[v], tab, K, tE[v], tW[v]);
      sE[v * B + i] = tE[v];
    }
    __syncthreads();
    {  // the flux at the cell's left face; the thread at ix = nx of an outflow instance has the last one
      double a[V], b[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const double x = sE[v * B + (i ? i - 1 : 0)];
        a[v] = bc != 0 && ix == 0 ? tW[v] : x;
        b[v] = bc != 0 && ix == I.nx ? x : tW[v];
      }
      flux1<PDE, N>(a, b, tab, K, G);
#pragma unroll
      for (int v = 0; v < V; ++v) sF[v * B + i] = G[v];
    }
    __syncthreads();
    double acc[V][N1];
#pragma unroll
    for (int v = 0; v < V; ++v) tE[v] = sF[v * B + (i < B - 1 ? i + 1 : i)];
    rhs1<PDE, N>(u, G, tE, tab, K, acc);
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int n = 0; n < N1; ++n) {
        u[v][n] = combine<N>(s, old[(v * N1 + n) * B + i], u[v][n], acc[v][n], tab, K);
        nw[(v * N1 + n) * B + i] = u[v][n];
      }
    __syncthreads();
    // indicator, on the cells that later stages or the result need
    bool near = false;
    fl = false;
    if (active && i >= 2 * s + 2 && i < B - 2 * s - 2) {
#pragma unroll
      for (int v = 0; v < V; ++v)
        fl |= tvb1<N>(u[v], nw[v * N1 * B + il], nw[v * N1 * B + ir], mh2, tab, K, near);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, fl), own = __ballot_sync(0xffffffffu, fl && mine);
    if (lane == 0) {
      s_warp[w] = __popc(bal);
      if (own) atomicAdd(&s_count, (unsigned)__popc(own));
    }
    __syncthreads();
    unsigned base = 0, nf = 0;
#pragma unroll
    for (int k = 0; k < B / 32; ++k) {
      if (k < w) base += s_warp[k];
      nf += s_warp[k];
    }
    if (fl) s_list[base + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)i;
    if (nf) {
      // limiter: the list's cells read the unlimited neighbours (nw); results go to cur
      __syncthreads();
      for (unsigned k = i; k < nf * V; k += B) {
        const int v = (int)(k / nf), c = (int)(k % nf), j = s_list[c], x = tile.x0 * kStepTile - kHalo + j;
        const bool gl = bc != 0 && x <= 0, gr = bc != 0 && x >= I.nx - 1;
        double l[N1], r[N1], d[2 * N];
        unsigned top = 0;
#pragma unroll
        for (int n = 0; n < N1; ++n) {
          const double a = nw[(v * N1 + n) * B + (gl ? j : j - 1)], b = nw[(v * N1 + n) * B + (gr ? j : j + 1)];
          l[n] = neg_if(a, gl && (n & 1));
          r[n] = neg_if(b, gr && (n & 1));
          top = max(top, max((unsigned)__double2hiint(a) & 0x7fffffffu, (unsigned)__double2hiint(b) & 0x7fffffffu));
          top = max(top, (unsigned)__double2hiint(nw[(v * N1 + n) * B + j]) & 0x7fffffffu);
        }
        diffs1<N>(l, nw[v * N1 * B + j], r, lt, K, d);
        if (top >= 0x7ff00000u) d[0] = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
        for (int q = 0; q < 2 * N; ++q) sd[(q * V + v) * B + c] = d[q];
        if constexpr (PDE == 1) {
          if (v == 0) {
            const double p0 = lt[L::P0];
            const Eig1 e = eig1(K.mul(nw[j], p0), K.mul(nw[N1 * B + j], p0), K.mul(nw[2 * N1 * B + j], p0), gam, K);
            se[c] = e.v;
            se[B + c] = e.hq2;
            se[2 * B + c] = e.c;
            se[3 * B + c] = e.ic;
            se[4 * B + c] = e.H;
            se[5 * B + c] = e.b1;
          }
        }
      }
      __syncthreads();
      if constexpr (PDE == 1) {
        for (unsigned k = i; k < nf * 2 * N; k += B) {
          const int q = (int)(k / nf), c = (int)(k % nf);
          const Eig1 e{se[c], se[B + c], se[2 * B + c], se[3 * B + c], se[4 * B + c], se[5 * B + c]};
          double* p = sd + (q * V) * B + c;
          double w0, w1, w2;
          to_char1(e, p[0], p[B], p[2 * B], K, w0, w1, w2);
          p[0] = w0;
          p[B] = w1;
          p[2 * B] = w2;
        }
        __syncthreads();
      }
      for (unsigned k = i; k < nf * V; k += B) {
        const int f = (int)(k / nf), c = (int)(k % nf);
        double d[2 * N], t[N];
#pragma unroll
        for (int q = 0; q < 2 * N; ++q) d[q] = sd[(q * V + f) * B + c];
        field1<N>(d, lt, K, t);
        if constexpr (PDE == 1) {
#pragma unroll
          for (int b = 0; b < N; ++b) sd[(b * V + f) * B + c] = t[b];
        } else {
#pragma unroll
          for (int b = 0; b < N; ++b) cur[(b + 1) * B + s_list[c]] = t[b];
        }
      }
      if constexpr (PDE == 1) {
        __syncthreads();
        for (unsigned k = i; k < nf * N; k += B) {
          const int b = (int)(k / nf), c = (int)(k % nf), j = s_list[c];
          const Eig1 e{se[c], se[B + c], se[2 * B + c], se[3 * B + c], se[4 * B + c], se[5 * B + c]};
          const double* p = sd + (b * V) * B + c;
          double rho, m, E;
          from_char1(e, p[0], p[B], p[2 * B], K, rho, m, E);
          cur[(b + 1) * B + j] = rho;
          cur[(N1 + b + 1) * B + j] = m;
          cur[(2 * N1 + b + 1) * B + j] = E;
        }
      }
      __syncthreads();
    }
  }
  if (mine) {
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int n = 0; n < N1; ++n)
        out[(long long)(v * N1 + n) * ctot + I.off + ix] = (n && fl ? cur : nw)[(v * N1 + n) * B + i];
  }
  if (i == 0) {  // all lists are counted before the last barrier
    if (s_count) {
      atomicAdd(totals, (unsigned long long)s_count);
      atomicAdd(totals + 1, (unsigned long long)s_count);
    }
    if (blockIdx.x == 0) atomicAdd(totals + 2, 3ull);
  }
}

template <int PDE, int N>
cudaError_t prep() {
  return cudaFuncSetAttribute(k_step1<PDE, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(double) * StepMem<PDE, N>::SIZE));
}

template <int PDE, int N>
void run_step(const LaunchArgs& a, double M, const Gamma& gm, unsigned long long* totals) {
  k_step1<PDE, N><<<a.ntiles, kStepThreads, sizeof(double) * StepMem<PDE, N>::SIZE, a.st>>>(
      a.un, a.out, a.inst, a.tiles, a.ctot, a.bc, M, a.gam, gm, totals);
}

}  // namespace s1

cudaError_t upload_tables_step1(const dgt::Tabs* tabs) {
  static double h[2][3][s1::kSTab], l[3][kLimTab];
  for (int p = 0; p < 2; ++p) {
    s1::pack<1>(tabs[0], p, h[p][0]);
    s1::pack<2>(tabs[1], p, h[p][1]);
    s1::pack<3>(tabs[2], p, h[p][2]);
  }
  pack_lim<1>(tabs[0], l[0]);
  pack_lim<2>(tabs[1], l[1]);
  pack_lim<3>(tabs[2], l[2]);
  cudaError_t e = cudaMemcpyToSymbol(s1::g_stab, h, sizeof(h));
  return e != cudaSuccess ? e : cudaMemcpyToSymbol(s1::g_lim, l, sizeof(l));
}

#define DG_DISPATCH1(PDE, N, CALL) \
  do {                                                   \
    if ((PDE) == 0 && (N) == 1) { constexpr int P_ = 0, N_ = 1; CALL; } \
    else if ((PDE) == 0 && (N) == 2) { constexpr int P_ = 0, N_ = 2; CALL; } \
    else if ((PDE) == 0 && (N) == 3) { constexpr int P_ = 0, N_ = 3; CALL; } \
    else if ((PDE) == 1 && (N) == 1) { constexpr int P_ = 1, N_ = 1; CALL; } \
    else if ((PDE) == 1 && (N) == 2) { constexpr int P_ = 1, N_ = 2; CALL; } \
    else { constexpr int P_ = 1, N_ = 3; CALL; } \
  } while (0)

static Gamma gamma_of(double gam) { return Gamma{gam - 1.0, -0.5 * (gam - 1.0), std::sqrt(gam)}; }

int tile_w1() { return s1::kBlock; }
int step_tile1() { return s1::kStepTile; }

cudaError_t prepare_step1(int pde, int N) {
  cudaError_t e = cudaSuccess;
  DG_DISPATCH1(pde, N, (e = s1::prep<P_, N_>()));
  return e;
}

// one step from a.un to a.out (another buffer); a.tiles: tiles of step_tile1() cells
void launch_step1(int pde, int N, const LaunchArgs& a, double M, unsigned long long* totals) {
  const Gamma gm = gamma_of(a.gam);
  DG_DISPATCH1(pde, N, (s1::run_step<P_, N_>(a, M, gm, totals)));
}

void launch_stage1(int pde, int N, const LaunchArgs& a, int stage, double dt_all) {
  const Gamma gm = gamma_of(a.gam);
  DG_DISPATCH1(pde, N, (s1::k_stage1<P_, N_><<<a.ntiles, s1::kBlock, 0, a.st>>>(a.un, a.us, a.out, a.inst, a.tiles,
                                                                                 a.ctot, a.bc, stage, dt_all, gm)));
}

void launch_flag1(int pde, int N, const LaunchArgs& a, double M, unsigned char* flags, Counters* cnt, int* lc,
                  int* li) {
  DG_DISPATCH1(pde, N, (s1::k_flag1<P_, N_><<<a.ntiles, s1::kBlock, 0, a.st>>>(a.us, a.inst, a.tiles, a.ctot, a.bc,
                                                                                M, flags, cnt, lc, li)));
}

void launch_limit1(int pde, int N, const LaunchArgs& a, const int* lc, const int* li, const Counters* cnt,
                   double* lim, int nblocks) {
  DG_DISPATCH1(pde, N, (s1::k_limit1<P_, N_><<<nblocks, 128, 0, a.st>>>(a.us, a.inst, a.ctot, a.bc, lc, li, cnt,
                                                                          lim, a.cap, a.gam)));
}

}  // namespace dg
