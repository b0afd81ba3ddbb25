// 2D kernels (Cartesian cells, total-degree P^N, N = 1..3; Burgers V = 1, Euler V = 4).
//
//   k_stage2    one stage of Eq. (5) fused in one kernel per tile (halo warps, shared
//               faces), an autotuner alternative to the split stage (dg_stage2.cu)
//   k_flag2     TVB minmod indicator (FP32 screen, FP64 where that is undecided) + ballot/scan
//               compaction of troubled cells
//   k_project2  initial L2 projection (Eq. (2))
//   k_speed2    largest characteristic speed over the cell means
//
// FP64 arithmetic is the bound on GB300 (the FP64 pipe runs at 1/64 of FP32), so the
// kernels are laid out to keep every lane of every FP64 warp instruction useful and to
// avoid recomputing traces or face fluxes.
#include "dg_ic.cuh"
#include "dg_shared.cuh"
#include "tables.h"

namespace dg {
namespace k2 {

constexpr int TX = 32;  // tile width = one warp
constexpr int TY = 8;   // rows per tile of the indicator and projection kernels

// ----------------------------------------------------------------------------- tables
template <int N>
struct Lay {
  static constexpr int Q = N + 1, NP = (N + 1) * (N + 2) / 2;
  static constexpr int N1 = N + 1;
  static constexpr int SIZE_DG = 2 * Q * Q * NP + N1 + 2 * Q * N1;
  static constexpr int SIZE_FLAG = 2 * NP + 1;
  static constexpr int SIZE_PROJ = 3 * 8 + 8 * N1;
  static constexpr int SIZE = SIZE_DG + SIZE_FLAG + SIZE_PROJ;
};
__host__ __device__ constexpr int base_of(int N) {
  return N == 1 ? 0 : (N == 2 ? Lay<1>::SIZE : Lay<1>::SIZE + Lay<2>::SIZE);
}
template <int N>
struct Off {
  using L = Lay<N>;
  static constexpr int Q = L::Q, NP = L::NP, N1 = L::N1;
  static constexpr int VDX = base_of(N);         // [Q*Q][NP] w w psi_a'(x_qx) psi_b(x_qy)
  static constexpr int VDY = VDX + Q * Q * NP;   // w w psi_a(x_qx) psi_b'(x_qy)
  static constexpr int P1 = VDY + Q * Q * NP;    // psi_n(1)
  static constexpr int PQ = P1 + N1;             // [Q][N1] psi_n(x_q)
  static constexpr int WPQ = PQ + Q * N1;        // [Q][N1] w_q psi_n(x_q)
  static constexpr int TE = WPQ + Q * N1;        // [NP] psi_a(1) psi_b(0)
  static constexpr int TN = TE + NP;             // psi_a(0) psi_b(1)
  static constexpr int C00 = TN + NP;            // psi_0(0)^2
  static constexpr int PX = C00 + 1;             // [8]
  static constexpr int PW = PX + 8;              // [8]
  static constexpr int PQP = PW + 8;             // [8] (count in slot 0)
  static constexpr int PP = PQP + 8;             // [8][N1]
  static constexpr int END = PP + 8 * N1;
};
static_assert(Off<3>::END == Lay<1>::SIZE + Lay<2>::SIZE + Lay<3>::SIZE, "table layout");
constexpr int kTabSize = Off<3>::END;

__constant__ double c_tab[kTabSize];
__constant__ float c_tef[3][10], c_tnf[3][10], c_c00f;  // TE, TN and C00 in FP32 (TVB screen)

#define T(x) c_tab[(x)]

template <int N>
void pack(const dgt::Tabs& t, double* h) {
  using O = Off<N>;
  constexpr int Q = O::Q, NP = O::NP, N1 = O::N1;
  for (int qy = 0; qy < Q; ++qy)
    for (int qx = 0; qx < Q; ++qx)
      for (int m = 0; m < NP; ++m) {
        int a = mode_a(m), b = mode_b(m), q = qy * Q + qx;
        double ww = t.gw[qx] * t.gw[qy];
        h[O::VDX + q * NP + m] = ww * t.dpsi_q[qx][a] * t.psi_q[qy][b];
        h[O::VDY + q * NP + m] = ww * t.psi_q[qx][a] * t.dpsi_q[qy][b];
      }
  for (int n = 0; n < N1; ++n) h[O::P1 + n] = t.psi_p1[n];
  for (int q = 0; q < Q; ++q)
    for (int n = 0; n < N1; ++n) {
      h[O::PQ + q * N1 + n] = t.psi_q[q][n];
      h[O::WPQ + q * N1 + n] = t.gw[q] * t.psi_q[q][n];
    }
  for (int m = 0; m < NP; ++m) {
    int a = mode_a(m), b = mode_b(m);
    h[O::TE + m] = t.psi_p1[a] * t.psi_0[b];
    h[O::TN + m] = t.psi_0[a] * t.psi_p1[b];
  }
  h[O::C00] = t.psi_0[0] * t.psi_0[0];
  for (int q = 0; q < t.QP; ++q) {
    h[O::PX + q] = t.px[q];
    h[O::PW + q] = t.pw[q];
    for (int n = 0; n < N1; ++n) h[O::PP + q * N1 + n] = t.ppsi[q][n];
  }
  h[O::PQP] = t.QP;
}

// ----------------------------------------------------------------------------- loads
// Loads the modes of cell (ix, iy) of instance I, applying the boundary condition for
// ghost cells: periodic wraps; outflow mirrors the boundary cell (modes odd in the
// normal direction change sign).
template <int V, int NP>
__device__ __forceinline__ void load_cell(const double* __restrict__ U, long long ctot, const Inst& I, int ix,
                                          int iy, int bc, double (&u)[V][NP]) {
  bool fx = false, fy = false;
  if (bc == 0) {
    ix = ix < 0 ? ix + I.nx : (ix >= I.nx ? ix - I.nx : ix);
    iy = iy < 0 ? iy + I.ny : (iy >= I.ny ? iy - I.ny : iy);
  } else {
    if (ix < 0) { ix = 0; fx = true; }
    if (ix >= I.nx) { ix = I.nx - 1; fx = true; }
    if (iy < 0) { iy = 0; fy = true; }
    if (iy >= I.ny) { iy = I.ny - 1; fy = true; }
  }
  const long long g = I.off + (long long)iy * I.nx + ix;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      double x = __ldg(U + (long long)(v * NP + m) * ctot + g);
      bool flip = (fx && (mode_a(m) & 1)) != (fy && (mode_b(m) & 1));
      u[v][m] = neg_if(x, flip);
    }
}

// Traces on the east (r = +1) and west (r = -1) faces at the Q face points:
// u(+-1, s_q) = sum_b psi_b(s_q) sum_a (+-1)^a U_ab psi_a(1).
template <int N, int V, int NP>
__device__ __forceinline__ void traces_x(const double (&u)[V][NP], double (&tE)[N + 1][V], double (&tW)[N + 1][V]) {
  using O = Off<N>;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    double ev[N + 1], od[N + 1];
#pragma unroll
    for (int b = 0; b <= N; ++b) {
      ev[b] = 0.0;
      od[b] = 0.0;
#pragma unroll
      for (int a = 0; a <= N - b; ++a) {
        double c = u[v][mode_idx(a, b)] * T(O::P1 + a);
        if (a & 1) od[b] += c; else ev[b] += c;
      }
    }
#pragma unroll
    for (int q = 0; q <= N; ++q) {
      double e = 0.0, w = 0.0;
#pragma unroll
      for (int b = 0; b <= N; ++b) {
        e = fma(ev[b] + od[b], T(O::PQ + q * (N + 1) + b), e);
        w = fma(ev[b] - od[b], T(O::PQ + q * (N + 1) + b), w);
      }
      tE[q][v] = e;
      tW[q][v] = w;
    }
  }
}

// Traces on the north (s = +1) and south (s = -1) faces.
template <int N, int V, int NP>
__device__ __forceinline__ void traces_y(const double (&u)[V][NP], double (&tN)[N + 1][V], double (&tS)[N + 1][V]) {
  using O = Off<N>;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    double ev[N + 1], od[N + 1];
#pragma unroll
    for (int a = 0; a <= N; ++a) {
      ev[a] = 0.0;
      od[a] = 0.0;
#pragma unroll
      for (int b = 0; b <= N - a; ++b) {
        double c = u[v][mode_idx(a, b)] * T(O::P1 + b);
        if (b & 1) od[a] += c; else ev[a] += c;
      }
    }
#pragma unroll
    for (int q = 0; q <= N; ++q) {
      double n = 0.0, s = 0.0;
#pragma unroll
      for (int a = 0; a <= N; ++a) {
        n = fma(ev[a] + od[a], T(O::PQ + q * (N + 1) + a), n);
        s = fma(ev[a] - od[a], T(O::PQ + q * (N + 1) + a), s);
      }
      tN[q][v] = n;
      tS[q][v] = s;
    }
  }
}

// Trace on one face at the Q face points for halo cells, which need a single side:
// dir 0: east face (r = +1); dir 1: north face (s = +1).  A halo cell that needs the west
// (south) trace passes its modes with the odd normal degrees negated (mirror image).
template <int N, int V, int NP>
__device__ __forceinline__ void trace_one(const double (&u)[V][NP], int dir, double (&tr)[N + 1][V]) {
  using O = Off<N>;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    double e[N + 1];
#pragma unroll
    for (int t = 0; t <= N; ++t) {  // t: transverse degree
      double s = 0.0;
#pragma unroll
      for (int n = 0; n <= N - t; ++n) {  // n: normal degree
        const int m = dir == 0 ? mode_idx(n, t) : mode_idx(t, n);
        s = fma(u[v][m], T(O::P1 + n), s);
      }
      e[t] = s;
    }
#pragma unroll
    for (int q = 0; q <= N; ++q) {
      double r = 0.0;
#pragma unroll
      for (int t = 0; t <= N; ++t) r = fma(e[t], T(O::PQ + q * (N + 1) + t), r);
      tr[q][v] = r;
    }
  }
}

// ----------------------------------------------------------------------------- stage
// One tile of TX x TYS cells per block (TYS = 4 or 8, chosen by the autotuner).  Warps
// 0..TYS-1 hold the interior rows, warp TYS the row below the tile, warp TYS+1 the row
// above it, warp TYS+2 the west (lanes 0..15) and
// east (lanes 16..31) halo cells, so that every trace and every face flux is computed
// exactly once per tile by a full warp.
template <int PDE, int N, int TYS>
__global__ void __launch_bounds__((TYS + 3) * 32, 1)
    k_stage2(const double* __restrict__ un, const double* __restrict__ us, double* __restrict__ out,
             const Inst* __restrict__ insts, const Tile* __restrict__ tiles, long long ctot, int bc, int stage,
             double dt_all, double gam, int ntiles, int* __restrict__ queue) {
  using O = Off<N>;
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N), Q = N + 1, QV = Q * V;
  // east traces, then x-face fluxes: [QV][TYS][TX+1]; north traces, then y-face fluxes:
  // [QV][TYS+1][TX] (dynamic shared memory, above the 48 KB static limit for Euler P2/P3)
  extern __shared__ double smem[];
  double* const sEb = smem;
  double* const sNb = smem + QV * TYS * (TX + 1);
#define sE(qv, r, c) sEb[((qv) * TYS + (r)) * (TX + 1) + (c)]
#define sN(qv, r, c) sNb[((qv) * (TYS + 1) + (r)) * TX + (c)]
  // one tile per block, or (queue != null) a persistent block taking tiles from the queue
  __shared__ int s_tile;
  int tix = blockIdx.x;
  if (queue) {
    if (threadIdx.x == 0) s_tile = atomicAdd(queue, 1);
    __syncthreads();
    tix = s_tile;
  }
  while (tix < ntiles) {
  const Tile tile = tiles[tix];
  const Inst I = insts[tile.inst];
  const int ncols = min(TX, I.nx - tile.x0), nrows = min(TYS, I.ny - tile.y0);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double gm1 = gam - 1.0;
  const double sx = 2.0 / I.hx, sy = 2.0 / I.hy, ihx = 1.0 / I.hx, ihy = 1.0 / I.hy;

  const bool interior = w < TYS && w < nrows && lane < ncols;
  double acc[V][NP];
  double trW[Q][V], trS[Q][V];
  // ---------------------------------------------------------------- phase 1
  if (interior) {
    double u[V][NP];
    load_cell<V, NP>(us, ctot, I, tile.x0 + lane, tile.y0 + w, bc, u);
    double tE[Q][V], tN[Q][V];
    traces_x<N>(u, tE, trW);
    traces_y<N>(u, tN, trS);
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        sE(q * V + v, w, lane + 1) = tE[q][v];
        sN(q * V + v, w + 1, lane) = tN[q][v];
      }
    // volume term: (2/hx) sum_q w w f psi_a' psi_b + (2/hy) sum_q w w g psi_a psi_b'
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int m = 0; m < NP; ++m) acc[v][m] = 0.0;
#pragma unroll
    for (int qx = 0; qx < Q; ++qx) {
      // sum factorisation: t_b(x_qx) = sum_a U_ab psi_a(x_qx), then u = sum_b t_b psi_b(y_qy)
      double tb[V][N + 1];
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int b = 0; b <= N; ++b) {
          double t = u[v][mode_idx(0, b)] * T(O::PQ + qx * (N + 1));
#pragma unroll
          for (int a = 1; a <= N - b; ++a) t = fma(u[v][mode_idx(a, b)], T(O::PQ + qx * (N + 1) + a), t);
          tb[v][b] = t;
        }
#pragma unroll
      for (int qy = 0; qy < Q; ++qy) {
        const int q = qy * Q + qx;
        double uq[V], f[V], g[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          double t = tb[v][0] * T(O::PQ + qy * (N + 1));
#pragma unroll
          for (int b = 1; b <= N; ++b) t = fma(tb[v][b], T(O::PQ + qy * (N + 1) + b), t);
          uq[v] = t;
        }
        vol_flux2<2, PDE>(uq, f, g, sx, sy, gm1);
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int m = 1; m < NP; ++m) {
            if (mode_a(m) >= 1) acc[v][m] = fma(f[v], T(O::VDX + q * NP + m), acc[v][m]);
            if (mode_b(m) >= 1) acc[v][m] = fma(g[v], T(O::VDY + q * NP + m), acc[v][m]);
          }
      }
    }
  } else if (w == TYS) {  // row below the tile: its north traces
    if (lane < ncols) {
      double u[V][NP], tN[Q][V];
      load_cell<V, NP>(us, ctot, I, tile.x0 + lane, tile.y0 - 1, bc, u);
      trace_one<N>(u, 1, tN);
#pragma unroll
      for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) sN(q * V + v, 0, lane) = tN[q][v];
    }
  } else if (w == TYS + 1) {  // row above the tile: its south traces (kept for phase 2)
    if (lane < ncols) {
      double u[V][NP];
      load_cell<V, NP>(us, ctot, I, tile.x0 + lane, tile.y0 + nrows, bc, u);
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int m = 0; m < NP; ++m)
          if (mode_b(m) & 1) u[v][m] = neg_if(u[v][m], true);
      trace_one<N>(u, 1, trS);
    }
  } else if (w == TYS + 2) {  // west halo (lanes < 16) east traces, east halo west traces
    const bool east = lane >= 16;
    const int row = east ? lane - 16 : lane;
    if (row < nrows) {
      double u[V][NP], tA[Q][V];
      load_cell<V, NP>(us, ctot, I, east ? tile.x0 + ncols : tile.x0 - 1, tile.y0 + row, bc, u);
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int m = 0; m < NP; ++m)
          u[v][m] = neg_if(u[v][m], east && (mode_a(m) & 1));
      trace_one<N>(u, 0, tA);
#pragma unroll
      for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          if (!east) sE(q * V + v, row, 0) = tA[q][v];
          trW[q][v] = tA[q][v];
        }
    }
  }
  __syncthreads();
  // ---------------------------------------------------------------- phase 2: face fluxes
  if (interior) {
    double uL[V], uR[V], fs[V];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        uL[v] = sE(q * V + v, w, lane);
        uR[v] = trW[q][v];
      }
      llf<2, PDE>(0, uL, uR, fs, ihx, gam, gm1);
#pragma unroll
      for (int v = 0; v < V; ++v) sE(q * V + v, w, lane) = fs[v];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        uL[v] = sN(q * V + v, w, lane);
        uR[v] = trS[q][v];
      }
      llf<2, PDE>(1, uL, uR, fs, ihy, gam, gm1);
#pragma unroll
      for (int v = 0; v < V; ++v) sN(q * V + v, w, lane) = fs[v];
    }
  } else if (w == TYS + 1) {
    if (lane < ncols) {
      double uL[V], fs[V];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
#pragma unroll
        for (int v = 0; v < V; ++v) uL[v] = sN(q * V + v, nrows, lane);
        llf<2, PDE>(1, uL, trS[q], fs, ihy, gam, gm1);
#pragma unroll
        for (int v = 0; v < V; ++v) sN(q * V + v, nrows, lane) = fs[v];
      }
    }
  } else if (w == TYS + 2) {
    const int row = lane - 16;
    if (lane >= 16 && row < nrows) {
      double uL[V], fs[V];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
#pragma unroll
        for (int v = 0; v < V; ++v) uL[v] = sE(q * V + v, row, ncols);
        llf<2, PDE>(0, uL, trW[q], fs, ihx, gam, gm1);
#pragma unroll
        for (int v = 0; v < V; ++v) sE(q * V + v, row, ncols) = fs[v];
      }
    }
  }
  __syncthreads();
  // ---------------------------------------------------------------- phase 3: lift + RK
  if (interior) {
#pragma unroll
  for (int v = 0; v < V; ++v) {
    // x faces: acc_ab -= psi_a(1) sum_q w_q psi_b(s_q) [F_E(q) - (-1)^a F_W(q)]
    double dxs[Q], sxs[Q], dys[Q], sys[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      double fe = sE(q * V + v, w, lane + 1), fw = sE(q * V + v, w, lane);
      double fn = sN(q * V + v, w + 1, lane), fsv = sN(q * V + v, w, lane);
      dxs[q] = fe - fw;
      sxs[q] = fe + fw;
      dys[q] = fn - fsv;
      sys[q] = fn + fsv;
    }
#pragma unroll
    for (int b = 0; b <= N; ++b) {
      double Sp = 0.0, Sm = 0.0, Tp = 0.0, Tm = 0.0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const double c = T(O::WPQ + q * (N + 1) + b);
        Sp = fma(c, dxs[q], Sp);
        Sm = fma(c, sxs[q], Sm);
        Tp = fma(c, dys[q], Tp);
        Tm = fma(c, sys[q], Tm);
      }
      // here b plays the transverse index: x faces use psi_b(s), y faces psi_a(r)
#pragma unroll
      for (int a = 0; a <= N - b; ++a) {
        const int mx = mode_idx(a, b);  // x faces: transverse degree b, normal degree a
        acc[v][mx] = fma(-T(O::P1 + a), (a & 1) ? Sm : Sp, acc[v][mx]);
        const int my = mode_idx(b, a);  // y faces: transverse degree b (in x), normal a
        acc[v][my] = fma(-T(O::P1 + a), (a & 1) ? Tm : Tp, acc[v][my]);
      }
    }
  }
  const long long g = I.off + (long long)(tile.y0 + w) * I.nx + tile.x0 + lane;
  const double dt = dt_all > 0.0 ? dt_all : I.dt;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      const long long idx = (long long)(v * NP + m) * ctot + g;
      double e = fma(dt, acc[v][m], us[idx]);
      double r;
      if (stage == 1) r = e;
      else if (stage == 2) r = fma(0.75, un[idx], 0.25 * e);
      else r = fma(1.0 / 3.0, un[idx], (2.0 / 3.0) * e);
      out[idx] = r;
    }
  }  // interior
  if (!queue) break;
  __syncthreads();  // shared memory and s_tile are reused by the next tile
  if (threadIdx.x == 0) s_tile = atomicAdd(queue, 1);
  __syncthreads();
  tix = s_tile;
  }  // tiles
}

#undef sE
#undef sN

// ----------------------------------------------------------------------------- indicator
// TVB modified minmod (Cockburn-Shu) on conserved variables, x test on the east/west
// edge midpoints and y test on the north/south ones.  The face values and means are
// formed without fused multiply-adds and in the order of a plain serial sum over the
// modes, so the decision is reproducible bit for bit; products whose table factor is
// exactly zero (psi_b(0) for odd b) are skipped, which leaves every partial sum unchanged.
//
// In FP64 that is 42 additions and products per variable (P2), bound by the FP64 pipe.  Nearly
// every comparison is far from a tie, so an FP32 screen with error margins decides them first
// (tvb_screen) and only cells with a comparison inside its margins take the FP64 pass.

// The FP64 decision of one cell, variable and direction (0: x, 1: y): bit 0 troubled, bit 1
// near threshold.
template <int PDE, int N>
__device__ __noinline__ int tvb_cell(const double* __restrict__ U, const Inst& I, int inst, int ix, int iy, int v,
                                     int dir, long long ctot, int bc, double M, const double* __restrict__ bcd) {
  using O = Off<N>;
  constexpr int NP = np_of(2, N);
  const double c00 = T(O::C00);
  const double* P = U + (long long)(v * NP) * ctot;
  const long long g = I.off + (long long)iy * I.nx + ix;
  bool near = false;
  // a neighbour's U_00: periodic wrap, outflow ghosts have the boundary cell's mean, kBcDmr
  // ghosts follow dmr_ghost
  auto nb_u00 = [&](int jx, int jy) -> double {
    if (bc == 0) {
      jx = jx < 0 ? jx + I.nx : (jx >= I.nx ? jx - I.nx : jx);
      jy = jy < 0 ? jy + I.ny : (jy >= I.ny ? jy - I.ny : jy);
    } else if (bc == kBcDmr && (jx < 0 || jx >= I.nx || jy < 0 || jy >= I.ny)) {
      const Ghost gh = dmr_ghost(I, inst, jx, jy, bcd, dmr_time(bcd, inst, 0));
      if (gh.c) return 2.0 * gh.c[v];
      return neg_if(__ldg(P + I.off + (long long)gh.jy * I.nx + gh.jx), gh.fv && v == 2);
    } else {
      jx = jx < 0 ? 0 : (jx >= I.nx ? I.nx - 1 : jx);
      jy = jy < 0 ? 0 : (jy >= I.ny ? I.ny - 1 : jy);
    }
    return __ldg(P + I.off + (long long)jy * I.nx + jx);
  };
  const double h = dir == 0 ? I.hx : I.hy;
  const long long mh2 = __double_as_longlong(M * h * h);
  const double mean = __dmul_rn(__ldg(P + g), c00);
  const double mL = __dmul_rn(dir == 0 ? nb_u00(ix - 1, iy) : nb_u00(ix, iy - 1), c00);
  const double mR = __dmul_rn(dir == 0 ? nb_u00(ix + 1, iy) : nb_u00(ix, iy + 1), c00);
  // values at the midpoints of the two edges.  The serial sums start from their first term
  // (0 + x = x up to the sign of a zero, which no decision below depends on).
  double up = 0.0, um = 0.0;
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    const int n = dir == 0 ? mode_a(m) : mode_b(m), t = dir == 0 ? mode_b(m) : mode_a(m);
    if (t & 1) continue;  // psi_t(0) = 0
    // lower = (-1)^n upper, term by term
    const double p = __dmul_rn(__ldg(P + (long long)m * ctot + g), dir == 0 ? T(O::TE + m) : T(O::TN + m));
    up = m == 0 ? p : __dadd_rn(up, p);
    um = m == 0 ? p : ((n & 1) ? __dsub_rn(um, p) : __dadd_rn(um, p));
  }
  const double dp = __dsub_rn(mR, mean), dm = __dsub_rn(mean, mL);
  int fl = tvb_changes_bits(__dsub_rn(up, mean), dp, dm, mh2, near);
  fl |= tvb_changes_bits(__dsub_rn(mean, um), dp, dm, mh2, near);
  return fl | (near ? 2 : 0);
}

// ---- FP32 screen (exactness argument).  With m the mean, d a mean difference and
// a = edge value - mean of the FP64 decision, S = sum_{n>=1} |U_n t_n| (t_n: table values):
//   - a: the FP64 value is within (NP + 1) 2^-53 (|m| + S) < 2^-49 (|m| + S) of the exact
//     sum_{n>=1} U_n t_n (U_0's product is the mean's, bit for bit).  In FP32 every U_n is
//     truncated (2^-23) and every product and sum rounded (2^-24, at most 10 of them):
//     within 2^-20 S.  Margin 2^-19 S + 2^-46 |m|.
//   - d: a mean is kept as two floats, its leading 24 bits and the rest, exact to 2^-47 |m|;
//     the differences of the parts and their sum round relative to the result (2^-24 each),
//     the FP64 means and difference to 2^-52 |m|.  Margin 2^-21 |d| + 2^-44 max |m|.
//   - every margin also holds 2^-100 for parts below the float range; infinities and NaN
//     satisfy none of the comparisons below.
//   - a value above mhi >= 0 with its margin has a known sign.
// A test is decided when its comparisons hold with the margins and the windows of
// tvb_changes_bits (2^-37 relative, 2^-39 of the largest magnitude) to spare: then the FP64
// test decides the same and is not near a threshold.
// double -> float by truncation without branches: values below 2^-126 give at most 2^-126,
// those above the float range (and NaN) an infinity or a NaN.
__device__ __forceinline__ float trunc_f(double x) {
  const int hi = __double2hiint(x);
  const int e = min(max((hi & 0x7fffffff) - (896 << 20), 0), 255 << 20);
  return __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)e, 3) | ((unsigned)hi & 0x80000000u));
}
struct Mean2 {  // U_00 (the mean over psi_0^2) as leading part and rest
  float h, l;
};
__device__ __forceinline__ Mean2 split_mean(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff) - 1023;
  Mean2 r;
  r.h = trunc_f(x);
  // low 29 bits times 2^(e - 52), in range for |x| in [2^-60, 2^120]; outside the rest is made
  // a NaN, which leaves the cell to FP64 (0 has none)
  const float sc = __uint_as_float((unsigned)(e - 52 + 127) << 23);
  const float l = __uint2float_rn(lo & 0x1fffffffu) * sc;
  r.l = __uint_as_float(__float_as_uint(l) | (hi & 0x80000000u));
  if (e < -60 || e > 120) r.l = (hi << 1) | lo ? __uint_as_float(0x7fc00000u) : 0.0f;
  return r;
}
__device__ __forceinline__ float mean_diff(Mean2 a, Mean2 b) { return (a.h - b.h) + (a.l - b.l); }

// The two tests of one direction (bit 0: the FP64 test finds a change; bit 1: undecided).
// a0, a1, ma: edge values minus mean (mean minus edge value) and margin; dp, dm, md: the mean
// differences and their margin; mlo, mhi: bounds of M h^2.
__device__ __forceinline__ int tvb_screen(float a0, float a1, float ma, float dp, float dm, float md, float mlo,
                                          float mhi) {
  const float p = fabsf(dp), q = fabsf(dm), mp = fmaf(p, 0x1p-21f, md), mq = fmaf(q, 0x1p-21f, md);
  const float plo = p - mp, qlo = q - mq, phi = p + mp, qhi = q + mq;
  const float lo2 = fminf(plo, qlo), hi2 = fminf(phi, qhi), top2 = fmaxf(phi, qhi);
  const bool same = (dp > 0.0f) == (dm > 0.0f);
  int r = 0;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float a = k ? a1 : a0, fa = fabsf(a), lo = fa - ma, hi = fa + ma;
    const float top = fmaxf(hi, top2) * 0x1p-38f;
    const bool sure = lo > mhi && plo > top && qlo > top;  // above M h^2, no mean difference near zero
    const bool agree = same && (a > 0.0f) == (dp > 0.0f);
    const bool yes = sure && (!agree || lo > hi2 * (1.0f + 0x1p-20f));
    const bool no = hi < mlo || (sure && agree && hi < lo2 * (1.0f - 0x1p-20f));
    r |= yes ? 1 : (no ? 0 : 2);
  }
  return r;
}

// One thread per cell of a 32 x 8 tile: screen, then the block's undecided cells (listed in
// shared memory, so that they fill whole warps) in FP64.  The tile's means and those of the
// cells around it are split once, into shared memory.
// Measured: 1024^2 Euler P2 0.07 ms (0.35 ms with every cell in FP64), P3 batch of 1.10 M
// cells 0.09 ms (0.49).
template <int PDE, int N>
__global__ void __launch_bounds__(256)
    k_flag2(const double* __restrict__ U, const Inst* __restrict__ insts, const Tile* __restrict__ tiles,
            long long ctot, int bc, double M, unsigned char* __restrict__ flags, Counters* cnt,
            int* __restrict__ list_cell, int* __restrict__ list_inst, const double* __restrict__ bcd) {
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N), BX = TX + 2, BY = TY + 2;
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ix = tile.x0 + lane, iy = tile.y0 + w;
  const bool active = ix < I.nx && iy < I.ny;
  const long long g = active ? I.off + (long long)iy * I.nx + ix : 0;
  __shared__ Mean2 s_mean[V][BY][BX];
  __shared__ unsigned char s_todo[TX * TY];
  __shared__ int s_res[TX * TY];
  __shared__ int s_n;
  __shared__ float s_mh2[2];  // M h^2, truncated
  if (threadIdx.x == 0) {
    s_n = 0;
    s_mh2[0] = trunc_f(M * I.hx * I.hx);
    s_mh2[1] = trunc_f(M * I.hy * I.hy);
  }
  for (int k = threadIdx.x; k < BX * BY; k += TX * TY) {
    const int cy = k / BX, cx = k % BX;
    int jx = tile.x0 + cx - 1, jy = tile.y0 + cy - 1;
    if (jx > I.nx || jy > I.ny || ((cx == 0 || cx == BX - 1) && (cy == 0 || cy == BY - 1))) continue;
    if (bc == 0) {
      jx = jx < 0 ? jx + I.nx : (jx >= I.nx ? jx - I.nx : jx);
      jy = jy < 0 ? jy + I.ny : (jy >= I.ny ? jy - I.ny : jy);
    } else {  // outflow ghosts have the boundary cell's mean
      jx = jx < 0 ? 0 : (jx >= I.nx ? I.nx - 1 : jx);
      jy = jy < 0 ? 0 : (jy >= I.ny ? I.ny - 1 : jy);
    }
    const double* p = U + I.off + (long long)jy * I.nx + jx;
#pragma unroll
    for (int v = 0; v < V; ++v) s_mean[v][cy][cx] = split_mean(__ldg(p + (long long)(v * NP) * ctot));
  }
  __syncthreads();
  int fl = 0;
  if (active) {
    // the double Mach reflection's ghosts are left to FP64
    if (bc == kBcDmr && (ix == 0 || iy == 0 || ix == I.nx - 1 || iy == I.ny - 1)) fl = 2;
    // (a negative M, which dg_step and dg_harvest take: mlo is not met then, and mhi must not
    // fall below 0, or a sign that the margin leaves open would count as known)
    const float xlo = s_mh2[0] * (1.0f - 0x1p-20f), ylo = s_mh2[1] * (1.0f - 0x1p-20f);
    const float xhi = s_mh2[0] < 0.0f ? 0x1p-100f : fmaf(s_mh2[0], 1.0f + 0x1p-20f, 0x1p-100f);
    const float yhi = s_mh2[1] < 0.0f ? 0x1p-100f : fmaf(s_mh2[1], 1.0f + 0x1p-20f, 0x1p-100f);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const double* P = U + (long long)(v * NP) * ctot + g;
      // edge values minus the mean: parts odd and even in the normal degree, and the sum of magnitudes
      float ox = 0.0f, ex = 0.0f, oy = 0.0f, ey = 0.0f, sx = 0.0f, sy = 0.0f;
#pragma unroll
      for (int m = 1; m < NP; ++m) {
        const int a = mode_a(m), b = mode_b(m);
        if ((a & 1) && (b & 1)) continue;  // psi_a(0) = psi_b(0) = 0
        const float u = trunc_f(__ldg(P + (long long)m * ctot));
        if (!(b & 1)) {
          const float t = u * c_tef[N - 1][m];
          if (a & 1) ox += t;
          else ex += t;
          sx += fabsf(t);
        }
        if (!(a & 1)) {
          const float t = u * c_tnf[N - 1][m];
          if (b & 1) oy += t;
          else ey += t;
          sy += fabsf(t);
        }
      }
      const Mean2 mC = s_mean[v][w + 1][lane + 1], mW = s_mean[v][w + 1][lane], mE = s_mean[v][w + 1][lane + 2];
      const Mean2 mS = s_mean[v][w][lane + 1], mN = s_mean[v][w + 2][lane + 1];
      // in units of U_00 the mean is U_00 psi_0^2; the differences below take that factor
      const float c = c_c00f, am = fabsf(mC.h) * c;
      const float bx = fmaf(fmaxf(am, c * fmaxf(fabsf(mE.h), fabsf(mW.h))), 0x1p-44f, 0x1p-100f);
      const float by = fmaf(fmaxf(am, c * fmaxf(fabsf(mN.h), fabsf(mS.h))), 0x1p-44f, 0x1p-100f);
      const float rm = fmaf(am, 0x1p-46f, 0x1p-100f);
      fl |= tvb_screen(ox + ex, ox - ex, fmaf(sx, 0x1p-19f, rm), c * mean_diff(mE, mC), c * mean_diff(mC, mW), bx, xlo, xhi);
      fl |= tvb_screen(oy + ey, oy - ey, fmaf(sy, 0x1p-19f, rm), c * mean_diff(mN, mC), c * mean_diff(mC, mS), by, ylo, yhi);
    }
    if (fl & 2) {
      s_todo[atomicAdd(&s_n, 1)] = (unsigned char)threadIdx.x;
      s_res[threadIdx.x] = 0;
    }
  }
  __syncthreads();
  // (a cell's variables and directions on neighbouring threads: the block waits for a few
  // cells, so the chain of dependent FP64 operations is kept short)
  for (int k = threadIdx.x; k < s_n * 2 * V; k += TX * TY) {
    const int t = s_todo[k / (2 * V)], v = (k >> 1) % V, dir = k & 1;
    const int r = tvb_cell<PDE, N>(U, I, tile.inst, tile.x0 + (t & 31), tile.y0 + (t >> 5), v, dir, ctot, bc, M, bcd);
    if (r) atomicOr(&s_res[t], r);
  }
  __syncthreads();
  bool near = false;
  if (fl & 2) {
    fl = s_res[threadIdx.x];
    near = (fl & 2) != 0;
  }
  fl &= 1;
  if (active) flags[g] = (unsigned char)(fl | (near ? 2 : 0));  // bit 0 troubled, bit 1 near threshold
  block_compact(fl, near ? 1 : 0, g, tile.inst, cnt, list_cell, list_inst);
}

// ----------------------------------------------------------------------------- projection
// Eq. (2) for the initial data: U_ab = sum_{qx,qy} w w u0(x, y) psi_a psi_b with N+4 Gauss
// points per direction.  Parameters per instance (see dg.h for the families).

template <int PDE, int N>
__global__ void k_project2(double* __restrict__ U, const Inst* __restrict__ insts, const int* __restrict__ cell_inst,
                           long long ncell, long long ctot, int kind, const double* __restrict__ params, int np,
                           double gam) {
  using O = Off<N>;
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N), N1 = N + 1;
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  const int ii = cell_inst[g];
  const Inst I = insts[ii];
  const int loc = (int)(g - I.off), ix = loc % I.nx, iy = loc / I.nx;
  const double* p = params + (long long)ii * np;
  const int QP = (int)T(O::PQP);
  double acc[V][NP];
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int m = 0; m < NP; ++m) acc[v][m] = 0.0;
  for (int qy = 0; qy < QP; ++qy)
    for (int qx = 0; qx < QP; ++qx) {
      const double x = I.xL + I.hx * (ix + 0.5 * (1.0 + T(O::PX + qx)));
      const double y = I.yL + I.hy * (iy + 0.5 * (1.0 + T(O::PX + qy)));
      double u[V];
      ic_eval2(kind, p, x, y, gam, u);
      const double ww = T(O::PW + qx) * T(O::PW + qy);
#pragma unroll
      for (int m = 0; m < NP; ++m) {
        const double c = ww * T(O::PP + qx * N1 + mode_a(m)) * T(O::PP + qy * N1 + mode_b(m));
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v][m] = fma(c, u[v], acc[v][m]);
      }
    }
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int m = 0; m < NP; ++m) U[(long long)(v * NP + m) * ctot + g] = acc[v][m];
}

template <int PDE, int N>
__global__ void k_speed2(const double* __restrict__ U, const Inst* __restrict__ insts, const int* __restrict__ cell_inst,
                         long long ncell, long long ctot, double gam, double* out) {
  using O = Off<N>;
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N);
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  double u[V];
  for (int v = 0; v < V; ++v) u[v] = U[(long long)(v * NP) * ctot + g] * T(O::C00);
  double sx, sy;
  if constexpr (PDE == 0) {
    sx = sy = fabs(u[0]);
  } else {
    const double r = 1.0 / u[0], vx = u[1] * r, vy = u[2] * r;
    const double p = (gam - 1.0) * (u[3] - 0.5 * u[0] * (vx * vx + vy * vy));
    const double c = sqrt(gam * p * r);
    sx = fabs(vx) + c;
    sy = fabs(vy) + c;
  }
  const int ii = cell_inst[g];
  atomic_max_nonneg(out + 2 * ii, sx);
  atomic_max_nonneg(out + 2 * ii + 1, sy);
}

#undef T

}  // namespace k2

// ----------------------------------------------------------------------------- host side

cudaError_t upload_tables2(const dgt::Tabs* tabs /* [3] for N = 1..3 */) {
  static double h[k2::kTabSize];
  for (int i = 0; i < k2::kTabSize; ++i) h[i] = 0.0;
  k2::pack<1>(tabs[0], h);
  k2::pack<2>(tabs[1], h);
  k2::pack<3>(tabs[2], h);
  static float te[3][10], tn[3][10];
  for (int n = 0; n < 3; ++n)
    for (int m = 0; m < np_of(2, n + 1); ++m) {
      const int base = n == 0 ? k2::Off<1>::TE : (n == 1 ? k2::Off<2>::TE : k2::Off<3>::TE);
      const int bn = n == 0 ? k2::Off<1>::TN : (n == 1 ? k2::Off<2>::TN : k2::Off<3>::TN);
      te[n][m] = (float)h[base + m];
      tn[n][m] = (float)h[bn + m];
    }
  const float c00 = (float)h[k2::Off<1>::C00];
  cudaError_t e = cudaMemcpyToSymbol(k2::c_tab, h, sizeof(h));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(k2::c_tef, te, sizeof(te));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(k2::c_tnf, tn, sizeof(tn));
  return e != cudaSuccess ? e : cudaMemcpyToSymbol(k2::c_c00f, &c00, sizeof(c00));
}

#define DG_DISPATCH2(PDE, N, CALL) \
  do {                                                   \
    if ((PDE) == 0 && (N) == 1) { constexpr int P_ = 0, N_ = 1; CALL; } \
    else if ((PDE) == 0 && (N) == 2) { constexpr int P_ = 0, N_ = 2; CALL; } \
    else if ((PDE) == 0 && (N) == 3) { constexpr int P_ = 0, N_ = 3; CALL; } \
    else if ((PDE) == 1 && (N) == 1) { constexpr int P_ = 1, N_ = 1; CALL; } \
    else if ((PDE) == 1 && (N) == 2) { constexpr int P_ = 1, N_ = 2; CALL; } \
    else { constexpr int P_ = 1, N_ = 3; CALL; } \
  } while (0)

int stage_threads2(int tys) { return (tys + 3) * 32; }

template <int PDE, int N, int TYS>
static size_t stage_smem2() {
  constexpr int QV = (N + 1) * nv_of(2, PDE);
  return sizeof(double) * (size_t)(QV * TYS * (k2::TX + 1) + QV * (TYS + 1) * k2::TX);
}

template <int PDE, int N>
static cudaError_t prep_stage2() {
  // opt in to more than 48 KB of dynamic shared memory (set per device, outside captures)
  cudaError_t e = cudaFuncSetAttribute(k2::k_stage2<PDE, N, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)stage_smem2<PDE, N, 8>());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k2::k_stage2<PDE, N, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)stage_smem2<PDE, N, 4>());
}

cudaError_t prepare2(int pde, int N) {
  cudaError_t e = cudaSuccess;
  DG_DISPATCH2(pde, N, (e = prep_stage2<P_, N_>()));
  return e;
}

template <int PDE, int N, int TYS>
static void run_stage2(const LaunchArgs& a, int stage, double dt_all, int* queue, int grid) {
  const size_t bytes = stage_smem2<PDE, N, TYS>();
  k2::k_stage2<PDE, N, TYS><<<queue ? grid : a.ntiles, (TYS + 3) * 32, bytes, a.st>>>(
      a.un, a.us, a.out, a.inst, a.tiles, a.ctot, a.bc, stage, dt_all, a.gam, a.ntiles, queue);
}
int tile_w2() { return k2::TX; }
int tile_h2() { return k2::TY; }

// queue != null: persistent launch of `grid` blocks popping tiles from *queue (zeroed by the
// caller before the launch); otherwise one block per tile
void launch_stage2(int pde, int N, const LaunchArgs& a, int stage, double dt_all, int tys, int* queue, int grid) {
  if (tys == 4) DG_DISPATCH2(pde, N, (run_stage2<P_, N_, 4>(a, stage, dt_all, queue, grid)));
  else DG_DISPATCH2(pde, N, (run_stage2<P_, N_, 8>(a, stage, dt_all, queue, grid)));
}

void launch_flag2(int pde, int N, const LaunchArgs& a, double M, unsigned char* flags, Counters* cnt, int* lc,
                  int* li) {
  DG_DISPATCH2(pde, N, (k2::k_flag2<P_, N_><<<a.ntiles, 256, 0, a.st>>>(a.us, a.inst, a.tiles, a.ctot, a.bc, M,
                                                                          flags, cnt, lc, li, a.bcd)));
}

void launch_scatter2(int pde, int N, const LaunchArgs& a, const double* lim, const int* lc, const Counters* cnt,
                     int nblocks) {
  DG_DISPATCH2(pde, N, (k_scatter<nv_of(2, P_), np_of(2, N_)><<<nblocks, 256, 0, a.st>>>(
                           a.out, a.ctot, lim, a.cap, lc, cnt)));
}

void launch_project2(int pde, int N, const LaunchArgs& a, const int* cell_inst, int kind, const double* params,
                     int np) {
  const int nb = (int)((a.ncell + 127) / 128);
  DG_DISPATCH2(pde, N, (k2::k_project2<P_, N_><<<nb, 128, 0, a.st>>>(a.out, a.inst, cell_inst, a.ncell, a.ctot,
                                                                       kind, params, np, a.gam)));
}

void launch_speed2(int pde, int N, const LaunchArgs& a, const int* cell_inst, double* out) {
  const int nb = (int)((a.ncell + 255) / 256);
  DG_DISPATCH2(pde, N, (k2::k_speed2<P_, N_><<<nb, 256, 0, a.st>>>(a.us, a.inst, cell_inst, a.ncell, a.ctot,
                                                                     a.gam, out)));
}

}  // namespace dg
