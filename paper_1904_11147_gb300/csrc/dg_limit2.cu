// 2D limiters on the compacted list of troubled cells (Sec. 3): CSWENO on the subcells of
// the 3 x 3 neighbourhood, and the parent WENO limiter (Qiu and Shu, ref. [qs1]) on the
// (2N+1)^2 whole cells around the troubled one.  Both reconstruct dimension by dimension
// (x sweep of every row, then y sweep at every x point), in characteristic fields at the
// troubled cell's mean for Euler, and project back with the tensor rule (Step 6).
//
//   k_limit2_euler    four lanes per troubled cell (8 cells per warp)
//   k_limit2_burgers  one lane per troubled cell
//
// Bound: the FP64 pipe.  Everything works on differences of neighbouring averages: the
// reconstruction ignores constants, so the cell averages themselves enter only as the value
// the result is added to, and the eigenvector products run on 2N differences instead of
// 2N+1 averages.  Structural zeros of the subcell averages are used (a half of a cell has
// no part of an even mode, a whole cell only that of psi_0), and the arithmetic has the
// three-register form of dg_weno.cuh, whose reconstruction leaves only the smoothness
// indicators to the FP64 pipe (the quotients are formed in integers, too).
//
// Per troubled cell of a 512^2 Euler mesh (half its cells troubled): P2 4.0 ns, P3 8.9 ns.  With FP64
// quotients and dense subcell sums: 5.1 and 11; with the line reconstruction inlined in
// both sweeps: 5.6 and 14; with it wholly in FP64 besides: 7.4 and 16; on averages instead of
// differences, with a reciprocal per stencil: 13 and 28.  The FP64 pipe is busy 82 % (P2) and
// 69 % (P3) of the time; the rest is the latency of the integer chains at 12 to 15 warps per SM.
#include "dg_shared.cuh"
#include "dg_weno.cuh"

namespace dg {
namespace lim2 {

__constant__ double c_lim[2][3][kLimTab];  // [CSWENO, parent][N - 1]

// Index of a row or column beyond the boundary: periodic, or the mirror image.
__device__ __forceinline__ int reflect(int j, int n, int bc) {
  if (bc == 0) {
    j %= n;
    return j < 0 ? j + n : j;
  }
  if (j < 0) j = -1 - j;
  if (j >= n) j = 2 * n - 1 - j;
  return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

// 2x and x/2 on the exponent: three integer instructions instead of an FP64 one of 67 clocks.  With
// the sums that no average needs left out, the subcell averages take 90 (P2) of the 650 FP64
// instructions a lane spent on a troubled cell less (1024^2 P2 step 11.1 -> 10.8 ms, P3 batch of 8 x
// 128 x 512 cells 30.0 -> 28.4 ms).  Numbers within a binade of the largest and the
// smallest normal ones, and non-finite ones, stay as they are: an error of 2^-1021 at most at the
// lower end (see kSmall); at the upper one the smoothness indicators overflow anyway.
__device__ __forceinline__ double exp_add(double x, int d) {
  const unsigned hi = (unsigned)__double2hiint(x), ex = (hi & 0x7ff00000u) - 0x00200000u;
  return __hiloint2double((int)(ex <= 0x7fb00000u ? hi + (unsigned)(d << 20) : hi), __double2loint(x));
}
__device__ __forceinline__ double dbl(double x) { return exp_add(x, 1); }
__device__ __forceinline__ double half(double x) { return exp_add(x, -1); }

// A cell whose data all lie below 2^-959 (exponent word below kSmall) is limited on them times 2^500:
// neither the halves above nor the reconstruction's quotients are exact down there.  The limiter commutes with the factor, since the smoothness indicators are
// far below eps either way.  The two steps it takes are functions that no other cell calls
// (multiplying in place under a condition took 5 to 8 % of the limiter's time).
constexpr unsigned kSmall = 64u << 20;
constexpr double kSmallUp = 0x1p500;

// Where the averages of one troubled cell and one variable go: the 2N x differences of row
// ky (item k between averages k and k + 1) and the row's middle average.
//   diff(ky, k), mid(ky): references into the cell's part of shared memory.
//
// CSWENO: subcell averages of the 3 x 3 neighbourhood.  A neighbour's modes, mirrored in x on
// the right side, give per transverse degree b the N - 1 differences inside it and the
// average next to the troubled cell; the y part then gives them for its N rows.
// Returns the largest exponent word of the modes: the averages of a non-finite state must stay
// non-finite whichever mode holds it.  SMALL: the modes times 2^500.
template <int N, bool SMALL, class Dst>
__device__ __forceinline__ unsigned subcell_diffs(const double* __restrict__ U, long long ctot, const Inst& I, int inst,
                                                  int ix, int iy, int v, int bc, const double* __restrict__ bcd,
                                                  const double* __restrict__ tab, const Reg64& K, Dst dst) {
  using L = LimTab<N>;
  constexpr int NP = np_of(2, N), N1 = N + 1;
  const double* ca = tab + L::CA;
  const double* cr = tab + L::CR;
  unsigned top = 0;
  // middle column first (the row's middle averages), then the outer ones; the rows above
  // and below before the middle one
#pragma unroll 1
  for (int k = 0; k < 9; ++k) {
    const int cx = k / 3, cy = k % 3;
    const int dx = cx == 0 ? 0 : (cx == 1 ? -1 : 1), dy = cy == 0 ? 0 : (cy == 1 ? -1 : 1);
    int jx = ix + dx, jy = iy + dy;
    bool fx = false, fy = false, fv = false;
    const double* cst = nullptr;  // kBcDmr constant ghost
    if (bc == 0) {
      jx = jx < 0 ? jx + I.nx : (jx >= I.nx ? jx - I.nx : jx);
      jy = jy < 0 ? jy + I.ny : (jy >= I.ny ? jy - I.ny : jy);
    } else if (bc == kBcDmr && (jx < 0 || jx >= I.nx || jy < 0 || jy >= I.ny)) {
      const Ghost gh = dmr_ghost(I, inst, jx, jy, bcd, dmr_time(bcd, inst, 0));
      cst = gh.c;
      jx = gh.jx;
      jy = gh.jy;
      fx = gh.fx;
      fy = gh.fy;
      fv = gh.fv && v == 2;
      if (cst) { jx = 0; jy = 0; }
    } else {
      if (jx < 0) { jx = 0; fx = true; }
      if (jx >= I.nx) { jx = I.nx - 1; fx = true; }
      if (jy < 0) { jy = 0; fy = true; }
      if (jy >= I.ny) { jy = I.ny - 1; fy = true; }
    }
    const double* p = U + (long long)(v * NP) * ctot + I.off + (long long)jy * I.nx + jx;
    const bool mx = fx != (dx > 0);  // the right neighbour is read mirrored
    double u[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      double x = __ldg(p + (long long)m * ctot);
      if (cst) x = m == 0 ? 2.0 * cst[v] : 0.0;
      if constexpr (SMALL) x *= kSmallUp;
      u[m] = neg_if(x, ((mx && (mode_a(m) & 1)) != (fy && (mode_b(m) & 1))) != fv);
    }
#pragma unroll
    for (int m = 0; m < NP; ++m) top = max(top, (unsigned)__double2hiint(u[m]) & 0x7fffffffu);
    // x part, times psi_0: q[j][b], j = 0..N-2 the differences inside, j = N-1 the average
    // next to (dx = 0: over) the troubled cell; the middle row has no part of b > 0
    double q[N][N1];
#pragma unroll
    for (int b = 0; b <= N; ++b) {
#pragma unroll
      for (int j = 0; j < N; ++j) q[j][b] = 0.0;
      if (b > 0 && (N == 1 || dy == 0)) continue;
      const double t = half(u[mode_idx(0, b)]);  // psi_0^2 = 1/2
      q[N - 1][b] = t;
      if (N == 1 || b == N || !dx) continue;
      const double u1 = u[mode_idx(1, b < N ? b : 0)];
      if constexpr (N == 2) {  // halves
        const double s = K.mul(ca[1], u1);
        q[0][b] = dbl(s);
        q[1][b] = K.add(t, s);
      } else if constexpr (N == 3) {  // thirds: even part u0 / 2 + ca2 u2 (middle third u0 / 2 - 2 ca2 u2), odd part ca1 u1 + ca3 u3
        const double od = b == 0 ? fma(ca[3], u[mode_idx(3, 0)], K.mul(ca[1], u1)) : K.mul(ca[1], u1);
        if (b <= 1) {
          const double e = K.mul(ca[2], u[mode_idx(2, b <= 1 ? b : 0)]), e3 = K.add(e, dbl(e));
          q[0][b] = K.sub(od, e3);
          q[1][b] = K.add(od, e3);
          q[2][b] = K.add(t, K.add(e, od));
        } else {
          q[0][b] = q[1][b] = od;
          q[2][b] = K.add(t, od);
        }
      }
    }
    // y part: rows r = 0..N-1 of the neighbour (dy = 0: the middle row)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (j < N - 1 && !dx) continue;
      double val[N];
      if (dy == 0) {
        val[0] = q[j][0];
      } else if constexpr (N == 1) {
        val[0] = q[0][0];
      } else if constexpr (N == 2) {
        val[0] = fma(-cr[1], q[j][1], q[j][0]);
        val[1] = fma(cr[1], q[j][1], q[j][0]);
      } else {
        const double e = fma(cr[2], q[j][2], q[j][0]), t = K.mul(cr[2], q[j][2]);
        const double od = j == 2 ? fma(cr[3], q[j][3], K.mul(cr[1], q[j][1])) : K.mul(cr[1], q[j][1]);
        val[0] = K.sub(e, od);
        val[2] = K.add(e, od);
        val[1] = K.sub(q[j][0], dbl(t));
      }
      const int row0 = dy == 0 ? N : (dy < 0 ? 0 : N + 1);
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (dy == 0 && r) break;
        const int ky = row0 + r;
        if (!dx) {
          dst.mid(ky) = val[r];
        } else if (j < N - 1) {
          // right neighbour: mirrored, so its differences come in reverse order and sign
          if (dx < 0) dst.diff(ky, j) = val[r];
          else dst.diff(ky, 2 * N - 1 - j) = -val[r];
        } else {
          const double c = dst.mid(ky);
          if (dx < 0) dst.diff(ky, N - 1) = K.sub(c, val[r]);
          else dst.diff(ky, N) = K.sub(val[r], c);
        }
      }
    }
  }
  return top;
}

// Parent WENO: means of the whole cells (ix - N .. ix + N) x (iy - N .. iy + N).
template <int N, bool SMALL, class Dst>
__device__ __forceinline__ unsigned cell_diffs(const double* __restrict__ U, long long ctot, const Inst& I, int ix,
                                               int iy, int v, int bc, const double* __restrict__ tab, const Reg64& K,
                                               Dst dst) {
  using L = LimTab<N>;
  unsigned top = 0;
  const double* p = U + (long long)(v * np_of(2, N)) * ctot + I.off;
  const double p0 = tab[L::P0];
#pragma unroll 1
  for (int ky = 0; ky < 2 * N + 1; ++ky) {
    const double* row = p + (long long)reflect(iy + ky - N, I.ny, bc) * I.nx;
    double prev = 0.0;
#pragma unroll
    for (int kx = 0; kx < 2 * N + 1; ++kx) {
      double x = __ldg(row + reflect(ix + kx - N, I.nx, bc));
      if constexpr (SMALL) x *= kSmallUp;
      top = max(top, (unsigned)__double2hiint(x) & 0x7fffffffu);
      const double a = K.mul(K.mul(x, p0), p0);
      if (kx) dst.diff(ky, kx - 1) = K.sub(a, prev);
      if (kx == N) dst.mid(ky) = a;
      prev = a;
    }
  }
  return top;
}

// The differences of listed cell g, variable v
template <int N, bool PARENT, bool SMALL, class Dst>
__device__ __forceinline__ unsigned stencil_diffs(const double* __restrict__ U, const Inst* __restrict__ insts,
                                                  long long ctot, int bc, long long g, int inst, int v,
                                                  const double* __restrict__ bcd, const double* __restrict__ tab,
                                                  const Reg64& K, Dst dst) {
  const Inst I = insts[inst];
  const int loc = (int)(g - I.off);
  const int ix = loc % I.nx, iy = loc / I.nx;
  if constexpr (PARENT) return cell_diffs<N, SMALL>(U, ctot, I, ix, iy, v, bc, tab, K, dst);
  else return subcell_diffs<N, SMALL>(U, ctot, I, inst, ix, iy, v, bc, bcd, tab, K, dst);
}
template <int N, bool PARENT, class Dst>
__device__ __noinline__ void stencil_diffs_small(const double* __restrict__ U, const Inst* __restrict__ insts,
                                                 long long ctot, int bc, long long g, int inst, int v,
                                                 const double* __restrict__ bcd, const double* __restrict__ tab, Dst dst) {
  const Reg64 K{tab[LimTab<N>::ONE], tab[LimTab<N>::NZ]};
  stencil_diffs<N, PARENT, true>(U, insts, ctot, bc, g, inst, v, bcd, tab, K, dst);
}
// the limited modes 1..NP-1 of a variable back to their size
template <int N>
__device__ __noinline__ void unscale_small(double* __restrict__ lim, long long cap) {
  for (int m = 1; m < np_of(2, N); ++m) lim[m * cap] *= 1.0 / kSmallUp;
}

// Eigenvector products of the 2D Euler flux Jacobian at the troubled cell's mean state,
// direction with normal velocity vn and tangential velocity vt.
struct Eig {
  double vx, vy, hq2, c, ic, H, b1;  // hq2 = |v|^2 / 2, b1 = (gamma - 1) / c^2
};
__device__ __forceinline__ Eig euler_eig(const double (&m)[4], double gam, const Reg64& K) {
  Eig e;
  const double gm1 = gam - 1.0;
  const double r = rcp_d(m[0]);
  e.vx = K.mul(m[1], r);
  e.vy = K.mul(m[2], r);
  e.hq2 = 0.5 * fma(e.vx, e.vx, K.mul(e.vy, e.vy));
  const double p = gm1 * fma(-m[0], e.hq2, m[3]);
  e.c = sqrt_d(gam * p * r);
  e.ic = rcp_d(e.c);
  e.H = K.mul(K.add(m[3], p), r);
  e.b1 = gm1 * e.ic * e.ic;
  return e;
}
// characteristic differences w = L u of (rho, normal momentum, tangential momentum, E)
__device__ __forceinline__ void to_char(const Eig& e, double vn, double vt, double hic, double hb1, double rho, double mn,
                                        double mt, double E, const Reg64& K, double (&w)[4]) {
  const double s = fma(-vt, mt, fma(-vn, mn, fma(e.hq2, rho, E)));  // (gamma-1) s = pressure difference
  const double a = K.mul(hb1, s), d = fma(-vn, rho, mn);
  w[0] = fma(-hic, d, a);
  w[1] = fma(-e.b1, s, rho);
  w[2] = fma(-vt, rho, mt);
  w[3] = fma(hic, d, a);
}
// conserved values R w
__device__ __forceinline__ void from_char(const Eig& e, double vn, double vt, const double (&w)[4], const Reg64& K,
                                          double& rho, double& mn, double& mt, double& E) {
  const double s = K.add(w[0], w[3]), t = K.mul(e.c, K.sub(w[3], w[0]));
  rho = K.add(s, w[1]);
  mn = fma(vn, rho, t);
  mt = fma(vt, rho, w[2]);
  E = fma(e.H, s, fma(vn, t, fma(e.hq2, w[1], K.mul(vt, w[2]))));
}

// The reconstruction of one line: 2N differences p[k stride] in shared memory, replaced by the
// values at the Step 1 points.  One copy for both sweeps: it is most of the kernel's code, and
// inlined twice it ran out of the instruction cache (1024^2 P2 step 13.3 -> 12.5 ms, P3 batch of
// 8 x 128 x 512 cells 37.5 -> 33.1 ms per step).  One lane per cell (Burgers) gains nothing from it.
template <int N, bool SPLIT>
__device__ __noinline__ void weno_line(double* p, int stride, const double* __restrict__ tab) {
  using L = LimTab<N>;
  const Reg64 K{tab[L::ONE], tab[L::NZ]};
  double d[2 * N], r[L::NG];
#pragma unroll
  for (int k = 0; k < 2 * N; ++k) d[k] = p[k * stride];
  weno_diff<N, SPLIT>(d, tab, K, r);
#pragma unroll
  for (int k = 0; k < L::NG; ++k) p[k * stride] = r[k];
}

// CSWENO or parent limiter for 2D Euler, four lanes per troubled cell: the list is often
// short (a few cells per SM sub-partition), and a cell's work has four-way parallelism at
// each step.  Lane q of a quad owns
//   conserved variable q            for the averages,
//   every fourth difference         for the products with the left eigenvectors (all four
//                                   variables of one difference: 9 instructions instead of 16),
//   characteristic field q          for the x sweep's rows,
//   x point q                       from there on: the right eigenvectors, the whole y sweep
//                                   of its column and the projection in y,
//   conserved variable q            for the projection in x.
// Values change owner through shared memory: per cell rows ky of 2N+1 items of 4 doubles
// (the 2N differences and, as item 2N, the middle averages).  The rows of all passes reuse
// the same items: a lane only overwrites values that it alone reads.
// A cell's items are 4 (mod 16) doubles apart: the 16 lanes of half a warp hit 32 banks.
// With a work counter (lq, zero at launch) a warp takes its next 8 cells from it, so the
// work spreads over the resident warps whatever the grid.
constexpr int kQuadThreads = 64;
// Blocks per SM.  P3: 6 (168 registers) 31.9 ms per step of the batch above, 5 33.1, 8 32.5; P2: 8
// (128 registers) 12.2 ms per 1024^2 step, 6 12.4.  P1 needs fewer registers than either allows.
__host__ __device__ constexpr int quad_blocks(int N) { return N == 3 ? 6 : 8; }

template <int N, bool PARENT>
__global__ void __launch_bounds__(kQuadThreads, quad_blocks(N))
    k_limit2_euler(const double* __restrict__ U, const Inst* __restrict__ insts, long long ctot, int bc,
                   const int* __restrict__ list_cell, const int* __restrict__ list_inst,
                   const Counters* __restrict__ cnt, double* __restrict__ lim, long long cap, double gam,
                   unsigned int* __restrict__ lq, const double* __restrict__ bcd) {
  using L = LimTab<N>;
  constexpr int NP = np_of(2, N), NS = 2 * N + 1, NG = L::NG, N1 = N + 1;
  constexpr int ROW = NS * 4, CELL = NS * ROW;
  static_assert(CELL % 16 == 4, "bank-conflict-free cell stride");
  constexpr bool SPLIT = N == 3 && !PARENT;
  __shared__ __align__(16) double tab[L::SIZE];
  __shared__ __align__(16) double buf[kQuadThreads / 4 * CELL];
  const unsigned int n = cnt->n_flag;
  if (blockIdx.x * (kQuadThreads / 4) >= n) return;  // whole blocks without a cell leave at once
  for (int k = threadIdx.x; k < L::SIZE; k += kQuadThreads) tab[k] = c_lim[PARENT][N - 1][k];
  __syncthreads();
  const Reg64 K{tab[L::ONE], tab[L::NZ]};
  const int lane = threadIdx.x & 31, q = lane & 3;
  const unsigned int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const unsigned int nwarps = (gridDim.x * blockDim.x) >> 5;
  double* const S = buf + (threadIdx.x >> 2) * CELL;
  struct Dst {
    double* S;
    int q;
    __device__ __forceinline__ double& diff(int ky, int k) const { return S[ky * ROW + 4 * k + q]; }
    __device__ __forceinline__ double& mid(int ky) const { return S[ky * ROW + 8 * N + q]; }
  };
  for (unsigned int it = 0;; ++it) {
    unsigned int base;
    if (lq) {
      unsigned int b0 = 0;
      if (lane == 0) b0 = atomicAdd(lq, 8u);
      base = __shfl_sync(0xffffffffu, b0, 0);
    } else {
      base = (warp + it * nwarps) * 8u;
    }
    if (base >= n) break;
    const unsigned int i0 = base + (lane >> 2);
    const bool active = i0 < n;
    const unsigned int i = active ? i0 : n - 1;  // idle quads repeat a valid entry
    const long long g = list_cell[i];
    const int inst = list_inst[i];
    Eig e;
    const unsigned quad = 0xfu << (lane & ~3);
    const unsigned top = stencil_diffs<N, PARENT, false>(U, insts, ctot, bc, g, inst, q, bcd, tab, K, Dst{S, q});
    const bool bad = !PARENT && __any_sync(quad, top >= 0x7ff00000u);
    const bool small = __all_sync(quad, top < kSmall);
    if (small) stencil_diffs_small<N, PARENT>(U, insts, ctot, bc, g, inst, q, bcd, tab, Dst{S, q});
    __syncwarp();
    {
      double m[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) m[v] = S[N * ROW + 8 * N + v];
      e = euler_eig(m, gam, K);
    }
    const double hic = 0.5 * e.ic, hb1 = 0.5 * e.b1;
    // left eigenvectors of the x direction
#pragma unroll 1
    for (int k = q; k < NS * 2 * N; k += 4) {
      double* p = S + (k / (2 * N)) * ROW + (k % (2 * N)) * 4;
      double w[4];
      to_char(e, e.vx, e.vy, hic, hb1, p[0], p[1], p[2], p[3], K, w);
#pragma unroll
      for (int f = 0; f < 4; ++f) p[f] = w[f];
    }
    __syncwarp();
    // x sweep: field q of every row; point values replace the differences
#pragma unroll 1
    for (int ky = 0; ky < NS; ++ky) weno_line<N, SPLIT>(S + ky * ROW + q, 4, tab);
    __syncwarp();
    double mid[4];  // the middle row's averages at x point q
    if (q < NG) {
      // back to conserved variables at x point q; y differences to characteristic fields
      double prev[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
      for (int ky = 0; ky < NS; ++ky) {
        double w[4], u[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) w[f] = S[ky * ROW + 4 * q + f];
        from_char(e, e.vx, e.vy, w, K, u[0], u[1], u[2], u[3]);
#pragma unroll
        for (int v = 0; v < 4; ++v) u[v] = K.add(u[v], S[ky * ROW + 8 * N + v]);
        if (ky) {
          double dv[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) dv[v] = K.sub(u[v], prev[v]);
          to_char(e, e.vy, e.vx, hic, hb1, dv[0], dv[2], dv[1], dv[3], K, w);
#pragma unroll
          for (int f = 0; f < 4; ++f) S[(ky - 1) * ROW + 4 * q + f] = w[f];
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          prev[v] = u[v];
          if (ky == N) mid[v] = u[v];
        }
      }
      // y sweep of the column, projected in y: t_b = sum_g w_g psi_b(y_g) (u(y_g) - mid)
#pragma unroll 1
      for (int f = 0; f < 4; ++f) {
        double r[NG];
        weno_line<N, SPLIT>(S + 4 * q + f, ROW, tab);
#pragma unroll
        for (int k = 0; k < NG; ++k) r[k] = S[k * ROW + 4 * q + f];
        double sp[NG / 2], sm[NG / 2];  // the points are symmetric, psi_b has the parity of b
#pragma unroll
        for (int k = 0; k < NG / 2; ++k) {
          sp[k] = K.add(r[k], r[NG - 1 - k]);
          sm[k] = K.sub(r[k], r[NG - 1 - k]);
        }
#pragma unroll
        for (int b = 0; b <= N; ++b) {
          double t = 0.0;
#pragma unroll
          for (int k = 0; k < NG / 2; ++k) {
            const double x = (b & 1) ? sm[k] : sp[k], c = tab[L::PG + k * N1 + b];
            t = k == 0 ? K.mul(c, x) : fma(c, x, t);
          }
          S[b * ROW + 4 * q + f] = t;
        }
      }
#pragma unroll 1
      for (int b = 0; b <= N; ++b) {
        double w[4], u[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) w[f] = S[b * ROW + 4 * q + f];
        from_char(e, e.vy, e.vx, w, K, u[0], u[2], u[1], u[3]);
#pragma unroll
        for (int v = 0; v < 4; ++v) S[b * ROW + 4 * q + v] = b == 0 ? fma(tab[L::PG0], mid[v], u[v]) : u[v];
      }
    }
    __syncwarp();
    // projection in x of variable q: U_ab = sum_g w_g psi_a(x_g) t_b(x_g)
#pragma unroll
    for (int b = 0; b <= N; ++b) {
      double t[NG];
#pragma unroll
      for (int k = 0; k < NG; ++k) t[k] = S[b * ROW + 4 * k + q];
#pragma unroll
      for (int a = b == 0 ? 1 : 0; a <= N - b; ++a) {
        double s = K.mul(tab[L::PG + a], t[0]);
#pragma unroll
        for (int k = 1; k < NG; ++k) s = fma(tab[L::PG + k * N1 + a], t[k], s);
        if (bad) s = __longlong_as_double(0x7ff8000000000000LL);
        if (active) lim[(long long)(q * NP + mode_idx(a, b)) * cap + i] = s;
      }
    }
    if (small && active) unscale_small<N>(lim + (long long)(q * NP) * cap + i, cap);
    __syncwarp();  // the next cell's averages overwrite the items
  }
}

// The same for Burgers, one lane per troubled cell (one variable: nothing to exchange); the
// rows live in shared memory, one column per lane.
constexpr int kCellThreads = 64;

template <int N, bool PARENT>
__global__ void __launch_bounds__(kCellThreads)
    k_limit2_burgers(const double* __restrict__ U, const Inst* __restrict__ insts, long long ctot, int bc,
                     const int* __restrict__ list_cell, const int* __restrict__ list_inst,
                     const Counters* __restrict__ cnt, double* __restrict__ lim, long long cap) {
  using L = LimTab<N>;
  constexpr int NP = np_of(2, N), NS = 2 * N + 1, NG = L::NG, N1 = N + 1;
  constexpr int ROW = NS * kCellThreads;
  constexpr bool SPLIT = N == 3 && !PARENT;
  __shared__ __align__(16) double tab[L::SIZE];
  __shared__ double buf[NS * ROW];
  const unsigned int n = cnt->n_flag;
  if (blockIdx.x * kCellThreads >= n) return;
  for (int k = threadIdx.x; k < L::SIZE; k += kCellThreads) tab[k] = c_lim[PARENT][N - 1][k];
  __syncthreads();
  const Reg64 K{tab[L::ONE], tab[L::NZ]};
  double* const S = buf + threadIdx.x;
  struct Dst {
    double* S;
    __device__ __forceinline__ double& diff(int ky, int k) const { return S[ky * ROW + k * kCellThreads]; }
    __device__ __forceinline__ double& mid(int ky) const { return S[ky * ROW + 2 * N * kCellThreads]; }
  };
  const Dst A{S};
  for (unsigned int i = blockIdx.x * kCellThreads + threadIdx.x; i < n; i += gridDim.x * kCellThreads) {
    const long long g = list_cell[i];
    const int inst = list_inst[i];
    const unsigned top = stencil_diffs<N, PARENT, false>(U, insts, ctot, bc, g, inst, 0, nullptr, tab, K, A);
    const bool bad = !PARENT && top >= 0x7ff00000u, small = top < kSmall;
    if (small) stencil_diffs_small<N, PARENT>(U, insts, ctot, bc, g, inst, 0, nullptr, tab, A);
#pragma unroll 1
    for (int ky = 0; ky < NS; ++ky) {
      double d[2 * N], r[NG];
#pragma unroll
      for (int k = 0; k < 2 * N; ++k) d[k] = A.diff(ky, k);
      weno_diff<N, SPLIT>(d, tab, K, r);
#pragma unroll
      for (int k = 0; k < NG; ++k) A.diff(ky, k) = K.add(r[k], A.mid(ky));
    }
    double acc[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) acc[m] = 0.0;
#pragma unroll 1
    for (int gx = 0; gx < NG; ++gx) {
      double d[2 * N], r[NG];
      double prev = A.diff(0, gx);
#pragma unroll
      for (int k = 0; k < 2 * N; ++k) {
        const double x = A.diff(k + 1, gx);
        d[k] = K.sub(x, prev);
        prev = x;
      }
      weno_diff<N, SPLIT>(d, tab, K, r);
      const double mid = A.diff(N, gx);
      double sp[NG / 2], sm[NG / 2];
#pragma unroll
      for (int k = 0; k < NG / 2; ++k) {
        sp[k] = K.add(r[k], r[NG - 1 - k]);
        sm[k] = K.sub(r[k], r[NG - 1 - k]);
      }
#pragma unroll
      for (int b = 0; b <= N; ++b) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < NG / 2; ++k) {
          const double x = (b & 1) ? sm[k] : sp[k], c = tab[L::PG + k * N1 + b];
          t = k == 0 ? K.mul(c, x) : fma(c, x, t);
        }
        if (b == 0) t = fma(tab[L::PG0], mid, t);
#pragma unroll
        for (int a = b == 0 ? 1 : 0; a <= N - b; ++a)
          acc[mode_idx(a, b)] = fma(tab[L::PG + gx * N1 + a], t, acc[mode_idx(a, b)]);
      }
    }
#pragma unroll
    for (int m = 1; m < NP; ++m)
      lim[(long long)m * cap + i] = bad ? __longlong_as_double(0x7ff8000000000000LL) : acc[m];
    if (small) unscale_small<N>(lim + i, cap);
  }
}

template <int N, bool PARENT>
void launch(int pde, const LaunchArgs& a, const int* lc, const int* li, const Counters* cnt, double* lim, int nblocks) {
  // nblocks counts blocks of 128 threads
  if (pde == 1) {
    if (a.lq) cudaMemsetAsync(a.lq, 0, sizeof(unsigned int), a.st);
    k_limit2_euler<N, PARENT><<<nblocks * (128 / kQuadThreads), kQuadThreads, 0, a.st>>>(
        a.us, a.inst, a.ctot, a.bc, lc, li, cnt, lim, a.cap, a.gam, a.lq, a.bcd);
  } else {
    k_limit2_burgers<N, PARENT><<<nblocks * (128 / kCellThreads), kCellThreads, 0, a.st>>>(
        a.us, a.inst, a.ctot, a.bc, lc, li, cnt, lim, a.cap);
  }
}

}  // namespace lim2

// tabs, ptabs: [3] for N = 1..3, CSWENO and parent
cudaError_t upload_tables_lim2(const dgt::Tabs* tabs, const dgt::Tabs* ptabs) {
  static double h[2][3][kLimTab];
  for (int k = 0; k < 2; ++k) {
    const dgt::Tabs* t = k ? ptabs : tabs;
    pack_lim<1>(t[0], h[k][0]);
    pack_lim<2>(t[1], h[k][1]);
    pack_lim<3>(t[2], h[k][2]);
  }
  return cudaMemcpyToSymbol(lim2::c_lim, h, sizeof(h));
}

void launch_limit2(int pde, int N, const LaunchArgs& a, const int* lc, const int* li, const Counters* cnt, double* lim,
                   int nblocks) {
  if (N == 1) lim2::launch<1, false>(pde, a, lc, li, cnt, lim, nblocks);
  else if (N == 2) lim2::launch<2, false>(pde, a, lc, li, cnt, lim, nblocks);
  else lim2::launch<3, false>(pde, a, lc, li, cnt, lim, nblocks);
}

void launch_parent2(int pde, int N, const LaunchArgs& a, const int* lc, const int* li, const Counters* cnt, double* lim,
                    int nblocks) {
  if (N == 1) lim2::launch<1, true>(pde, a, lc, li, cnt, lim, nblocks);
  else if (N == 2) lim2::launch<2, true>(pde, a, lc, li, cnt, lim, nblocks);
  else lim2::launch<3, true>(pde, a, lc, li, cnt, lim, nblocks);
}

}  // namespace dg
