// Split 2D stage of Eq. (5), two passes without halo work:
//   k_face2  one thread per face: the traces of the two cells at the Q face points, the
//            local Lax-Friedrichs flux there, and its projection onto the transverse modes
//              P_b = sum_q w_q psi_b(s_q) [f(uL) + f(uR) - alpha (uR - uL)],  b = 0..N,
//            stored in planes [v*(N+1) + b][face] (x faces and y faces apart);
//   k_cell2  one thread per cell: the volume term, the lifting of the four faces' P_b and
//            the stage combination.
// Every face flux is computed once; all lanes of every warp do the same work.
//
// Bound: the FP64 pipe.  Traces and volume point values are linear in the modes: they are
// formed in fixed point on the integer pipes (dg_weno.cuh), over psi_0 = 1/sqrt(2) and doubled
// (2 sum_t (e_t / psi_0) psi_t(s) psi_0 = e_0 + sum_{t>=1} e_t sqrt(2) psi_t(s)); the fluxes are homogeneous in the state (Euler of degree 1,
// Burgers of degree 2), so the factor is taken back in the final scalings.  The Gauss points
// are symmetric and psi_t has the parity of t: sums and differences over pairs of points.
// Every quadrature sum is kept relative to its outermost weight (one product less), and all
// those factors, 2/h, the time step and the stage's weight go into one set of constants per
// block.  The density's volume term needs no quadrature: its flux is the momentum, a
// polynomial.  Arithmetic in the three-register form of dg_weno.cuh.
//
// Measured per launch (Euler; in parentheses with the traces and point values in FP64, and
// before that with plain sums and products, constant operands, products with every weight and
// 32-wide face tiles): 1024^2 P2 face pass 0.70 ms (0.87, 1.09), cell pass 0.81 ms (0.88,
// 1.19); P3 batch of 1.10 M cells 1.04 ms (1.46, 1.84) and 1.98 ms (1.98, 3.18); 1537 x 1021 P1
// 0.68 ms (0.80, 1.02) and 0.44 ms (0.44, 0.66).  With the traces in one function the face pass is
// 8 % (P2) and 16 % (P3) faster still: 512^2 0.18 and 0.25 ms, the FP64 pipe 84 % busy.
#include <cmath>
#include <cstring>

#include "dg_shared.cuh"
#include "dg_weno.cuh"

namespace dg {
namespace st2 {

template <int N>
struct STab {
  static constexpr int N1 = N + 1, Q = N + 1, NP = (N + 1) * (N + 2) / 2, NX = (Q + 1) / 2;
  // constants
  static constexpr int ONE = 0, NZ = 1, C38 = 2, HALF = 3;
  static constexpr int GM1 = 4, HGM1 = 5, SG = 6;   // gamma - 1, -(gamma - 1) / 2, sqrt(gamma) (set by the block)
  static constexpr int RA = 7, RB = 8;              // weights of u^n and of the stage's input (set by the block)
  static constexpr int KP1 = 9;                     // [N1] sqrt(2) psi_n(1) 2^61 (integers)
  static constexpr int KQ = KP1 + N1;               // [NX][N1] sqrt(2) psi_n(x_q) 2^62, x_q <= 0 (integers)
  static constexpr int KD = KQ + NX * N1;           // [NX][N1] sqrt(2) psi_n(x_q) in FP64
  static constexpr int KAP = KD + NX * N1;          // [N1] w psi_b at the second point over the first
  static constexpr int KAD = KAP + N1;              // [N1] w psi_b' at the second point over the first
  // times (2/hx) dt times the stage's weight times 2^-d
  static constexpr int XF = KAD + N1;
  static constexpr int CX = XF;                     // [NX][NP] volume, x derivative: w psi_a'(x_p) times the y sum's factor
  static constexpr int LX = CX + NX * NP;           // [NP] lifting of the x faces
  static constexpr int DX = LX + NP;                // [4] density: integrals psi_1' psi_0, psi_2' psi_1, psi_3' psi_2, psi_3' psi_0
  // the same for y
  static constexpr int YF = DX + 4;
  static constexpr int CY = YF;
  static constexpr int LY = CY + NX * NP;
  static constexpr int DY = LY + NP;
  static constexpr int SIZE = (DY + 4 + 1) / 2 * 2;
  static constexpr int FACE = (XF + 1) / 2 * 2;     // the part the face pass needs
};
constexpr int kSTab = STab<3>::SIZE;
constexpr int kFaceChunk = 128, kCellChunk = 256;  // faces, cells per block

__device__ double g_stab[3][kSTab];

template <int N>
void pack(const dgt::Tabs& t, double* h) {
  using S = STab<N>;
  constexpr int N1 = S::N1, Q = S::Q, NP = S::NP, NX = S::NX;
  h[S::ONE] = 1.0;
  h[S::NZ] = -0.0;
  h[S::C38] = 0.375;
  h[S::HALF] = 0.5;
  auto put = [&](int k, long long i) { std::memcpy(h + k, &i, sizeof(i)); };
  auto wp = [&](int q, int b) { return t.gw[q] * t.psi_q[q][b]; };
  auto wd = [&](int q, int b) { return t.gw[q] * t.dpsi_q[q][b]; };
  for (int n = 0; n < N1; ++n) {
    put(S::KP1 + n, t.kp1_fix[n]);
    for (int q = 0; q < NX; ++q) {
      put(S::KQ + q * N1 + n, t.kq_fix[q][n]);
      h[S::KD + q * N1 + n] = t.kq[q][n];
    }
    h[S::KAP + n] = wp(1, n) / wp(0, n);
    h[S::KAD + n] = n ? wd(1, n) / wd(0, n) : 0.0;
  }
  for (int m = 0; m < NP; ++m) {
    const int a = mode_a(m), b = mode_b(m);
    for (int p = 0; p < NX; ++p) {
      h[S::CX + p * NP + m] = wd(p, a) * wp(0, b);
      h[S::CY + p * NP + m] = wp(p, a) * wd(0, b);
    }
    h[S::LX + m] = -0.5 * t.psi_p1[a] * wp(0, b);
    h[S::LY + m] = -0.5 * t.psi_p1[b] * wp(0, a);
  }
  // integral of psi_a' psi_k (exact with the Gauss rule), times 2: of the undoubled momentum
  auto dpk = [&](int a, int k) {
    double s = 0.0;
    for (int q = 0; q < Q; ++q) s += wd(q, a) * t.psi_q[q][k];
    return 2.0 * s;
  };
  const double d[4] = {dpk(1, 0), N >= 2 ? dpk(2, 1) : 0.0, N >= 3 ? dpk(3, 2) : 0.0, N >= 3 ? dpk(3, 0) : 0.0};
  for (int k = 0; k < 4; ++k) h[S::DX + k] = h[S::DY + k] = d[k];
}

// y sums relative to the outermost weight, psi_b (or psi_b') of even parity: over S = sums of
// symmetric pairs (and the middle point), of odd parity: over D = differences
template <int N>
__device__ __forceinline__ double rel_sum(bool even, const double (&S)[(N + 1) / 2], const double (&D)[(N + 1) / 2],
                                          double mid, double kap) {
  if constexpr (N == 1) return even ? S[0] : D[0];
  else if constexpr (N == 2) return even ? fma(kap, mid, S[0]) : D[0];
  else return even ? fma(kap, S[1], S[0]) : fma(kap, D[1], D[0]);
}

// Velocities, pressure and reciprocal density of a 2D Euler state (m1, m2: momentum).
__device__ __forceinline__ void euler_state(double rho, double m1, double m2, double E, const double* __restrict__ c,
                                            int gm1, int hgm1, const Reg64& K, double& r, double& v1, double& v2,
                                            double& p) {
  r = rcp_k(rho, K);
  v1 = K.mul(m1, r);
  v2 = K.mul(m2, r);
  p = fma(c[hgm1], fma(m1, v1, K.mul(m2, v2)), K.mul(c[gm1], E));  // (gamma-1)(E - rho |v|^2 / 2)
}

// Tiles: chunk Tile::x0 of kFaceChunk faces of the instance, row by row; Tile::pad = 0 for x
// faces (k = 0..nx, j < ny), 1 for y faces (k < nx, j = 0..ny).  Face k of a row lies between
// cells k-1 and k.  (Chunks of the face index instead of 32-wide tiles: a row of nx + 1 faces
// left most lanes of its last warp idle, 6 % of all warps at nx = 512.)
// FP64 instructions per face (Euler): 104, 166, 226 for P1, P2, P3.
template <int N>
struct TraceVal {
  double v[N + 1];
};

// The doubled traces of one variable at the Q points of a face: p its plane of mode 0 at the cell,
// fn and ft: modes of odd normal or transverse degree negated, wall: the whole variable negated.
// One copy for both sides and all variables: inlined eight times it waited for instructions (2.1 of
// some 14 cycles per instruction; two P2 steps of 512^2 cells, few of them troubled, 3.95 ->
// 3.87 ms, one step of 960 x 240 cells 1.60 -> 1.56 ms).
template <int N>
__device__ __noinline__ TraceVal<N> trace(const double* __restrict__ p, long long ctot, int dir, bool fn, bool ft, bool wall,
                                          const double* cst, const long long* __restrict__ itab) {
  using T = STab<N>;
  constexpr int NP = np_of(2, N), Q = N + 1, N1 = N + 1;
  TraceVal<N> o;
  double u[NP];
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    const int n = mode_a(m), t = mode_b(m);
    const int pm = dir ? mode_idx(t, n) : m;
    double x = __ldg(p + (long long)pm * ctot);
    if (cst) x = m == 0 ? 2.0 * *cst : 0.0;  // constant state: U_00 = 2 mean, no other mode
    u[m] = neg_if(x, ((fn && (n & 1)) != (ft && (t & 1))) != wall);
  }
  // sums over the normal degree in units of 8 X, then at the points.  Below 2^62.5 all of them: X
  // below 2^63, 2^62, 2^61, sum_t |KQ_t| sum_{n <= N-t} |KP1_n| = 3.7, 9.5, 19.6 and 4 |e_1| / |X| at most
  // 1/2, 1.37, 2.49 for N = 1, 2, 3.
  constexpr int F = 11 - N;
  long long X[NP], e[N1], val[Q];
  const int E = align_modes<NP, F, 3>(u, X);
#pragma unroll
  for (int t = 0; t <= N; ++t) {
    long long z = X[mode_idx(0, t)] >> 3;
#pragma unroll
    for (int n = 1; n <= N - t; ++n) z += mul_rn(itab[T::KP1 + n], X[mode_idx(n, t)]);
    e[t] = z;
  }
  eval_fix<N>(e, itab + T::KQ, val);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    o.v[q] = E < 2047 ? pack_s64<true>(val[q], E - 1072 - F) : __longlong_as_double(0x7ff8000000000000LL);
  return o;
}

template <int PDE, int N>
__global__ void __launch_bounds__(kFaceChunk) k_face2(const double* __restrict__ us, const Inst* __restrict__ insts,
                                               const Tile* __restrict__ tiles, long long ctot, int bc, Gamma gm,
                                               double* __restrict__ fx, long long fxt, double* __restrict__ fy,
                                               long long fyt, const double* __restrict__ bcd, int stage,
                                               double dt_all) {
  using T = STab<N>;
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N), Q = N + 1, N1 = N + 1;
  __shared__ __align__(16) double tab[T::FACE];
  if (threadIdx.x < T::XF) {
    const int k = threadIdx.x;
    double x = g_stab[N - 1][k];
    if (k == T::GM1) x = gm.gm1;
    if (k == T::HGM1) x = gm.hgm1;
    if (k == T::SG) x = gm.sg;
    tab[k] = x;
  }
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  const int dir = tile.pad;
  const unsigned face = (unsigned)tile.x0 * kFaceChunk + threadIdx.x, row = (unsigned)I.nx + (dir == 0);
  const int j = (int)(face / row), k = (int)(face - (unsigned)j * row);
  __syncthreads();
  if (j >= I.ny + dir) return;
  const Reg64 K{tab[T::ONE], tab[T::NZ]};
  const long long* itab = reinterpret_cast<const long long*>(tab);
  // variables in the order (rho, normal momentum, tangential momentum, E) and modes by
  // (normal degree n, transverse degree t): the planes are read in that order
  double tr[2][Q][V];
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    int ix = dir == 0 && side == 0 ? k - 1 : k, iy = dir == 1 && side == 0 ? j - 1 : j;
    bool fX = false, fY = false, fv = false;
    const double* cst = nullptr;
    if (ix < 0 || ix >= I.nx || iy < 0 || iy >= I.ny) {
      if (bc == 0) {  // periodic
        ix = ix < 0 ? ix + I.nx : (ix >= I.nx ? ix - I.nx : ix);
        iy = iy < 0 ? iy + I.ny : (iy >= I.ny ? iy - I.ny : iy);
      } else if (bc == kBcDmr) {
        // the stage's input holds at t^n, t^n + dt, t^n + dt/2 for stages 1, 2, 3
        const double t_in = dmr_time(bcd, tile.inst, 2) +
                            (stage == 1 ? 0.0 : (stage == 2 ? 1.0 : 0.5)) * (dt_all > 0.0 ? dt_all : I.dt);
        const Ghost gh = dmr_ghost(I, tile.inst, ix, iy, bcd, t_in);
        cst = gh.c;
        ix = gh.c ? 0 : gh.jx;
        iy = gh.c ? 0 : gh.jy;
        fX = gh.fx;
        fY = gh.fy;
        fv = gh.fv;
      } else {  // outflow: the boundary cell mirrored
        if (ix < 0) { ix = 0; fX = true; }
        if (ix >= I.nx) { ix = I.nx - 1; fX = true; }
        if (iy < 0) { iy = 0; fY = true; }
        if (iy >= I.ny) { iy = I.ny - 1; fY = true; }
      }
    }
    // the trace on the right cell's -1 side: modes of odd normal degree negated
    const bool fn = (dir == 0 ? fX : fY) != (side == 1), ft = dir == 0 ? fY : fX;
    const double* p = us + I.off + (long long)iy * I.nx + ix;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int pv = (V == 4 && (v == 1 || v == 2) && dir) ? 3 - v : v;
      const bool wall = fv && pv == 2;
      const TraceVal<N> o = trace<N>(p + (long long)pv * NP * ctot, ctot, dir, fn, ft, wall, cst ? cst + pv : nullptr, itab);
#pragma unroll
      for (int q = 0; q < Q; ++q) tr[side][q][v] = o.v[q];
    }
  }
  double G[Q][V];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const double* L = tr[0][q];
    const double* R = tr[1][q];
    if constexpr (PDE == 0) {
      // f(uL) + f(uR) - alpha (uR - uL) = [uL^2 + uR^2 + 2 alpha (uL - uR)] / 2
      const double a = max_speed(L[0], R[0]), d = K.sub(L[0], R[0]);
      G[q][0] = fma(K.mul(tab[T::HALF], L[0]), L[0], fma(K.mul(tab[T::HALF], R[0]), R[0], K.mul(a, d)));
    } else {
      double rL, vL, wL, pL, rR, vR, wR, pR;
      euler_state(L[0], L[1], L[2], L[3], tab, T::GM1, T::HGM1, K, rL, vL, wL, pL);
      euler_state(R[0], R[1], R[2], R[3], tab, T::GM1, T::HGM1, K, rR, vR, wR, pR);
      const double c38 = tab[T::C38], half = tab[T::HALF], sg = tab[T::SG];
      const double a = max_speed(fma(sg, sqrt_t(K.mul(pL, rL), K, c38, half), fabs(vL)),
                                 fma(sg, sqrt_t(K.mul(pR, rR), K, c38, half), fabs(vR)));
      G[q][0] = fma(a, K.sub(L[0], R[0]), K.add(L[1], R[1]));
      G[q][1] = fma(a, K.sub(L[1], R[1]), fma(L[1], vL, fma(R[1], vR, K.add(pL, pR))));
      G[q][2] = fma(a, K.sub(L[2], R[2]), fma(L[2], vL, K.mul(R[2], vR)));
      G[q][3] = fma(a, K.sub(L[3], R[3]), fma(K.add(L[3], pL), vL, K.mul(K.add(R[3], pR), vR)));
    }
  }
  // P_b over w_0 psi_b(s_0)
  double* const base = dir == 0 ? fx + I.fx + (long long)j * (I.nx + 1) + k : fy + I.fy + (long long)j * I.nx + k;
  const long long stride = dir == 0 ? fxt : fyt;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int pv = (V == 4 && (v == 1 || v == 2) && dir) ? 3 - v : v;
    double S[Q / 2], D[Q / 2];
#pragma unroll
    for (int q = 0; q < Q / 2; ++q) {
      S[q] = K.add(G[q][v], G[Q - 1 - q][v]);
      D[q] = K.sub(G[q][v], G[Q - 1 - q][v]);
    }
#pragma unroll
    for (int b = 0; b <= N; ++b)
      base[(long long)(pv * N1 + b) * stride] = rel_sum<N>(!(b & 1), S, D, G[Q / 2][v], tab[T::KAP + b]);
  }
}

// One thread per cell; Tile::x0: chunk of kCellChunk cells of the instance.
// Two blocks per SM (at most 128 registers) except for Euler P3; Euler P2 and P3 keep the cell's
// modes in shared memory (one slot per thread and mode).  Point values in fixed point pay for
// P2 (Euler 878 -> 809 us at 1024^2, Burgers 211 -> 198 us); P1 has too little to move (439 -> 470 us)
// and P3 no registers for it (1.98 -> 2.74 ms): those stay in FP64.  Euler P2 pays for it with
// register spills (588 B stored and 836 B loaded per thread; 104 and 116 B with FP64 values, plain
// sums and no modes in shared memory) and a second read of the modes for the combination; one
// block per SM, with room for both, is no faster (13.5 against 13.3 ms per 1024^2 step).
__host__ __device__ constexpr bool fixed_values(int N) { return N == 2; }
__host__ __device__ constexpr bool smem_modes(int pde, int N) { return pde == 1 && N >= 2; }

template <int PDE, int N>
__global__ void __launch_bounds__(kCellChunk, (PDE == 1 && N == 3) ? 1 : 2)
    k_cell2(const double* __restrict__ un, const double* __restrict__ us, double* __restrict__ out,
            const Inst* __restrict__ insts, const Tile* __restrict__ tiles, long long ctot, int stage, double dt_all,
            const double* __restrict__ fx, long long fxt, const double* __restrict__ fy, long long fyt, Gamma gm) {
  using T = STab<N>;
  constexpr int V = nv_of(2, PDE), NP = np_of(2, N), Q = N + 1, N1 = N + 1, NX = T::NX, NH = Q / 2;
  constexpr int V0 = PDE == 1 ? 1 : 0;  // first variable whose volume term needs quadrature
  __shared__ __align__(16) double tab[T::SIZE];
  const Tile tile = tiles[blockIdx.x];
  const Inst I = insts[tile.inst];
  if (threadIdx.x < T::SIZE) {
    const int k = threadIdx.x;
    const double wb = stage == 1 ? 1.0 : (stage == 2 ? 0.25 : 2.0 / 3.0);
    const double dt = dt_all > 0.0 ? dt_all : I.dt;
    double x = g_stab[N - 1][k];
    if (k == T::GM1) x = gm.gm1;
    if (k == T::HGM1) x = gm.hgm1;
    if (k == T::RA) x = stage == 2 ? 0.75 : 1.0 / 3.0;
    if (k == T::RB) x = wb;
    // the states behind X, Y and the P_b are doubled: 2^-d (exact)
    if (k >= T::XF) x *= (k >= T::YF ? I.sy : I.sx) * (dt * wb) * (PDE == 1 ? 0.5 : 0.25);
    tab[k] = x;
  }
  const unsigned loc = (unsigned)tile.x0 * kCellChunk + threadIdx.x;
  const int iy = (int)(loc / (unsigned)I.nx), ix = (int)(loc - (unsigned)iy * (unsigned)I.nx);
  __syncthreads();
  if (iy >= I.ny) return;
  const Reg64 K{tab[T::ONE], tab[T::NZ]};
  const long long g = I.off + loc;
  constexpr bool kFix = fixed_values(N), kSmemU = smem_modes(PDE, N);
  const long long* itab = reinterpret_cast<const long long*>(tab);
  extern __shared__ long long s_x[];  // the modes as doubles or aligned integers
  long long xr[kSmemU ? 1 : V][kSmemU ? 1 : NP];
  int E[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    double u[NP];
    long long X[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      u[m] = __ldg(us + (long long)(v * NP + m) * ctot + g);
      X[m] = __double_as_longlong(u[m]);
    }
    if constexpr (kFix) E[v] = align_modes<NP, 8, 2>(u, X);  // |X| < 2^61; sums below 2^62, 4 |tb_1| below 2^62.3
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      if constexpr (kSmemU) s_x[(v * NP + m) * kCellChunk + threadIdx.x] = X[m];
      else xr[v][m] = X[m];
    }
  }
  auto x = [&](int v, int m) -> long long {
    if constexpr (kSmemU) return s_x[(v * NP + m) * kCellChunk + threadIdx.x];
    else return xr[v][m];
  };
  auto u = [&](int v, int m) -> double {
    if constexpr (kFix) return __ldg(us + (long long)(v * NP + m) * ctot + g);
    else return __longlong_as_double(x(v, m));
  };
  // acc[v][m]: the stage's weight times dt times the right-hand side
  double acc[V][NP];
#pragma unroll
  for (int v = V0; v < V; ++v)
#pragma unroll
    for (int m = 0; m < NP; ++m) acc[v][m] = 0.0;
  auto add_to = [&](int v, int m, bool first, double c, double x) {
    acc[v][m] = first ? K.mul(c, x) : fma(c, x, acc[v][m]);
  };
  // x points in symmetric pairs (-x_p, x_p), the middle point (N = 2) last.  y sums of a
  // column: Gs_b of f with psi_b, b < N; Hs_b of g with psi_b', b >= 1.
#pragma unroll
  for (int p = 0; p < NX; ++p) {
    const bool mid = (Q & 1) && p == Q / 2;
    double tb[kFix ? 1 : 2][kFix ? 1 : V][N1];  // FP64: over psi_0, at -x_p and x_p (parts even and odd in a)
    if constexpr (!kFix) {
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int b = 0; b <= N; ++b) {
          const double* c = tab + T::KD + p * N1;
          double ev = u(v, mode_idx(0, b));
          if (N - b >= 2) ev = fma(c[N >= 2 ? 2 : 0], u(v, mode_idx(N - b >= 2 ? 2 : 0, b)), ev);
          tb[0][v][b] = tb[1][v][b] = ev;
          if (mid || b == N) continue;
          const double u1 = u(v, mode_idx(b < N ? 1 : 0, b));
          if (N - b >= 3) {
            const double od = fma(c[3 <= N ? 3 : 0], u(v, mode_idx(N - b >= 3 ? 3 : 0, b)), K.mul(c[1], u1));
            tb[0][v][b] = K.add(ev, od);
            tb[1][v][b] = K.sub(ev, od);
          } else {
            tb[0][v][b] = fma(c[1], u1, ev);
            tb[1][v][b] = fma(-c[1], u1, ev);
          }
        }
    }
    double Gs[V][N], Hs[V][N];  // of the column at -x_p
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (mid && side) break;
      double col[V][Q];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        if constexpr (kFix) {
          // x sums over psi_0 at -x_p (side 0) or x_p in units of 4 X (formed again for each side: the
          // integer pipes have the time, the registers are short), then the y points
          const long long* c = itab + T::KQ + p * N1;
          long long tb[N1], val[Q];
  #pragma unroll
          for (int b = 0; b <= N; ++b) {
            long long ev = x(v, mode_idx(0, b)) >> 2, od = 0;
            if (N - b >= 2) ev += mul_rn(c[N >= 2 ? 2 : 0], x(v, mode_idx(N - b >= 2 ? 2 : 0, b)));
            if (!mid && b < N) od = mul_rn(c[1], x(v, mode_idx(b < N ? 1 : 0, b)));
            if (N - b >= 3) od += mul_rn(c[3 <= N ? 3 : 0], x(v, mode_idx(N - b >= 3 ? 3 : 0, b)));
            tb[b] = side == 0 ? ev + od : ev - od;
          }
          eval_fix<N>(tb, itab + T::KQ, val);
  #pragma unroll
          for (int q = 0; q < Q; ++q)
            col[v][q] = E[v] < 2047 ? pack_s64<true>(val[q], E[v] - 1081) : __longlong_as_double(0x7ff8000000000000LL);
        } else {
          eval_gauss2<N>(tb[side][v], tab + T::KD, K, col[v]);
        }
      }
      double F[V][Q], H[V][Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if constexpr (PDE == 0) {
          F[0][q] = H[0][q] = K.mul(K.mul(tab[T::HALF], col[0][q]), col[0][q]);
        } else {
          double r, vx, vy, pr;
          const double mx = col[1][q], my = col[2][q], E = col[3][q];
          euler_state(col[0][q], mx, my, E, tab, T::GM1, T::HGM1, K, r, vx, vy, pr);
          const double ep = K.add(E, pr);
          F[1][q] = fma(mx, vx, pr);
          F[2][q] = H[1][q] = K.mul(my, vx);
          F[3][q] = K.mul(ep, vx);
          H[2][q] = fma(my, vy, pr);
          H[3][q] = K.mul(ep, vy);
        }
      }
#pragma unroll
      for (int v = V0; v < V; ++v) {
        double fS[NH], fD[NH], hS[NH], hD[NH], gn[N], hn[N];
#pragma unroll
        for (int q = 0; q < NH; ++q) {
          fS[q] = K.add(F[v][q], F[v][Q - 1 - q]);
          fD[q] = K.sub(F[v][q], F[v][Q - 1 - q]);
          hS[q] = K.add(H[v][q], H[v][Q - 1 - q]);
          hD[q] = K.sub(H[v][q], H[v][Q - 1 - q]);
        }
#pragma unroll
        for (int b = 0; b < N; ++b) {
          gn[b] = rel_sum<N>(!(b & 1), fS, fD, F[v][Q / 2], tab[T::KAP + b]);
          hn[b] = rel_sum<N>(!(b & 1), hS, hD, H[v][Q / 2], tab[T::KAD + b + 1]);  // psi_{b+1}'
        }
        if (mid) {
#pragma unroll
          for (int m = 1; m < NP; ++m) {
            const int a = mode_a(m), b = mode_b(m);
            if (a & 1) add_to(v, m, false, tab[T::CX + p * NP + m], gn[a ? b : 0]);  // psi_a'(0) = 0 for even a
            if (b && !(a & 1)) add_to(v, m, false, tab[T::CY + p * NP + m], hn[b ? b - 1 : 0]);
          }
        } else if (side == 0) {
#pragma unroll
          for (int b = 0; b < N; ++b) {
            Gs[v][b] = gn[b];
            Hs[v][b] = hn[b];
          }
        } else {
          double gS[N], gD[N], sS[N], sD[N];
#pragma unroll
          for (int b = 0; b < N; ++b) {
            gS[b] = K.add(Gs[v][b], gn[b]);
            gD[b] = K.sub(Gs[v][b], gn[b]);
            sS[b] = K.add(Hs[v][b], hn[b]);
            sD[b] = K.sub(Hs[v][b], hn[b]);
          }
#pragma unroll
          for (int m = 1; m < NP; ++m) {
            const int a = mode_a(m), b = mode_b(m);
            if (a) add_to(v, m, p == 0, tab[T::CX + p * NP + m], (a & 1) ? gS[a ? b : 0] : gD[a ? b : 0]);
            if (b) add_to(v, m, p == 0 && a == 0, tab[T::CY + p * NP + m], (a & 1) ? sD[b ? b - 1 : 0] : sS[b ? b - 1 : 0]);
          }
        }
      }
    }
  }
  if constexpr (PDE == 1) {  // density: the x (y) flux is the x (y) momentum
#pragma unroll
    for (int m = 1; m < NP; ++m) {
      const int a = mode_a(m), b = mode_b(m);
      if (a) {
        add_to(0, m, true, tab[T::DX + a - 1], u(1, mode_idx(a - 1, b)));
        if (a == 3) add_to(0, m, false, tab[T::DX + 3], u(1, mode_idx(0, b)));
      }
      if (b) {
        add_to(0, m, a == 0, tab[T::DY + b - 1], u(2, mode_idx(a, b - 1)));
        if (b == 3) add_to(0, m, false, tab[T::DY + 3], u(2, mode_idx(a, 0)));
      }
    }
  }
  // - (1/hx) psi_a(1) [P_b(E) -+ P_b(W)] - (1/hy) psi_b(1) [P_a(N) -+ P_a(S)], then the stage
  const double* const pw = fx + I.fx + (long long)iy * (I.nx + 1) + ix;  // west face; east = pw + 1
  const double* const ps = fy + I.fy + (long long)iy * I.nx + ix;        // south face; north = ps + nx
#pragma unroll
  for (int v = 0; v < V; ++v) {
#pragma unroll
    for (int t = 0; t <= N; ++t) {  // transverse degree
      const long long pl = (long long)(v * N1 + t);
      const double PW = __ldg(pw + pl * fxt), PE = __ldg(pw + pl * fxt + 1);
      const double PS = __ldg(ps + pl * fyt), PN = __ldg(ps + pl * fyt + I.nx);
      const double Dx = K.sub(PE, PW), Sx = K.add(PE, PW), Dy = K.sub(PN, PS), Sy = K.add(PN, PS);
#pragma unroll
      for (int n = 0; n <= N - t; ++n) {  // normal degree
        const int mx = mode_idx(n, t), my = mode_idx(t, n);
        add_to(v, mx, mx == 0, tab[T::LX + mx], (n & 1) ? Sx : Dx);
        add_to(v, my, false, tab[T::LY + my], (n & 1) ? Sy : Dy);
      }
    }
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      const long long idx = (long long)(v * NP + m) * ctot + g;
      if (stage == 1) out[idx] = K.add(u(v, m), acc[v][m]);
      else out[idx] = fma(tab[T::RA], un[idx], fma(tab[T::RB], u(v, m), acc[v][m]));
    }
  }
}

// The traces alone (dg_refined_arith): out[q][i] from the modes x[m][i], i < n.
template <int N>
__global__ void __launch_bounds__(256) k_trace_probe(const double* __restrict__ x, double* __restrict__ out, long long n) {
  using T = STab<N>;
  __shared__ __align__(16) double tab[T::FACE];
  if (threadIdx.x < T::XF) tab[threadIdx.x] = g_stab[N - 1][threadIdx.x];
  __syncthreads();
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
    const TraceVal<N> o = trace<N>(x + i, n, 0, false, false, false, nullptr, reinterpret_cast<const long long*>(tab));
#pragma unroll
    for (int q = 0; q <= N; ++q) out[q * n + i] = o.v[q];
  }
}

// dynamic shared memory of the cell pass: the modes of its 256 cells
constexpr size_t cell_smem(int pde, int N) {
  return smem_modes(pde, N) ? sizeof(long long) * 4 * ((N + 1) * (N + 2) / 2) * kCellChunk : 0;
}

template <int PDE, int N>
void launch(const LaunchArgs& a, int stage, double dt_all, const Tile* face_tiles, int nface_tiles, double* fx,
            long long fxt, double* fy, long long fyt) {
  const Gamma gm{a.gam - 1.0, -0.5 * (a.gam - 1.0), std::sqrt(a.gam)};
  k_face2<PDE, N><<<nface_tiles, kFaceChunk, 0, a.st>>>(a.us, a.inst, face_tiles, a.ctot, a.bc, gm, fx, fxt, fy, fyt,
                                                        a.bcd, stage, dt_all);
  k_cell2<PDE, N><<<a.ntiles, kCellChunk, cell_smem(PDE, N), a.st>>>(a.un, a.us, a.out, a.inst, a.tiles, a.ctot, stage,
                                                                     dt_all, fx, fxt, fy, fyt, gm);
}

}  // namespace st2

cudaError_t upload_tables_stage2(const dgt::Tabs* tabs) {
  static double h[3][st2::kSTab];
  st2::pack<1>(tabs[0], h[0]);
  st2::pack<2>(tabs[1], h[1]);
  st2::pack<3>(tabs[2], h[2]);
  return cudaMemcpyToSymbol(st2::g_stab, h, sizeof(h));
}

// opt in to more than 48 KB of dynamic shared memory (set per device, outside captures)
cudaError_t prepare_stage2_split(int pde, int N) {
  if (!st2::cell_smem(pde, N)) return cudaSuccess;
  const int bytes = (int)st2::cell_smem(pde, N);
  return N == 2 ? cudaFuncSetAttribute(st2::k_cell2<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
                : cudaFuncSetAttribute(st2::k_cell2<1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

void launch_trace_probe(cudaStream_t st, int N, const double* x, double* out, long long n, int nblocks) {
  if (N == 1) st2::k_trace_probe<1><<<nblocks, 256, 0, st>>>(x, out, n);
  else if (N == 2) st2::k_trace_probe<2><<<nblocks, 256, 0, st>>>(x, out, n);
  else st2::k_trace_probe<3><<<nblocks, 256, 0, st>>>(x, out, n);
}

int face_chunk2() { return st2::kFaceChunk; }
int cell_chunk2() { return st2::kCellChunk; }

// split form: the face pass over the face chunks, then the cell pass over the cell chunks (a.tiles)
void launch_stage2_split(int pde, int N, const LaunchArgs& a, int stage, double dt_all, const Tile* face_tiles,
                         int nface_tiles, double* fx, long long fxt, double* fy, long long fyt) {
#define DG_S2(P, NN) st2::launch<P, NN>(a, stage, dt_all, face_tiles, nface_tiles, fx, fxt, fy, fyt)
  if (pde == 0) {
    if (N == 1) DG_S2(0, 1);
    else if (N == 2) DG_S2(0, 2);
    else DG_S2(0, 3);
  } else {
    if (N == 1) DG_S2(1, 1);
    else if (N == 2) DG_S2(1, 2);
    else DG_S2(1, 3);
  }
#undef DG_S2
}

}  // namespace dg
