// 1D initial projection (Eq. (2)) and the largest characteristic speed over the cell means
// (P^N, N = 1..3; Burgers V = 1, Euler V = 3).  The step itself is in dg_step1.cu.
#include "dg_ic.cuh"
#include "dg_shared.cuh"
#include "tables.h"

namespace dg {
namespace k1 {


template <int N>
struct Off {
  static constexpr int N1 = N + 1;
  static constexpr int P0 = (N - 1) * 64;  // psi_0
  static constexpr int PX = P0 + 1;        // [8] points and
  static constexpr int PW = PX + 8;        // [8] weights of the projection rule
  static constexpr int PQP = PW + 8;       // their number
  static constexpr int PP = PQP + 1;       // [8][N1] psi_n at the points
  static constexpr int END = PP + 8 * N1;
};
static_assert(Off<3>::END <= 192, "one row of 64 per degree");
constexpr int kTabSize = 192;

__constant__ double c_tab[kTabSize];
#define T(x) c_tab[(x)]

template <int N>
void pack(const dgt::Tabs& t, double* h) {
  using O = Off<N>;
  h[O::P0] = t.psi_0[0];
  for (int q = 0; q < t.QP; ++q) {
    h[O::PX + q] = t.px[q];
    h[O::PW + q] = t.pw[q];
    for (int n = 0; n <= N; ++n) h[O::PP + q * O::N1 + n] = t.ppsi[q][n];
  }
  h[O::PQP] = t.QP;
}

template <int PDE, int N>
__global__ void k_project1(double* __restrict__ U, const Inst* __restrict__ insts, const int* __restrict__ cell_inst,
                           long long ncell, long long ctot, int kind, const double* __restrict__ params, int np,
                           double gam) {
  using O = Off<N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1;
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  const int ii = cell_inst[g];
  const Inst I = insts[ii];
  const int ix = (int)(g - I.off);
  const double* p = params + (long long)ii * np;
  const int QP = (int)T(O::PQP);
  double acc[V][N1];
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int n = 0; n < N1; ++n) acc[v][n] = 0.0;
  for (int q = 0; q < QP; ++q) {
    const double x = I.xL + I.hx * (ix + 0.5 * (1.0 + T(O::PX + q)));
    double u[V];
    ic_eval1(kind, p, x, gam, u);
#pragma unroll
    for (int n = 0; n < N1; ++n) {
      const double c = T(O::PW + q) * T(O::PP + q * N1 + n);
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v][n] = fma(c, u[v], acc[v][n]);
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int n = 0; n < N1; ++n) U[(long long)(v * N1 + n) * ctot + g] = acc[v][n];
}

template <int PDE, int N>
__global__ void k_speed1(const double* __restrict__ U, const Inst* __restrict__ insts, const int* __restrict__ cell_inst,
                         long long ncell, long long ctot, double gam, double* out) {
  using O = Off<N>;
  constexpr int V = nv_of(1, PDE), N1 = N + 1;
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  double u[V];
  for (int v = 0; v < V; ++v) u[v] = U[(long long)(v * N1) * ctot + g] * T(O::P0);
  double s;
  if constexpr (PDE == 0) {
    s = fabs(u[0]);
  } else {
    const double r = 1.0 / u[0], vel = u[1] * r;
    const double p = (gam - 1.0) * (u[2] - 0.5 * u[0] * vel * vel);
    s = fabs(vel) + sqrt(gam * p * r);
  }
  atomic_max_nonneg(out + 2 * cell_inst[g], s);
}

#undef T
}  // namespace k1


cudaError_t upload_tables1(const dgt::Tabs* tabs) {
  static double h[k1::kTabSize];
  for (int i = 0; i < k1::kTabSize; ++i) h[i] = 0.0;
  k1::pack<1>(tabs[0], h);
  k1::pack<2>(tabs[1], h);
  k1::pack<3>(tabs[2], h);
  return cudaMemcpyToSymbol(k1::c_tab, h, sizeof(h));
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

void launch_scatter1(int pde, int N, const LaunchArgs& a, const double* lim, const int* lc, const Counters* cnt,
                     int nblocks) {
  DG_DISPATCH1(pde, N, (k_scatter<nv_of(1, P_), np_of(1, N_)><<<nblocks, 256, 0, a.st>>>(a.out, a.ctot, lim, a.cap,
                                                                                          lc, cnt)));
}

void launch_project1(int pde, int N, const LaunchArgs& a, const int* cell_inst, int kind, const double* params,
                     int np) {
  const int nb = (int)((a.ncell + 127) / 128);
  DG_DISPATCH1(pde, N, (k1::k_project1<P_, N_><<<nb, 128, 0, a.st>>>(a.out, a.inst, cell_inst, a.ncell, a.ctot,
                                                                       kind, params, np, a.gam)));
}

void launch_speed1(int pde, int N, const LaunchArgs& a, const int* cell_inst, double* out) {
  const int nb = (int)((a.ncell + 255) / 256);
  DG_DISPATCH1(pde, N, (k1::k_speed1<P_, N_><<<nb, 256, 0, a.st>>>(a.us, a.inst, cell_inst, a.ncell, a.ctot,
                                                                     a.gam, out)));
}

}  // namespace dg
