// Host-side tables of the method for one polynomial degree N (1..3).
//
// Everything here is derived at library start-up from the definitions in Sec. 2 and
// Sec. 3 of the paper (basis, quadrature rules, CSWENO reconstruction rows, linear
// weights, smoothness-indicator quadratic forms, subcell averages).
#pragma once

#ifdef __CUDACC__
#define DGT_HD __host__ __device__
#else
#define DGT_HD
#endif

namespace dgt {

constexpr int kMaxN = 3;
constexpr int kMaxQ = 8;   // Gauss points (N+4 <= 7 for the initial projection)
constexpr int kMaxS = 7;   // stencil cells 2N+1
constexpr int kMaxG = 4;   // reconstruction points per direction

struct Tabs {
  int N, Q, NG, NS;
  // (N+1)-point Gauss-Legendre rule of the weak form (Eq. (5)), weights sum to 2
  double gx[kMaxQ], gw[kMaxQ];
  double psi_q[kMaxQ][kMaxN + 1], dpsi_q[kMaxQ][kMaxN + 1];
  double psi_p1[kMaxN + 1], psi_m1[kMaxN + 1], psi_0[kMaxN + 1];
  // the same basis values over psi_0 = 1/sqrt(2): sqrt(2) psi_n at the Gauss points and at 1
  // (2^62 and 2^61 times them as integers, for fixed-point sums)
  double kq[kMaxQ][kMaxN + 1];
  long long kq_fix[kMaxQ][kMaxN + 1], kp1_fix[kMaxN + 1];
  // CSWENO (Sec. 3, Steps 1-6)
  double rp[kMaxG], rw[kMaxG];               // Step 1 points (reference r) and weights
  double psiG[kMaxG][kMaxN + 1];             // psi_n at the Step 1 points
  double C[kMaxN + 1][kMaxG][kMaxN + 1];     // p_i(x_g) = sum_k C[i][g][k] avg[i+k]
  double gam[kMaxG][kMaxN + 1];              // Eq. (8)
  double B[kMaxN + 1][kMaxN + 1][kMaxN + 1]; // beta_i = sum_kl avg[i+k] B[i][k][l] avg[i+l]
  double SA[kMaxS][kMaxN + 1];               // average of psi_n over stencil cell k
  int OFF[kMaxS];                            // -1 / 0 / +1: neighbour holding stencil cell k
  int neg[kMaxG];                            // point g has a negative linear weight
  double gpn[kMaxG][kMaxN + 1], gmn[kMaxG][kMaxN + 1]; // normalised split weights
  double sgp[kMaxG], sgm[kMaxG];                        // sigma+, sigma-
  // The reconstruction of Steps 2-5 on the 2N differences d_k = avg[k+1] - avg[k] of
  // neighbouring stencil averages (p_i - avg[N] and beta_i ignore constants), as the 2D
  // limiters evaluate it.  With e = (d_i .. d_{i+N-1}) of stencil i, read from its far end
  // for i <= N/2 and mirrored for the others, beta_i / M is a sum of squares,
  //   N = 1: e_0^2;  N = 2: (e_0 + k e_1)^2 + o e_1^2;
  //   N = 3: (e_0 + k e_1 + l e_2)^2 + m (e_1 + n e_2)^2 + o e_2^2,
  // with the same constants for stencils i and N - i (class min(i, N - i)).  bform = {eps / M, o, m, k, l, n}.
  double bform[2][6];
  // p_i(x_g) - avg[N] = sum_j E_gij d_{i+j}.  With P_i proportional to 1 / (eps + beta_i)^2 and
  // wh[g][i] = gamma_gi over its value at the reference stencil weno_ref(N, g),
  // wc[g][i][j] = wh[g][i] E_gij,
  //   u_g - avg[N] = sum_ij wc_gij P_i d_{i+j} / sum_i wh_gi P_i.
  // At a point with one negative weight (sigma+ and sigma- of the split) wh and wc of that
  // stencil are taken with |gamma|; qsp = {4 sigma+ - sigma- - 1, 4 sigma- - sigma+ + 1}.
  // brel = M of the outer stencils over M of the inner ones (1 for N = 1).
  double wh[kMaxG][kMaxN + 1], wc[kMaxG][kMaxN + 1][kMaxN], qsp[2], brel;
  // initial projection: (N+4)-point Gauss rule
  int QP;
  double px[kMaxQ], pw[kMaxQ], ppsi[kMaxQ][kMaxN + 1];
  double gam_resid;                          // residual of the full Eq. (8) system
};

// Stencil whose weight is 1 in wh, and the stencil with a negative linear weight of the
// CSWENO P3 rule at its inner points (-1: none).
DGT_HD constexpr int weno_ref(int N, int g) { return N == 3 && g == 1 ? 2 : 1; }
DGT_HD constexpr int weno_neg(int N, int g, bool parent) {
  return N == 3 && !parent && g == 1 ? 3 : (N == 3 && !parent && g == 2 ? 0 : -1);
}

// Whether wh and wc fit the kernels' fixed point (weno_diff): as 64-bit constants (|wc| < 2, wh < 2), and
// in the sums over the stencils, of terms below |wc| 2^60 in 2^63 and below wh 2^61 in 2^63.  At a point
// with a negative weight the two parts are summed apart.
bool sums_fit(const Tabs& t, bool parent);

// Fills t for degree N; returns 0 on success.  parent: the limiter tables of the parent
// WENO limiter (whole cells j-N .. j+N) instead of CSWENO's subcells.
int build_tables(int N, Tabs* t, bool parent = false);

}  // namespace dgt
