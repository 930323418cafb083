// dg_adjoint.cuh -- discrete adjoint (vector-Jacobian product) of the FP64 split-form DGSEM
// right-hand side L(U) for ONE polynomial degree; included after dg_kernels.cuh in the same
// translation unit (same anonymous namespace, same constant tables).
//
// Given a cotangent lambda of Ut = L(U), the kernels form Ubar = (dL/dU)^T lambda, the transpose
// of exactly the operator the forward kernels apply (zero-diagonal flux differencing with the
// SBP surface identity, Riemann flux once per face point, BR1 lifting with central face values,
// -(1/(2 w_b)) phi_nb for the neighbour's viscous flux, -1/J). With l = -lambda/J per node:
//
//   adj_face    per face point: c = s/w_0 (l_L - l_R) is the cotangent of F*(U_L, U_R, n); its
//               transposed Jacobian goes to both sides' face slots. Roe and LLF: hand-written
//               reverse mode of the forward statements; EC: forward-mode dual numbers (5 seeds per
//               pass, 2 passes) through the same templated code the forward kernel runs.
//   adj_visc    (Navier-Stokes) per element: transpose the viscous divergence (D^T sweeps of l,
//               neighbour term through the face), the contravariant projection and the
//               Navier-Stokes-Fourier flux (pointwise, at the viscous stress the forward lifting
//               recorded for this state), then the lifting (D^T sweeps, central face value):
//               cotangents of (u, v, w, T) per node plus face slots for the neighbour's share.
//   adj_volume  per element: the two-point flux differencing transposed pair by pair. With
//               sums S = x_i + x_m the Kennedy-Gruber / Pirozzoli fluxes are polynomials in
//               (S_rho, S_u, S_p, S_X), so each pair adds the same cotangent vector to both of its
//               nodes' primitive accumulators (in 64-bit fixed point); then per node the primitive cotangents (plus the
//               viscous ones) are chained to the conservative variables, the face slots are added,
//               and either Ubar is written or the LSERK(5,4) reverse stage is applied in place.
#pragma once
#include "dg_dual.cuh"

namespace {

// ---------------------------------------------------------------------------------------------
// reverse-mode derivatives of the Riemann fluxes (the statements of riemann<double>, transposed)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double sgn_of(double x) { return x < 0.0 ? -1.0 : 1.0; }  // d|x|/dx, +1 at 0

// primitives of one side: ir = 1/rho (given: (1/sqrt(rho))^2, as the forward solver forms it),
// u = m ir, p = (gamma-1)(E - |m|^2 ir / 2)
struct Side {
  double ir, u[3], p, un;
};

__device__ __forceinline__ Side side_of(const double U[5], const double nv[3], double gm1, double ir) {
  Side s;
  s.ir = ir;
  s.u[0] = U[1] * s.ir;
  s.u[1] = U[2] * s.ir;
  s.u[2] = U[3] * s.ir;
  s.p = gm1 * (U[4] - 0.5 * (U[1] * s.u[0] + U[2] * s.u[1] + U[3] * s.u[2]));
  s.un = s.u[0] * nv[0] + s.u[1] * nv[1] + s.u[2] * nv[2];
  return s;
}

// cotangents of (u, p, un, ir) of one side -> cotangent of U (added to g)
__device__ __forceinline__ void side_back(const double U[5], const Side &s, const double nv[3], double gm1,
                                          double cu[3], double cp, double cun, double cir, double g[5]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) cu[k] += cun * nv[k];
  // p = gm1 (E - |m|^2 ir / 2): dp/dE = gm1, dp/dm_k = -gm1 u_k, dp/dir = -gm1 |m|^2 / 2
  g[4] += gm1 * cp;
  const double m2 = U[1] * U[1] + U[2] * U[2] + U[3] * U[3];
  cir -= 0.5 * gm1 * m2 * cp;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    g[1 + k] += cu[k] * s.ir - gm1 * s.u[k] * cp;
    cir += cu[k] * U[1 + k];
  }
  g[0] -= cir * s.ir * s.ir;
}

// Euler flux F = (rho un, m un + p n, (E + p) un) of one side, reversed: adds dF^T cF to the side's
// cotangents (cu, cp, cun) and to g directly
__device__ __forceinline__ void flux_back(const double U[5], const Side &s, const double nv[3], const double cF[5],
                                          double &cp, double &cun, double g[5]) {
  cun += cF[0] * U[0] + cF[1] * U[1] + cF[2] * U[2] + cF[3] * U[3] + cF[4] * (U[4] + s.p);
  cp += cF[1] * nv[0] + cF[2] * nv[1] + cF[3] * nv[2] + cF[4] * s.un;
#pragma unroll
  for (int v = 0; v < 5; ++v) g[v] += cF[v] * s.un;
}

// gL = (dF*/dU_L)^T cF, gR = (dF*/dU_R)^T cF for the LLF flux
__device__ void llf_vjp(const double UL[5], const double UR[5], const double nv[3], double gam, const double cF[5],
                        double gL[5], double gR[5]) {
  const double gm1 = gam - 1.0;
  const double rsL = rsq(UL[0]), rsR = rsq(UR[0]);
  const Side L = side_of(UL, nv, gm1, rsL * rsL), R = side_of(UR, nv, gm1, rsR * rsR);
  const double cL = sqr_int(gam * L.p * L.ir), cR = sqr_int(gam * R.p * R.ir);
  const double aL = fabs(L.un) + cL, aR = fabs(R.un) + cR;
  const bool rwins = aR > aL;  // the forward's max picks the right argument only when strictly larger
  const double lam = rwins ? aR : aL;
  double clam = 0.0, hF[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    hF[v] = 0.5 * cF[v];
    gL[v] = 0.5 * lam * cF[v];
    gR[v] = -0.5 * lam * cF[v];
    clam -= 0.5 * cF[v] * (UR[v] - UL[v]);
  }
  double cuL[3] = {0, 0, 0}, cuR[3] = {0, 0, 0}, cpL = 0, cpR = 0, cunL = 0, cunR = 0, cirL = 0, cirR = 0;
  flux_back(UL, L, nv, hF, cpL, cunL, gL);
  flux_back(UR, R, nv, hF, cpR, cunR, gR);
  // lam = |un_X| + sqrt(gamma p_X / rho_X) of the winning side X
  if (rwins) {
    cunR += clam * sgn_of(R.un);
    cpR += clam * 0.5 * cR * rcp_int(R.p);
    gR[0] -= clam * 0.5 * cR * R.ir;
  } else {
    cunL += clam * sgn_of(L.un);
    cpL += clam * 0.5 * cL * rcp_int(L.p);
    gL[0] -= clam * 0.5 * cL * L.ir;
  }
  side_back(UL, L, nv, gm1, cuL, cpL, cunL, cirL, gL);
  side_back(UR, R, nv, gm1, cuR, cpR, cunR, cirR, gR);
}

// the same for Roe's flux (no entropy fix), statement by statement in reverse; as in the forward
// solver, one reciprocal square root per side (1/rho = rs^2, sqrt(rho) = rho rs, 1/(2 sqrt(rho)) = rs/2)
// and one for the sound speed (c = c^2 rc, 1/c^2 = rc^2, 1/(2c) = rc/2)
__device__ void roe_vjp(const double UL[5], const double UR[5], const double nv[3], double gam, const double cF[5],
                        double gL[5], double gR[5]) {
  const double gm1 = gam - 1.0;
  const double rsL = rsq(UL[0]), rsR = rsq(UR[0]);
  const Side L = side_of(UL, nv, gm1, rsL * rsL), R = side_of(UR, nv, gm1, rsR * rsR);
  // forward
  const double sL = UL[0] * rsL, sR = UR[0] * rsR;
  const double iw = rcp_int(sL + sR);
  double ut[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) ut[k] = (sL * L.u[k] + sR * R.u[k]) * iw;
  const double EpL = UL[4] + L.p, EpR = UR[4] + R.p;
  const double hL = EpL * L.ir, hR = EpR * R.ir;
  const double Ht = (sL * hL + sR * hR) * iw;
  const double q2 = ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2];
  const double c2 = gm1 * (Ht - 0.5 * q2);
  const double rc = rsq(c2);
  const double ct = c2 * rc, ic2 = rc * rc;
  const double rt = sL * sR;
  const double unt = ut[0] * nv[0] + ut[1] * nv[1] + ut[2] * nv[2];
  const double dr = UR[0] - UL[0], dp = R.p - L.p;
  const double du[3] = {R.u[0] - L.u[0], R.u[1] - L.u[1], R.u[2] - L.u[2]};
  const double dun = du[0] * nv[0] + du[1] * nv[1] + du[2] * nv[2];
  const double A1 = dp - rt * ct * dun, A5 = dp + rt * ct * dun;
  const double a1 = 0.5 * A1 * ic2, a5 = 0.5 * A5 * ic2, a2 = dr - dp * ic2;
  double dt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) dt[k] = du[k] - dun * nv[k];
  const double s1 = fabs(unt - ct), s5 = fabs(unt + ct), l2 = fabs(unt);
  const double l1a1 = s1 * a1, l5a5 = s5 * a5, l2a2 = l2 * a2, l2r = l2 * rt;
  const double utdt = ut[0] * dt[0] + ut[1] * dt[1] + ut[2] * dt[2];
  // reverse: F = (FL + FR - D) / 2
  double cD[5], hF[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) { hF[v] = 0.5 * cF[v]; cD[v] = -hF[v]; }
  double cnt = cD[1] * nv[0] + cD[2] * nv[1] + cD[3] * nv[2];  // sum_k cD_k n_k
  double cut_dot = cD[1] * ut[0] + cD[2] * ut[1] + cD[3] * ut[2];
  const double c_l1a1 = cD[0] + cut_dot - ct * cnt + cD[4] * (Ht - unt * ct);
  const double c_l5a5 = cD[0] + cut_dot + ct * cnt + cD[4] * (Ht + unt * ct);
  const double c_l2a2 = cD[0] + cut_dot + cD[4] * 0.5 * q2;
  const double c_l2r = cD[1] * dt[0] + cD[2] * dt[1] + cD[3] * dt[2] + cD[4] * utdt;
  const double sum15 = l1a1 + l5a5 + l2a2;
  double c_ut[3], c_dt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    c_ut[k] = cD[1 + k] * sum15 + cD[4] * l2r * dt[k];
    c_dt[k] = (cD[1 + k] + cD[4] * ut[k]) * l2r;
  }
  double c_ct = (l5a5 - l1a1) * (cnt + cD[4] * unt);
  double c_unt = cD[4] * ct * (l5a5 - l1a1);
  double c_Ht = cD[4] * (l1a1 + l5a5);
  double c_q2 = cD[4] * 0.5 * l2a2;
  // products with the wave speeds
  const double c_a1 = c_l1a1 * s1, c_a5 = c_l5a5 * s5, c_a2 = c_l2a2 * l2;
  const double c_s1 = c_l1a1 * a1, c_s5 = c_l5a5 * a5;
  const double c_l2 = c_l2a2 * a2 + c_l2r * rt;
  double c_rt = c_l2r * l2;
  const double g1 = sgn_of(unt - ct), g5 = sgn_of(unt + ct), g2 = sgn_of(unt);
  c_unt += g1 * c_s1 + g5 * c_s5 + g2 * c_l2;
  c_ct += -g1 * c_s1 + g5 * c_s5;
  // tangential jump dt = du - dun n
  double c_du[3];
  double c_dun = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) { c_du[k] = c_dt[k]; c_dun -= c_dt[k] * nv[k]; }
  // wave strengths
  double c_dr = c_a2, c_dp = -c_a2 * ic2, c_ic2 = -c_a2 * dp;
  c_dp += 0.5 * (c_a1 + c_a5) * ic2;
  const double cdiff = 0.5 * (c_a5 - c_a1) * ic2;  // cotangent of rt ct dun
  c_rt += cdiff * ct * dun;
  c_ct += cdiff * rt * dun;
  c_dun += cdiff * rt * ct;
  c_ic2 += 0.5 * (c_a1 * A1 + c_a5 * A5);
#pragma unroll
  for (int k = 0; k < 3; ++k) { c_du[k] += c_dun * nv[k]; c_ut[k] += c_unt * nv[k]; }
  // Roe averages
  double c_c2 = -c_ic2 * ic2 * ic2 + c_ct * 0.5 * rc;
  c_Ht += gm1 * c_c2;
  c_q2 -= 0.5 * gm1 * c_c2;
#pragma unroll
  for (int k = 0; k < 3; ++k) c_ut[k] += 2.0 * ut[k] * c_q2;
  // the weights: d ut/d sL = iw (uL - ut), d Ht/d sL = iw (hL - Ht) (the same for R), d ut/d uL = sL iw
  double xL = c_Ht * (hL - Ht), xR = c_Ht * (hR - Ht);
  const double wL = sL * iw, wR = sR * iw;
  const double c_hL = c_Ht * wL, c_hR = c_Ht * wR;
  double cuL[3], cuR[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    xL += c_ut[k] * (L.u[k] - ut[k]);
    xR += c_ut[k] * (R.u[k] - ut[k]);
    cuL[k] = c_ut[k] * wL - c_du[k];
    cuR[k] = c_ut[k] * wR + c_du[k];
  }
  const double c_sL = c_rt * sR + iw * xL, c_sR = c_rt * sL + iw * xR;
  // enthalpies h = (E + p) ir
  double cpL = -c_dp + c_hL * L.ir, cpR = c_dp + c_hR * R.ir;
  double cirL = c_hL * EpL, cirR = c_hR * EpR;
#pragma unroll
  for (int v = 0; v < 5; ++v) { gL[v] = 0.0; gR[v] = 0.0; }
  gL[4] += c_hL * L.ir;
  gR[4] += c_hR * R.ir;
  gL[0] += -c_dr + c_sL * 0.5 * rsL;
  gR[0] += c_dr + c_sR * 0.5 * rsR;
  double cunL = 0.0, cunR = 0.0;
  flux_back(UL, L, nv, hF, cpL, cunL, gL);
  flux_back(UR, R, nv, hF, cpR, cunR, gR);
  side_back(UL, L, nv, gm1, cuL, cpL, cunL, cirL, gL);
  side_back(UR, R, nv, gm1, cuR, cpR, cunR, cirR, gR);
}

// ---------------------------------------------------------------------------------------------
// adjoint of the face kernel
// ---------------------------------------------------------------------------------------------
// Bound by the FP64 pipe (88 % busy). 64 threads per block, as in the face kernel: at 1500 to 3000 face points 18.5 us
// with 128, 17.0 with 64; at N = 7, 7^3 53.4 and 49.2 us; from 10^5 points on the same.
template <int SF>
__global__ void __launch_bounds__(FACE_THREADS) k_adj_face(const DgDevice d, const double *__restrict__ U,
                                                  const double *__restrict__ lam, double *__restrict__ slots) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.nF * nn) return;
  const int f = (int)(t / nn), pq = (int)(t % nn), p = pq % n, q = pq / n;
  const int *F5 = d.face + 5 * f;
  const int eL = F5[0], fL = F5[1], eR = F5[2], fR = F5[3], o = F5[4];
  int p2, q2;
  orient_map(o, p, q, p2, q2);
  const int nodeL = face_node(fL, p, q), nodeR = face_node(fR, p2, q2);
  const int pqR = p2 + n * q2;
  const double *nr = d.nrm + (size_t)f * 4 * nn + pq;
  double UL[5], UR[5], cF[5];
  load_state<double>(d, U, eL, nodeL, UL);
  load_state<double>(d, U, eR, nodeR, UR);
  const double iJL = d.invJ[(size_t)eL * nnn + nodeL], iJR = d.invJ[(size_t)eR * nnn + nodeR];
  const double sw = nr[3 * nn] * c_invw[0];  // w_0 = w_N
#pragma unroll
  for (int v = 0; v < 5; ++v)
    cF[v] = sw * (iJR * lam[((size_t)eR * 5 + v) * nnn + nodeR] - iJL * lam[((size_t)eL * 5 + v) * nnn + nodeL]);
  if (SF != SF_EC) {  // hand-written reverse mode
    const double nv[3] = {nr[0], nr[nn], nr[2 * nn]};
    double gL[5], gR[5];
    if (SF == SF_ROE) roe_vjp(UL, UR, nv, d.gamma, cF, gL, gR);
    else llf_vjp(UL, UR, nv, d.gamma, cF, gL, gR);
    double *oL = slots + ((size_t)eL * 6 + fL) * 5 * nn + pq;
    double *oR = slots + ((size_t)eR * 6 + fR) * 5 * nn + pqR;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      oL[k * nn] = gL[k];
      oR[k * nn] = gR[k];
    }
    return;
  }
  // entropy-conservative flux: forward-mode dual numbers through riemann<>
  using D5 = Dual<5>;
  const D5 nv[3] = {D5(nr[0]), D5(nr[nn]), D5(nr[2 * nn])};
  const D5 gam(d.gamma), zero(0.0);
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    D5 A[5], B[5], Fd[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      A[v] = D5(UL[v]);
      B[v] = D5(UR[v]);
      if (side == 0) A[v].d[v] = 1.0;
      else B[v].d[v] = 1.0;
    }
    riemann<D5>(SF, A, B, nv, gam, zero, zero, Fd);
    double *out = slots + ((size_t)(side ? eR : eL) * 6 + (side ? fR : fL)) * 5 * nn + (side ? pqR : pq);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      double gk = 0.0;
#pragma unroll
      for (int v = 0; v < 5; ++v) gk += cF[v] * Fd[v].d[k];
      out[k * nn] = gk;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// adjoint of the lifting + viscous flux + viscous divergence (Navier-Stokes)
// The flux is linear in the lifted gradients except for the work term u.tau, whose derivative
// needs the viscous stress tau at the state: the forward lifting records it per node (the record
// the reverse sweep keeps with each stage state), so no gradient is formed here.
//
// One thread per node. In FP64 the node's two D^T sweeps are 24 n products of ~120 others, on a pipe of two
// lanes per clock and SM (92 % busy, N = 5). They are formed in the fixed point of dg_fixed.cuh instead
// (3 IMAD.WIDE each, ~25 lanes per clock), from values at the element's largest per variable; an element whose
// values leave the range of the scales (infinities, NaN, magnitudes near the ends of FP64) keeps FP64 sweeps.
// Windows (value x scale, log2): D_mi / 32 < 62, a column sum of |D| / 32 <= 0.81 (N = 7); l and H < 60; one
// direction's cross sums < 62.4; results 2^-56 (2^-55 with three directions summed) of the largest value, where
// the FP64 sums round at 2^-53 of their partial sums, ~10 times the largest value.
// Per launch at N = 5, 12^3: 225 us with FP64 sweeps, 131 us (errors of the product against extended precision 0.77 to
// 0.95 of those with FP64 kernels).
// The diagonal of D in the second sweep, D_00 = -N(N+1)/4 = -D_NN, is the face term (1/w_b)(+-1/2): they cancel.
// shared memory per element: L[4][nnn] (l of momentum and energy), H[12][nnn] (cotangent of the
// direction-d reference derivative of w_q), as fixed-point values or (general path) doubles
// ---------------------------------------------------------------------------------------------
constexpr int ADJV_SLOTS = 16;
constexpr int ADJV_THREADS = round32(LIFT_EPB * nnn);
constexpr int ADJV_BLOCKS = ADJV_THREADS >= 512 ? 1 : 896 / ADJV_THREADS;  // per SM (bounds the registers)
constexpr int ADJV_DROP = 3;

// the neighbour's volume node facing face point (pp, qq) of element e's face f
__device__ __forceinline__ void neighbour_node(const DgDevice &d, size_t e, int f, int pp, int qq, int &nb, int &fnb,
                                               int &nbnode, int &nbpq) {
  const int *ef = d.ef + (e * 6 + f) * 4;
  nb = ef[0];
  fnb = ef[1];
  int p2, q2;
  orient_map(ef[2], pp, qq, p2, q2);
  nbnode = face_node(fnb, p2, q2);
  nbpq = p2 + n * q2;
}

// the largest |x| of an element (high word) for its threads' values x[4][K], into mx[4]
template <int K>
__device__ __forceinline__ void adjv_max(const double (&x)[K][4], bool on, int *mx) {
  constexpr bool WARP = LIFT_EPB == 1 || nnn % 32 == 0;  // a warp's nodes belong to one element
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int h = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) h = max(h, on ? fx_hi_abs(x[k][q]) : 0);
    if (WARP) {
      h = __reduce_max_sync(0xffffffffu, h);
      if (threadIdx.x % 32 == 0) atomicMax(mx + q, h);
    } else if (on) {
      atomicMax(mx + q, h);
    }
  }
}
// fixed-point exponents of the four variables; false: the element takes the FP64 sweeps
__device__ __forceinline__ bool adjv_scale(const int *mx, int E[4]) {
  bool ok = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ex = fx_exponent(mx[q]);
    E[q] = max(ex, 128);
    ok = ok && (mx[q] == 0 || (ex >= 128 && ex <= 1900));
  }
  return ok;
}
__device__ __forceinline__ long long adjv_store(double x, bool fx, int E) {
  return fx ? fx_from(x, E, ADJV_DROP) + FX_BIAS : __double_as_longlong(x);
}
// r[q] = sum_m D_mi x_q,m along a line (S at node 0 of it, q apart by nnn): fixed value, window a
__device__ __forceinline__ void adjv_sweep(const long long *S, int st, const int2 *row, int a, fx_t r[4]) {
  FxSum s[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) s[q] = fx_zero(a);
#pragma unroll
  for (int m = 0; m < n; ++m) {
    const FxD w = fx_const(row[m]);
#pragma unroll
    for (int q = 0; q < 4; ++q) fx_acc(s[q], w, fx_biased(S[q * nnn + m * st]));
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = fx_value(s[q], a);
}
__device__ __noinline__ double adjv_sweep_general(const long long *S, int st, int id) {
  double r = 0.0;
#pragma unroll 1
  for (int m = 0; m < n; ++m)
    if (m != id) r += c_D[m * n + id] * __longlong_as_double(S[m * st]);
  return r;
}

__global__ void __launch_bounds__(ADJV_THREADS, ADJV_BLOCKS)
    k_adj_visc(const DgDevice d, const double *__restrict__ U, const double *__restrict__ lam,
               const double *__restrict__ tau, double *__restrict__ cotW, double *__restrict__ sigma) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  long long *Ls = reinterpret_cast<long long *>(sm_raw);  // [EPB][4][nnn]
  long long *Hs = Ls + LIFT_EPB * 4 * nnn;                // [EPB][12][nnn]
  // D^T in shared memory, rows padded: the sweeps index it by the thread's own node, which would
  // serialise a constant-memory load
  __shared__ int2 sD[n][n + 1];
  __shared__ int s_mx[LIFT_EPB][2][4];
  for (int t = threadIdx.x; t < nn; t += blockDim.x) sD[t / n][t % n] = c_DT[t];
  for (int t = threadIdx.x; t < LIFT_EPB * 8; t += blockDim.x) (&s_mx[0][0][0])[t] = 0;
  __syncthreads();
  const int le = threadIdx.x / nnn < LIFT_EPB ? threadIdx.x / nnn : LIFT_EPB - 1, node = threadIdx.x % nnn;
  const int e = blockIdx.x * LIFT_EPB + le;
  const bool on = threadIdx.x < LIFT_EPB * nnn && e < d.nE;
  const size_t gi = (size_t)e * 5 * nnn + node;
  const int ijk[3] = {node % n, (node / n) % n, node / nn};
  double l[1][4], u[3], iJ;
  if (on) {
    const double ir = rcp_int(U[gi]);  // u as the lifting forms it
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = U[gi + (1 + k) * nnn] * ir;
    iJ = d.invJ[(size_t)e * nnn + node];
#pragma unroll
    for (int q = 0; q < 4; ++q) l[0][q] = -iJ * lam[gi + (1 + q) * nnn];
  }
  adjv_max<1>(l, on, s_mx[le][0]);
  __syncthreads();
  int E[4];
  bool fx = adjv_scale(s_mx[le][0], E);
  long long *L = Ls + le * 4 * nnn, *H = Hs + le * 12 * nnn;
  if (on) {
#pragma unroll
    for (int q = 0; q < 4; ++q) L[q * nnn + node] = adjv_store(l[0][q], fx, E[q]);
  }
  __syncthreads();
  double h[3][4], om[3];
  if (on) {
    // reverse seed: zeta[dd][q] = cotangent of the contravariant viscous flux Fv^dd_q at this node
    double zeta[3][4];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const int id = ijk[dd];
      const int st = dd == 0 ? 1 : dd == 1 ? n : nn;
      const int base = node - id * st;
      if (fx) {
        fx_t r[4];
        adjv_sweep(L + base, st, sD[id], 4, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) zeta[dd][q] = fx_to(-r[q], E[q] - 1079);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) zeta[dd][q] = -adjv_sweep_general(L + q * nnn + base, st, id);
      }
      if (id == 0 || id == N) {  // the neighbour's viscous divergence reads this node's flux
        const int f = 2 * dd + (id == N ? 1 : 0);
        const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
        int nb, fnb, nbnode, nbpq;
        neighbour_node(d, e, f, pp, qq, nb, fnb, nbnode, nbpq);
        const double sgf = (f & 1) ? 0.5 : -0.5;
        const double kn = c_invw[id] * sgf * -d.invJ[(size_t)nb * nnn + nbnode];  // (1/w_b)(+-1/2) l = -lam/J
#pragma unroll
        for (int q = 0; q < 4; ++q) zeta[dd][q] += kn * lam[((size_t)nb * 5 + 1 + q) * nnn + nbnode];
      }
    }
    double Ja[3][3];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd)
#pragma unroll
      for (int c = 0; c < 3; ++c) Ja[dd][c] = d.Ja[(((size_t)e * 3 + dd) * 3 + c) * nnn + node];
    // the lifting forms tau and the heat flux from J grad w with 1/J in mu and kappa; their
    // transposes carry the same factors, and with them the 1/J of H below
    const double mu = d.mu * iJ, kappa = d.kappa * iJ;
    const double *tr = tau + (size_t)e * 6 * nnn + node;
    const double txx = tr[0], tyy = tr[nnn], tzz = tr[2 * nnn], txy = tr[3 * nnn], txz = tr[4 * nnn],
                 tyz = tr[5 * nnn];
    const double ta[3][3] = {{txx, txy, txz}, {txy, tyy, tyz}, {txz, tyz, tzz}};
    // Z[c][q]: cotangent of the Cartesian viscous flux F_c,q (F_c,k = tau_kc; F_c,3 = u.tau_c + kappa dT/dx_c)
    double Z[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < 4; ++q) Z[c][q] = Ja[0][c] * zeta[0][q] + Ja[1][c] * zeta[1][q] + Ja[2][c] * zeta[2][q];
    double Y[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      om[k] = Z[0][3] * ta[k][0] + Z[1][3] * ta[k][1] + Z[2][3] * ta[k][2];
#pragma unroll
      for (int c = 0; c < 3; ++c) Y[k][c] = Z[c][k] + Z[c][3] * u[k];
    }
    const double trY = Y[0][0] + Y[1][1] + Y[2][2];
    // mu (Y + Y^T - 2/3 tr Y), symmetric
    double Gm[4][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Gm[k][k] = 2.0 * mu * (Y[k][k] - trY * (1.0 / 3.0));
#pragma unroll
      for (int c = 0; c < k; ++c) Gm[k][c] = Gm[c][k] = mu * (Y[k][c] + Y[c][k]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) Gm[3][c] = kappa * Z[c][3];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
#pragma unroll
      for (int q = 0; q < 4; ++q) h[dd][q] = Ja[dd][0] * Gm[q][0] + Ja[dd][1] * Gm[q][1] + Ja[dd][2] * Gm[q][2];
      const int id = ijk[dd];
      if (id == 0 || id == N) {
        const int f = 2 * dd + (id == N ? 1 : 0);
        const int pq = (dd == 0 ? ijk[1] : ijk[0]) + n * (dd == 2 ? ijk[1] : ijk[2]);
        const double hs = (id == N ? 0.5 : -0.5) * c_invw[id];
        double *sg = sigma + ((size_t)e * 6 + f) * 4 * nn + pq;
#pragma unroll
        for (int q = 0; q < 4; ++q) sg[q * nn] = hs * h[dd][q];
      }
    }
  }
  adjv_max<3>(h, on, s_mx[le][1]);
  __syncthreads();
  fx = adjv_scale(s_mx[le][1], E);
  if (on) {
#pragma unroll
    for (int dd = 0; dd < 3; ++dd)
#pragma unroll
      for (int q = 0; q < 4; ++q) H[(dd * 4 + q) * nnn + node] = adjv_store(h[dd][q], fx, E[q]);
  }
  __syncthreads();
  if (!on) return;
  double cw[4];
  if (fx) {
    fx_t c[4] = {0, 0, 0, 0};
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const int st = dd == 0 ? 1 : dd == 1 ? n : nn;
      fx_t r[4];
      adjv_sweep(H + dd * 4 * nnn + node - ijk[dd] * st, st, sD[ijk[dd]], 3, r);
#pragma unroll
      for (int q = 0; q < 4; ++q) c[q] += r[q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) cw[q] = fx_to(c[q], E[q] - 1078);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cw[q] = 0.0;
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        const int st = dd == 0 ? 1 : dd == 1 ? n : nn;
        cw[q] += adjv_sweep_general(H + (dd * 4 + q) * nnn + node - ijk[dd] * st, st, ijk[dd]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) cw[k] += om[k];
#pragma unroll
  for (int q = 0; q < 4; ++q) cotW[((size_t)e * 4 + q) * nnn + node] = cw[q];
}

// ---------------------------------------------------------------------------------------------
// transposed pair terms in FP64 (the general path)
// ---------------------------------------------------------------------------------------------
// one node's staged values for the transposed pair terms
struct AdjNode {
  double r, u, v, w, p, x, l[5], jx, jy, jz;
};

// the six primitive cotangents of the pair (i, m), shared by both nodes. The pair cotangents
// c_v = D'_im l_i,v + D'_mi l_m,v are D'_im t_v with t_v = l_i,v + (D_mi/D_im) l_m,v (the mass part's
// factor 2, D/4 against D/8, is in the staged l_0); D'_im = D_im/8 then scales phi, the pressure
// cotangent and F0 once instead of every c_v.
template <int VF>
__device__ __forceinline__ void adj_pair(const AdjNode &a, const AdjNode &b, double de, double dr, double g[6]) {
  const double Sr = a.r + b.r, Su = a.u + b.u, Sv = a.v + b.v, Sw = a.w + b.w;
  const double Sp = a.p + b.p, Sx = a.x + b.x;
  const double Sjx = a.jx + b.jx, Sjy = a.jy + b.jy, Sjz = a.jz + b.jz;
  const double t0 = a.l[0] + dr * b.l[0];
  const double t1 = a.l[1] + dr * b.l[1];
  const double t2 = a.l[2] + dr * b.l[2];
  const double t3 = a.l[3] + dr * b.l[3];
  const double t4 = a.l[4] + dr * b.l[4];
  const double Vp = Su * Sjx + Sv * Sjy + Sw * Sjz;
  const double F0 = de * (Sr * Vp);                                   // D'_im F0
  const double phi = de * (t0 + t1 * Su + t2 * Sv + t3 * Sw + t4 * Sx);  // d(c.F)/dF0
  double gV = phi * Sr, gP = de * (t1 * Sjx + t2 * Sjy + t3 * Sjz);
  if (VF == VF_KG) {
    const double c4 = de * t4;
    gV += 0.5 * c4 * Sp;
    gP += 0.5 * c4 * Vp;
  }
  g[0] = phi * Vp;
  g[1] = t1 * F0 + gV * Sjx;
  g[2] = t2 * F0 + gV * Sjy;
  g[3] = t3 * F0 + gV * Sjz;
  g[4] = gP;
  g[5] = t4 * F0;
}

// ---------------------------------------------------------------------------------------------
// adjoint of the volume kernel, its transposed pair terms in the 64-bit fixed point of dg_fixed.cuh
// (phases, lanes and general path as k_volume_fx). With the sums S = x_i + x_m and the pair cotangents
// t_v = Q_im (l_i,v / w_i - l_m,v / w_m) w_0 (D_im l_i + D_mi l_m = Q_im (l_i / w_i - l_m / w_m)), both
// nodes of a pair get the same cotangents of (rho, u, v, w, 4p, X):
//   phi = t_0 + t_k S_u,k + t_4 S_X, F0 = S_rho V, V = S_u . S_J, gV = phi S_rho (+ 2 t_4 S_p for KG):
//   (phi V, t_k F0 + gV S_J,k, t_k S_J,k (+ t_4 V / 2 for KG), t_4 F0), all times 1 / (8 w_0)
// (l_0 doubled: its split-form factor is D/4, the others' D/8). 25 products a pair (28 for KG) against
// ~49 FP64 instructions.
// ---------------------------------------------------------------------------------------------
struct FxAdj {
  int ok;
  int none;                            // no cotangent in the element: ok, the pair cotangents are zero
  int er, eu, ep, ex, e0, e1, e4;      // exponents: rho, u, p, X, l of mass, momentum, energy
  int e[3], top;                       // of the metric terms' directions, as FxScale
  int av, aa, ab, af, ag, a0, ak, ax;  // windows of V, t_k S_u,k, t_4 S_X, F0, phi S_rho and the outputs
  int pa, pb, p0;                      // right shifts of t_k S_u,k, t_4 S_X and t_0 to phi's scale
  int va, vb;                          // KG: right shifts of phi S_rho and t_4 S_p to gV's
  int kf, kv;                          // right shifts of F0 and gV before t_k F0 + gV S_J,k
  int ga, gb;                          // right shifts of t_k S_J,k and (KG) t_4 V to the output's scale
  int k0, k1, kp, kx;                  // cotangents are fixed value x 2^(k + e_d) / (8 w_0): rho, u, 4p, X
};

// upper bound of log2(2^a + 2^b) in 2^-20
__device__ __forceinline__ int fx_lsum(int a, int b) {
  const int d = abs(a - b) >> 20;
  return max(a, b) + (d == 0 ? 1048576 : d == 1 ? 613400 : d == 2 ? 337600 : d == 3 ? 178400 : 91800);
}

// Bounds (value x scale, log2): S_rho, S_p < 63, S_u, S_J, S_X, l differences < 61; t < 61. V, phi, F0 and gV fill at
// most 62.2 and a line's sum of each output at most 62.2, by windows and shifts from the element's maxima; the
// halved sum of three directions then stays below 63, and every group of cross sums h l' + l h' too.
template <int VF>
__device__ __forceinline__ FxAdj fx_adj_scales(const int *mx, int4 mj) {
  // mx: high words: rho max, rho min, |u| max, p max, p min, x max, x min (minima signed), |l| of mass, momentum, energy,
  // |u| + |v| + |w| max
  FxAdj s;
  s.er = fx_exponent(mx[0]); s.ep = fx_exponent(mx[3]); s.ex = fx_exponent(mx[5]);
  const int j0 = fx_exponent(mj.x), j1 = fx_exponent(mj.y), j2 = fx_exponent(mj.z);
  s.e[0] = fx_unit(mj.x); s.e[1] = fx_unit(mj.y); s.e[2] = fx_unit(mj.z);
  const int jt = max(s.e[0], max(s.e[1], s.e[2])), jb = min(s.e[0], min(s.e[1], s.e[2]));
  s.top = jt - jb <= FX_NEAR ? jt : -1000;
  constexpr int ej = 1023;
  s.eu = max(fx_exponent(mx[2]), (1996 - s.er + s.ep) >> 1);
  // exponents of l: a group far below the others' shares of phi takes a scale 2^-40 of theirs
  s.none = (mx[7] | mx[8] | mx[9]) == 0;
  const int r0 = s.none ? 1023 : fx_exponent(mx[7]), r1 = s.none ? 1023 : fx_exponent(mx[8]),
            r4 = s.none ? 1023 : fx_exponent(mx[9]);
  const int ph = max(r0, max(r1 + s.eu, r4 + s.ex) - 1023);
  s.e0 = max(r0, ph - 40); s.e1 = max(r1, ph - s.eu + 1023 - 40); s.e4 = max(r4, ph - s.ex + 1023 - 40);
  const int lo = min(min(min(s.er, s.ep), min(s.ex, min(j0, min(j1, j2)))), min(min(s.e0, s.e1), s.e4));
  const int hi = max(max(max(s.er, s.ep), max(s.ex, max(j0, max(j1, j2)))), max(max(max(s.e0, s.e1), s.e4), s.eu));
  const int sr = 1084 - s.er, su = 1082 - s.eu, sp = 1084 - s.ep, sx = 1082 - s.ex, sj = 1082 - ej;
  const int l0 = 1082 - s.e0, l1 = 1082 - s.e1, l4 = 1082 - s.e4;
  // log2 bounds in 2^-20: of sums S and differences of l (twice the maxima), then of the products
  constexpr int L = 1 << 20, LIM = (int)(62.2 * L);
  const int lr = fx_lg(mx[0]) + L, lu = max(fx_lg(mx[2]), (s.eu - 1023) << 20) + L, lp = fx_lg(mx[3]) + L,
            lx = fx_lg(mx[5]) + L, lj = 2 * L, lv = lu + mj.w + L;  // (|Ja^d| < 2 in its units)
  const int t0 = max(fx_lg(mx[7]), (s.e0 - 1023) << 20) + L, t1 = max(fx_lg(mx[8]), (s.e1 - 1023) << 20) + L,
            t4 = max(fx_lg(mx[9]), (s.e4 - 1023) << 20) + L;
  const int la = t1 + max(fx_lg(mx[10]), (s.eu - 1023) << 20) + L, lb = t4 + lx, lf = lr + lv,
            lphi = fx_lsum(fx_lsum(la, lb), t0);
  auto window = [&](int bound, int scale) { return min(max(((LIM - bound) >> 20) - scale, 0), 10); };
  s.av = window(lv, su + sj - 64);
  const int sv = su + sj - 64 + s.av;
  s.aa = window(la, l1 + su - 64);
  s.ab = window(lb, l4 + sx - 64);
  const int fa = l1 + su - 64 + s.aa, fb = l4 + sx - 64 + s.ab;
  const int sf = min(min(min(fa, fb), l0), (LIM - lphi) >> 20);  // phi
  s.pa = min(fa - sf, 62); s.pb = min(fb - sf, 62); s.p0 = min(l0 - sf, 62);
  s.af = window(lf, sr + sv - 64);
  const int sF = sr + sv - 64 + s.af;  // F0
  int lg = lphi + lr;
  s.ag = window(lg, sf + sr - 64);
  int sg = sf + sr - 64 + s.ag;  // gV
  s.va = s.vb = 0;
  if (VF == VF_KG) {
    const int a = sg, b = l4 + sp - 62 - 1;  // t_4 S_p with window 2; the factor 2
    lg = fx_lsum(lg, t4 + lp + L);
    sg = min(min(a, b), (LIM - lg) >> 20);
    s.va = min(a - sg, 62); s.vb = min(b - sg, 62);
  }
  const int lk = fx_lsum(t1 + lf, lg + lj) + FX_LGR, c0 = sf + sv - 64, cx = l4 + sF - 64;
  int ka = l1 + sF - 64, kb = sg + sj - 64, sk = min(ka, kb);
  s.kf = min(ka - sk, 62); s.kv = min(kb - sk, 62);
  s.ak = window(lk, sk);
  s.a0 = window(lphi + lv + FX_LGR, c0);
  s.ax = window(t4 + lf + FX_LGR, cx);
  const int pA = l1 + sj - 61, pB = l4 + sv - 62 + 1;  // t_k S_J,k with window 3; t_4 V with window 2, the factor 1/2
  int lP = t1 + mj.w + L + FX_LGR, sP = pA;
  if (VF == VF_KG) {
    lP = fx_lsum(lP, t4 + lv - L + FX_LGR);
    sP = min(sP, pB);
  }
  sP = min(sP, (LIM - lP) >> 20);
  s.ga = min(pA - sP, 62);
  s.gb = VF == VF_KG ? min(pB - sP, 62) : 0;
  s.k0 = 1 - (c0 + s.a0); s.k1 = 1 - (sk + s.ak); s.kp = 1 - sP; s.kx = 1 - (cx + s.ax);  // (halved sums)
  const int km = max(max(abs(s.k0), abs(s.k1)), max(abs(s.kp), abs(s.kx)));
  s.ok = mx[1] > 0 && mx[4] > 0 && mx[6] > 0 && s.er - (mx[1] >> 20) <= 8 && s.ep - (mx[4] >> 20) <= 8 &&
         s.ex - (mx[6] >> 20) <= 8 && lo >= 850 && hi <= 1200 && km <= 700 && mj.w < FX_FAR;
  return s;
}

struct FxAdjNode {
  fx_t r, u, v, w, p, x, jx, jy, jz, l[5];
};
// element slots (FX_PS each): 0-5 rho, u, v, w, p, X; 6 + 8 dir + c: metric terms (c < 3), weighted l (c = 3 + v);
// a line's six cotangents of node i then replace the first six of its direction's eight
constexpr int FXA_SLOTS = 30;
template <int VF>
__device__ __forceinline__ FxAdjNode fx_adj_load(const fx_t *__restrict__ S, int a, int dir) {
  const fx_t *J = S + (6 + 8 * dir) * FX_PS + a;
  FxAdjNode q{S[a], S[FX_PS + a], S[2 * FX_PS + a], S[3 * FX_PS + a], VF == VF_KG ? S[4 * FX_PS + a] : 0,
              S[5 * FX_PS + a], J[0], J[FX_PS], J[2 * FX_PS]};
#pragma unroll
  for (int v = 0; v < 5; ++v) q.l[v] = J[(3 + v) * FX_PS];
  return q;
}

template <int VF>
__device__ __forceinline__ void fx_adj_pair(const FxAdjNode &a, const FxAdjNode &b, FxD q, const FxAdj &c, fx_t g[6]) {
  const FxD Sj[3] = {fx_biased(a.jx + b.jx), fx_biased(a.jy + b.jy), fx_biased(a.jz + b.jz)};
  const FxD Su[3] = {fx_biased(a.u + b.u), fx_biased(a.v + b.v), fx_biased(a.w + b.w)};
  const FxD Sr = fx_biased(a.r + b.r);
  fx_t t0;
  FxD t[4];  // momentum, energy
  {
    FxSum s = fx_zero(1);
    fx_acc(s, q, fx_split(a.l[0] - b.l[0]));
    t0 = fx_value(s, 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s = fx_zero_biased(1);
      fx_acc(s, q, fx_split(a.l[1 + k] - b.l[1 + k]));
      t[k] = fx_biased(fx_value(s, 1));
    }
  }
  FxSum s = fx_zero_biased(c.av), z;
#pragma unroll
  for (int k = 0; k < 3; ++k) fx_acc(s, Su[k], Sj[k]);
  const FxD V = fx_biased(fx_value(s, c.av));
  s = fx_zero(c.aa);
#pragma unroll
  for (int k = 0; k < 3; ++k) fx_acc(s, t[k], Su[k]);
  z = fx_zero(c.ab);
  fx_acc(z, t[3], fx_biased(a.x + b.x));
  const FxD phi = fx_split(fx_shr(fx_value(s, c.aa), c.pa) + fx_shr(fx_value(z, c.ab), c.pb) + fx_shr(t0, c.p0));
  s = fx_zero(c.a0);
  fx_acc(s, phi, V);
  g[0] = fx_value(s, c.a0);
  s = fx_zero(c.af);
  fx_acc(s, Sr, V);
  const fx_t F0 = fx_value(s, c.af);
  const FxD Fk = fx_split(fx_shr(F0, c.kf));
  s = fx_zero(c.ag);
  fx_acc(s, phi, Sr);
  fx_t gv = fx_value(s, c.ag);
  s = fx_zero(3);
#pragma unroll
  for (int k = 0; k < 3; ++k) fx_acc(s, t[k], Sj[k]);
  g[4] = fx_shr(fx_value(s, 3), c.ga);
  if (VF == VF_KG) {
    z = fx_zero(2);
    fx_acc(z, t[3], fx_biased(a.p + b.p));
    gv = fx_shr(gv, c.va) + fx_shr(fx_value(z, 2), c.vb);
    z = fx_zero(2);
    fx_acc(z, t[3], V);
    g[4] += fx_shr(fx_value(z, 2), c.gb);
  }
  const FxD gV = fx_split(fx_shr(gv, c.kv));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    s = fx_zero(c.ak);
    fx_acc(s, t[k], Fk);
    fx_acc(s, gV, Sj[k]);
    g[1 + k] = fx_value(s, c.ak);
  }
  s = fx_zero(c.ax);
  fx_acc(s, t[3], fx_split(F0));
  g[5] = fx_value(s, c.ax);
}

// general path: the pair phase in FP64 on the staged doubles (slots as in the fixed-point phase; 4 p, l unweighted). Whole
// product with every element general, N = 7, 12^3, Euler: 1327 us, 1832 with a thread per node that formed all its pairs
// itself, 1240 with the former FP64 line kernel; N = 5, Navier-Stokes: 805, 941 and 941 us.
template <int VF>
__device__ __noinline__ void fx_adj_general_lines(double *S) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int gr = threadIdx.x >> 5; gr < 3 * FX_GROUPS; gr += FX_THREADS / 32) {
    const FxLine q = fx_line(gr, lane);
    double *Sl = S + q.lel * FXA_SLOTS * FX_PS + q.pb;
    auto load = [&](int m) {
      const double *P = Sl + m * q.ps, *J = P + (6 + 8 * q.dir) * FX_PS;
      AdjNode a{P[0], P[FX_PS], P[2 * FX_PS], P[3 * FX_PS], P[4 * FX_PS], P[5 * FX_PS]};
#pragma unroll
      for (int v = 0; v < 5; ++v) a.l[v] = J[(3 + v) * FX_PS];
      a.jx = J[0]; a.jy = J[FX_PS]; a.jz = J[2 * FX_PS];
      return a;
    };
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int s = 1; s <= n / 2; ++s) {
      const int m = q.idx + s < n ? q.idx + s : q.idx + s - n, j = q.idx >= s ? q.idx - s : q.idx - s + n;
      double g[6];
      adj_pair<VF>(load(q.idx), load(m), c_De[q.idx * n + m], c_Dr[q.idx * n + m], g);
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        acc[v] += g[v];
        if (2 * s != n) acc[v] += __shfl_sync(0xffffffffu, g[v], q.l0 + j);
      }
    }
    __syncwarp();
    if (q.own) {
#pragma unroll
      for (int v = 0; v < 6; ++v) Sl[(6 + 8 * q.dir + v) * FX_PS + q.idx * q.ps] = acc[v];
    }
  }
}

constexpr size_t FXA_SMEM = sizeof(fx_t) * FX_EPB * FXA_SLOTS * FX_PS;
constexpr int FXA_MINB = 704 / FX_THREADS < 1 ? 1 : 704 / FX_THREADS;  // >= 80 registers per thread

// One thread per node. The CTAs per SM give 80 registers at N = 3..5 (140 B spilled; with two thirds of the CTAs
// and no spill N = 5 is 20 % slower, N = 3 3 % faster). Measured per launch, Pirozzoli + Navier-Stokes N = 5, 12^3:
// 0.166 ms against 0.395 with FP64 line threads; KG Euler N = 3, 21 x 18 x 15: 94 against 241 us. Bound by issue and
// the FMA-heavy pipe, like k_volume_fx.
template <int VF>
__global__ void __launch_bounds__(FX_THREADS, FXA_MINB) k_adj_volume(const DgDevice d, const double *__restrict__ U,
                                                              const double *lam, const double *__restrict__ fslots,
                                                              const double *__restrict__ cotW,
                                                              const double *__restrict__ sigma, double *out,
                                                              double *gbar, int mode, double dt, double A, double B,
                                                              int update_g) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  fx_t *S = reinterpret_cast<fx_t *>(sm_raw);  // [EPB][FXA_SLOTS][FX_PS]
  __shared__ int s_mx[FX_EPB][11];
  __shared__ FxAdj s_sc[FX_EPB];
  __shared__ int2 s_rho[FX_H], s_Q[nn];
  const int e0 = blockIdx.x * FX_EPB, tid = threadIdx.x;
  const double gm1 = d.gamma - 1.0;
  for (int t = tid; t < FX_EPB * 11; t += FX_THREADS) {
    const int k = t % 11;
    s_mx[t / 11][k] = (k == 1 || k == 4 || k == 6) ? 0x7fffffff : 0;
  }
  for (int t = tid; t < FX_H; t += FX_THREADS) s_rho[t] = c_rho[t * FX_H];  // w_0 / w
  for (int t = tid; t < nn; t += FX_THREADS) s_Q[t] = c_Qx[t];
  __syncthreads();
  const int le = tid / nnn, node = tid % nnn, e = e0 + le;
  const bool on = tid < FX_EPB * nnn && e < d.nE;
  const int ijk[3] = {node % n, (node / n) % n, node / nn};
  double r = 1.0, ir = 1.0, u[3], p = 1.0, X = 1.0, l[5];
  {
    int h[11] = {0, 0x7fffffff, 0, 0, 0x7fffffff, 0, 0x7fffffff, 0, 0, 0, 0};
    if (on) {
      double Uv[5];
      load_state<double>(d, U, e, node, Uv);
      r = Uv[0];
      ir = rcp_int(r);
#pragma unroll
      for (int k = 0; k < 3; ++k) u[k] = Uv[1 + k] * ir;
      p = gm1 * (Uv[4] - 0.5 * (Uv[1] * u[0] + Uv[2] * u[1] + Uv[3] * u[2]));
      if (!(r > 0.0) || !(p > 0.0) || !isfinite(Uv[4])) flag_set(d.flag, 1);
      X = VF == VF_PIR ? (Uv[4] + p) * ir : Uv[4] * ir;
      const double miJ = -d.invJ[(size_t)e * nnn + node];
      // l = -lambda/J, the mass component doubled
#pragma unroll
      for (int k = 0; k < 5; ++k) l[k] = (k == 0 ? 2.0 * miJ : miJ) * lam[((size_t)e * 5 + k) * nnn + node];
      h[0] = fx_hi_abs(r); h[1] = __double2hiint(r);
      h[2] = max(max(fx_hi_abs(u[0]), fx_hi_abs(u[1])), fx_hi_abs(u[2]));
      h[3] = fx_hi_abs(p); h[4] = __double2hiint(p);
      h[5] = fx_hi_abs(X); h[6] = __double2hiint(X);
      h[7] = fx_hi_abs(l[0]);
      h[8] = max(max(fx_hi_abs(l[1]), fx_hi_abs(l[2])), fx_hi_abs(l[3]));
      const int low = __double2loint(l[0]) | __double2loint(l[1]) | __double2loint(l[2]) | __double2loint(l[3]) | __double2loint(l[4]);
      h[9] = max(fx_hi_abs(l[4]), low != 0 ? 1 : 0);  // (all three zero: no cotangent, subnormal ones included)
      h[10] = fx_hi_abs(fabs(u[0]) + fabs(u[1]) + fabs(u[2]));
    }
    bool each = on;
    if (FX_EPB == 1) {
#pragma unroll
      for (int k = 0; k < 11; ++k)
        h[k] = (k == 1 || k == 4 || k == 6) ? __reduce_min_sync(0xffffffffu, h[k]) : __reduce_max_sync(0xffffffffu, h[k]);
      each = (tid & 31) == 0 && on;
    }
    if (each) {
#pragma unroll
      for (int k = 0; k < 11; ++k) {
        if (k == 1 || k == 4 || k == 6) atomicMin(&s_mx[le][k], h[k]);
        else atomicMax(&s_mx[le][k], h[k]);
      }
    }
  }
  __syncthreads();
  int good = 1;
  if (tid < FX_EPB && e0 + tid < d.nE) {
    s_sc[tid] = fx_adj_scales<VF>(s_mx[tid], d.jmax[e0 + tid]);
    good = s_sc[tid].ok;
  }
  const bool ok = __syncthreads_and(good);
  // a block without a cotangent has no pair terms (most of them, for a product with a pointwise or wall-local quantity)
  bool none = ok;
#pragma unroll
  for (int k = 0; k < FX_EPB; ++k) none = none && (e0 + k >= d.nE || s_sc[k].none);
  if (ok && !none) {
    if (on) {
      const FxAdj &c = s_sc[le];
      constexpr fx_t HB = FX_BIAS / 2;
      fx_t *Se = S + le * FXA_SLOTS * FX_PS + fx_idx(node);
      Se[0] = fx_from(r, c.er, 1) + HB;
#pragma unroll
      for (int k = 0; k < 3; ++k) Se[(1 + k) * FX_PS] = fx_from(u[k], c.eu, 3) + HB;
      if (VF == VF_KG) Se[4 * FX_PS] = fx_from(p, c.ep, 1) + HB;
      Se[5 * FX_PS] = fx_from(X, c.ex, 3) + HB;
      const double *Je = d.Ja + (size_t)e * 9 * nnn + node;
#pragma unroll
      for (int k = 0; k < 9; ++k) Se[(6 + 8 * (k / 3) + k % 3) * FX_PS] = fx_from(__ldg(Je + k * nnn), 1023 + c.e[k / 3], 3) + HB;
      FxD lf[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) lf[v] = fx_split(fx_from(l[v], v == 0 ? c.e0 : v < 4 ? c.e1 : c.e4, 3));
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        const FxD w = fx_const(s_rho[min(ijk[dd], N - ijk[dd])]);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          FxSum s = fx_zero(2);
          fx_acc(s, w, lf[v]);
          Se[(9 + 8 * dd + v) * FX_PS] = fx_value(s, 2);
        }
      }
    }
    __syncthreads();
    const int lane = tid & 31;
    for (int gr = tid >> 5; gr < 3 * FX_GROUPS; gr += FX_THREADS / 32) {
      const FxLine q = fx_line(gr, lane);
      const int dir = q.dir, idx = q.idx, l0 = q.l0, lel = q.lel, pb = q.pb, ps = q.ps;
      fx_t *Sl = S + lel * FXA_SLOTS * FX_PS;
      const FxAdjNode ni = fx_adj_load<VF>(Sl, pb + idx * ps, dir);
      fx_t acc[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 1
      for (int s = 1; s <= n / 2; ++s) {
        const int m = idx + s < n ? idx + s : idx + s - n;
        fx_t g[6];
        fx_adj_pair<VF>(ni, fx_adj_load<VF>(Sl, pb + m * ps, dir), fx_const(s_Q[idx * n + m]), s_sc[lel], g);
        const int src = l0 + (idx >= s ? idx - s : idx - s + n);
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          acc[v] += g[v];
          if (2 * s != n) acc[v] += __shfl_sync(0xffffffffu, g[v], src);
        }
      }
      __syncwarp();
      if (q.own) {
#pragma unroll
        for (int v = 0; v < 6; ++v) Sl[(6 + 8 * dir + v) * FX_PS + pb + idx * ps] = acc[v];
      }
    }
  } else if (on && !ok) {
    double *Se = reinterpret_cast<double *>(S) + le * FXA_SLOTS * FX_PS + fx_idx(node);
    const double *Je = d.Ja + (size_t)e * 9 * nnn + node;
    Se[0] = r; Se[4 * FX_PS] = 4.0 * p; Se[5 * FX_PS] = X;
#pragma unroll
    for (int k = 0; k < 3; ++k) Se[(1 + k) * FX_PS] = u[k];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
#pragma unroll
      for (int k = 0; k < 3; ++k) Se[(6 + 8 * dd + k) * FX_PS] = __ldg(Je + (3 * dd + k) * nnn);
#pragma unroll
      for (int v = 0; v < 5; ++v) Se[(9 + 8 * dd + v) * FX_PS] = l[v];
    }
  }
  if (!ok) {
    __syncthreads();
    fx_adj_general_lines<VF>(reinterpret_cast<double *>(S));
  }
  __syncthreads();
  if (!on) return;
  double gp[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (ok && !none) {
    const fx_t *Se = S + le * FXA_SLOTS * FX_PS + fx_idx(node);
    const FxAdj &c = s_sc[le];
    const double w8 = 0.125 * c_invw[0];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const int k = v == 0 ? c.k0 : v < 4 ? c.k1 : v == 4 ? c.kp : c.kx;
      const fx_t a = Se[(6 + v) * FX_PS], b = Se[(14 + v) * FX_PS], z = Se[(22 + v) * FX_PS];
      if (c.top != -1000)
        gp[v] = w8 * fx_to((a >> (1 + c.top - c.e[0])) + (b >> (1 + c.top - c.e[1])) + (z >> (1 + c.top - c.e[2])), k + c.top);
      else
        gp[v] = w8 * (fx_to(a, k - 1 + c.e[0]) + fx_to(b, k - 1 + c.e[1]) + fx_to(z, k - 1 + c.e[2]));
    }
  } else if (!ok) {
    const double *Se = reinterpret_cast<const double *>(S) + le * FXA_SLOTS * FX_PS + fx_idx(node);
#pragma unroll
    for (int v = 0; v < 6; ++v) gp[v] = Se[(6 + v) * FX_PS] + Se[(14 + v) * FX_PS] + Se[(22 + v) * FX_PS];
  }
  const bool ns = d.equations == 1;
  const double iR = 1.0 / d.R;
  double g_r = gp[0], g_u[3] = {gp[1], gp[2], gp[3]}, g_p = 4.0 * gp[4];
  const double g_x = gp[5];
  if (ns) {  // cotangents of (u, v, w, T) from the viscous adjoint, own part + the neighbours' face shares
    double cw[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) cw[q] = cotW[((size_t)e * 4 + q) * nnn + node];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const int id = ijk[dd];
      if (id != 0 && id != N) continue;
      const int f = 2 * dd + (id == N ? 1 : 0);
      const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
      int nb, fnb, nbnode, nbpq;
      neighbour_node(d, e, f, pp, qq, nb, fnb, nbnode, nbpq);
      const double *sg = sigma + ((size_t)nb * 6 + fnb) * 4 * nn + nbpq;
#pragma unroll
      for (int q = 0; q < 4; ++q) cw[q] += sg[q * nn];
    }
    g_u[0] += cw[0];
    g_u[1] += cw[1];
    g_u[2] += cw[2];
    g_p += cw[3] * ir * iR;         // T = p / (rho R)
    g_r -= cw[3] * p * ir * ir * iR;
  }
  // chain to U = (rho, m, E): u = m / rho, p = (gamma-1)(E - |m|^2 / (2 rho)), X = h = (E + p)/rho
  // (Pirozzoli) or e = E/rho (KG). With gx = g_X/rho, p reaches U with weight a = (gamma-1) g_p, and
  // for h also through E + p: a = (gamma-1)(g_p + gx), and dh/dE = gamma/rho = (gamma-1)/rho + 1/rho
  const double q2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double gx = g_x * ir;
  const double a = VF == VF_PIR ? gm1 * (g_p + gx) : gm1 * g_p;
  double gU[5];
  gU[0] = g_r - ir * (g_u[0] * u[0] + g_u[1] * u[1] + g_u[2] * u[2]) + (0.5 * a) * q2 - gx * X;
#pragma unroll
  for (int k = 0; k < 3; ++k) gU[1 + k] = ir * g_u[k] - a * u[k];
  gU[4] = a + gx;
  // advective surface terms: transposed Riemann-flux Jacobians in this element's face slots
#pragma unroll
  for (int dd = 0; dd < 3; ++dd) {
    const int id = ijk[dd];
    if (id != 0 && id != N) continue;
    const int f = 2 * dd + (id == N ? 1 : 0);
    const int pq = (dd == 0 ? ijk[1] : ijk[0]) + n * (dd == 2 ? ijk[1] : ijk[2]);
    const double *fs = fslots + ((size_t)e * 6 + f) * 5 * nn + pq;
#pragma unroll
    for (int v = 0; v < 5; ++v) gU[v] += fs[v * nn];
  }
  const size_t gi = (size_t)e * 5 * nnn + node;
  if (mode == 0) {
#pragma unroll
    for (int v = 0; v < 5; ++v) out[gi + v * nnn] = gU[v];
  } else {  // reverse LSERK stage: Ubar += dt * VJP; gbar = A gbar + B Ubar (gbar is lam, read above)
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double ub = out[gi + v * nnn] + dt * gU[v];
      out[gi + v * nnn] = ub;
      if (update_g) gbar[gi + v * nnn] = A * gbar[gi + v * nnn] + B * ub;
    }
  }
}

// gradient of the kinetic-energy integral sum_e sum_ijk w_i w_j w_k J rho |u|^2 / 2
__global__ void __launch_bounds__(256) k_ke_grad(const DgDevice d, const double *__restrict__ U,
                                                 double *__restrict__ grad) {
  const long long total = (long long)d.nE * nnn;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const size_t e = (size_t)(t / nnn);
    const int node = (int)(t % nnn);
    const double wq = c_w[node % n] * c_w[(node / n) % n] * c_w[node / nn] * d.J[t];
    const double *Ue = U + e * 5 * nnn + node;
    const double ir = 1.0 / Ue[0];
    const double u = Ue[nnn] * ir, v = Ue[2 * nnn] * ir, w = Ue[3 * nnn] * ir;
    double *G = grad + e * 5 * nnn + node;
    G[0] = -0.5 * wq * (u * u + v * v + w * w);
    G[nnn] = wq * u;
    G[2 * nnn] = wq * v;
    G[3 * nnn] = wq * w;
    G[4 * nnn] = 0.0;
  }
}

// ---------------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------------
void launch_adj_face(const DgDevice &d, const double *U, const double *lam, double *slots, cudaStream_t s) {
  const long long pts = (long long)d.nF * nn;
  const unsigned grid = (unsigned)((pts + FACE_THREADS - 1) / FACE_THREADS);
  switch (d.sflux) {
    case SF_LLF: k_adj_face<SF_LLF><<<grid, FACE_THREADS, 0, s>>>(d, U, lam, slots); break;
    case SF_ROE: k_adj_face<SF_ROE><<<grid, FACE_THREADS, 0, s>>>(d, U, lam, slots); break;
    default: k_adj_face<SF_EC><<<grid, FACE_THREADS, 0, s>>>(d, U, lam, slots); break;
  }
}

void launch_adj_visc(const DgDevice &d, const double *U, const double *lam, const double *tau, double *cotW,
                     double *sigma, cudaStream_t s) {
  const size_t smem = sizeof(double) * LIFT_EPB * ADJV_SLOTS * nnn;
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_adj_visc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  k_adj_visc<<<(d.nE + LIFT_EPB - 1) / LIFT_EPB, ADJV_THREADS, smem, s>>>(d, U, lam, tau, cotW, sigma);
}

template <int VF>
void launch_adj_volume_t(const DgDevice &d, const double *U, const double *lam, const double *fslots,
                         const double *cotW, const double *sigma, double *out, double *gbar, int mode, double dt,
                         double A, double B, int update_g, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_adj_volume<VF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FXA_SMEM);
    attr_set = true;
  }
  k_adj_volume<VF><<<(d.nE + FX_EPB - 1) / FX_EPB, FX_THREADS, FXA_SMEM, s>>>(d, U, lam, fslots, cotW, sigma, out,
                                                                            gbar, mode, dt, A, B, update_g);
}

void launch_adj_volume(const DgDevice &d, const double *U, const double *lam, const double *fslots,
                       const double *cotW, const double *sigma, double *out, double *gbar, int mode, double dt,
                       double A, double B, int update_g, cudaStream_t s) {
  if (d.vflux == VF_KG)
    launch_adj_volume_t<VF_KG>(d, U, lam, fslots, cotW, sigma, out, gbar, mode, dt, A, B, update_g, s);
  else
    launch_adj_volume_t<VF_PIR>(d, U, lam, fslots, cotW, sigma, out, gbar, mode, dt, A, B, update_g, s);
}

void launch_ke_grad(const DgDevice &d, const double *U, double *grad, cudaStream_t s) {
  k_ke_grad<<<8 * 152, 256, 0, s>>>(d, U, grad);
}

}  // namespace
