// dg_kernels.cuh -- sm_103a kernels of the split-form DGSEM right-hand side for ONE polynomial
// degree. Included by dg_kernels_nN.cu with DG_N defined; everything lives in an anonymous
// namespace so each translation unit has its own constant-memory tables.
//
// Per RK stage (Sec. 2; Sec. 4.1):
//   [indicator -> spread]   modified Persson indicator on rho*p (Sec. 4.1, Eq. (7)), alpha per element
//   face                    Riemann flux s F*(U_L, U_R, n) once per face point (Roe / LLF / EC),
//                           BR1 face jumps w* - w for the lifting (Navier-Stokes)
//   [lift]                  BR1 gradients of (u, v, w, T) and the contravariant viscous flux
//   volume                  split-form flux differencing along the three line families, viscous
//                           divergence, surface terms, FV subcell operator + blend (Sec. 4.1,
//                           Eq. (6)), Jacobian, and the fused LSERK(5,4) stage update
//
// Algebra used by the volume kernel (exact identities of the LGL/SBP operator): with
// D_00 = -1/(2 w_0), D_NN = 1/(2 w_N) and zero interior diagonal, the diagonal volume term
// 2 D_ii F(U_i) cancels the -F(U_i)/w_b part of the strong-form surface term, so the kernel
// sums off-diagonal pairs only and adds (1/w_b) F*_out at boundary nodes; for the viscous
// (BR1 central) flux the same cancellation leaves -(1/(2 w_b)) phi_nb, the neighbour's outward
// normal viscous flux. Pair symmetry F#(U_i,U_m) = F#(U_m,U_i) halves the two-point fluxes.
//
// FP64 path: the volume operator (KG and Pirozzoli, with or without the blend), the lifting, the indicator and the
// adjoint's volume and viscous kernels form their sums in 64-bit fixed point on the integer pipes (dg_fixed.cuh,
// dg_fixed_lift.cuh, dg_adjoint.cuh): this GPU's FP64 pipe takes 2 lanes per clock and SM, a 32 x 32 + 64-bit integer
// multiply-add 25, so a product in three of those costs a quarter of an FMA. k_volume below serves FP64 for the EC and
// central fluxes.
//
// Arithmetic type R: double for the FP64 path; float for the FP32-bulk path, where the flux,
// lifting and accumulation arithmetic is FP32 while U is read as FP64, metrics and Jacobian are
// computed in FP64 (the kernels read an FP32 rounding of Ja), and the LSERK register and state
// accumulate in FP64 (the FP32 kernels of dg_fp32.cuh form the stage increment as an FP32 product). In FP32 the state is carried with E' = E - p_ref/(gamma-1) so that the
// pressure p' = p - p_ref is formed from O(1) numbers; the momentum flux uses p' throughout
// (volume, surface and subcell fluxes). The constant p_ref part of that flux contributes
// p_ref times the discrete metric identity sum_d D_d Ja^d, which is zero, so the shift is exact.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "dg_convert.cuh"
#include "dg_internal.h"
#include "dg_invariants_node.cuh"
#include "dg_log.cuh"
#include "dg_recip.cuh"
#include "dg_wall.cuh"

#ifndef DG_N
#error "define DG_N before including dg_kernels.cuh"
#endif

namespace {

constexpr int N = DG_N;
constexpr int n = N + 1;
constexpr int nn = n * n;
constexpr int nnn = nn * n;
constexpr int PS = n * (n + 1) * n;  // padded stride of one staged node quantity

__constant__ double c_D[nn];      // D_im
__constant__ double c_D2[nn];     // 2 D_im, zero diagonal
__constant__ double c_Dq[nn];     // D_im / 4 (scaled mass flux), zero diagonal
__constant__ double c_De[nn];     // D_im / 8 (scaled momentum / energy flux), zero diagonal
__constant__ double c_Dr[nn];     // D_mi / D_im (i != m; the LGL D has no zero off the diagonal), zero diagonal
__constant__ double c_w[n], c_invw[n], c_xi[n], c_xh[n + 1];
__constant__ double c_ihx[n];  // 1 / (xi_i - xi_{i-1}), i = 1..N (minmod slopes)
// even-odd halves of the zero-diagonal D (n even, h = n/2): the LGL D is centro-antisymmetric,
// D_{N-i,N-m} = -D_im, so y = D' f splits into VP (f_m + f_{N-m}) and VM (f_m - f_{N-m}), m < h:
// VP_im = (D'_im + D'_{i,N-m}) / 2, VM_im = (D'_im - D'_{i,N-m}) / 2, y_i = A_i + B_i, y_{N-i} = B_i - A_i
constexpr int EO_H = (n % 2 == 0) ? n / 2 : 1;
__constant__ double c_VP[EO_H * EO_H], c_VM[EO_H * EO_H];
__constant__ float f_VP[EO_H * EO_H], f_VM[EO_H * EO_H];
__constant__ float f_D[nn], f_D2[nn], f_Dq[nn], f_De[nn];
__constant__ float f_w[n], f_invw[n], f_xi[n], f_xh[n + 1], f_ihx[n];

// basis tables in the arithmetic type
template <typename R> struct Tab;
template <> struct Tab<double> {
  static __device__ __forceinline__ double D(int k) { return c_D[k]; }
  static __device__ __forceinline__ double D2(int k) { return c_D2[k]; }
  static __device__ __forceinline__ double Dq(int k) { return c_Dq[k]; }
  static __device__ __forceinline__ double De(int k) { return c_De[k]; }
  static __device__ __forceinline__ double w(int k) { return c_w[k]; }
  static __device__ __forceinline__ double invw(int k) { return c_invw[k]; }
  static __device__ __forceinline__ double xi(int k) { return c_xi[k]; }
  static __device__ __forceinline__ double xh(int k) { return c_xh[k]; }
  static __device__ __forceinline__ double ihx(int k) { return c_ihx[k]; }
  static __device__ __forceinline__ double VP(int k) { return c_VP[k]; }
  static __device__ __forceinline__ double VM(int k) { return c_VM[k]; }
};
template <> struct Tab<float> {
  static __device__ __forceinline__ float D(int k) { return f_D[k]; }
  static __device__ __forceinline__ float D2(int k) { return f_D2[k]; }
  static __device__ __forceinline__ float Dq(int k) { return f_Dq[k]; }
  static __device__ __forceinline__ float De(int k) { return f_De[k]; }
  static __device__ __forceinline__ float w(int k) { return f_w[k]; }
  static __device__ __forceinline__ float invw(int k) { return f_invw[k]; }
  static __device__ __forceinline__ float xi(int k) { return f_xi[k]; }
  static __device__ __forceinline__ float xh(int k) { return f_xh[k]; }
  static __device__ __forceinline__ float ihx(int k) { return f_ihx[k]; }
  static __device__ __forceinline__ float VP(int k) { return f_VP[k]; }
  static __device__ __forceinline__ float VM(int k) { return f_VM[k]; }
};

// per-context constants in the arithmetic type (precomputed on the host)
template <typename R> struct Cst;
template <> struct Cst<double> {
  static __device__ __forceinline__ double gam(const DgDevice &d) { return d.gamma; }
  static __device__ __forceinline__ double gm1(const DgDevice &d) { return d.gm1; }
  static __device__ __forceinline__ double igm1(const DgDevice &d) { return d.igm1; }
  static __device__ __forceinline__ double iR(const DgDevice &d) { return d.iR; }
  static __device__ __forceinline__ double pref(const DgDevice &d) { return d.p_ref; }
  static __device__ __forceinline__ double href(const DgDevice &d) { return d.href; }
  static __device__ __forceinline__ double mu(const DgDevice &d) { return d.mu; }
  static __device__ __forceinline__ double kappa(const DgDevice &d) { return d.kappa; }
};
template <> struct Cst<float> {
  static __device__ __forceinline__ float gam(const DgDevice &d) { return d.gamma_f; }
  static __device__ __forceinline__ float gm1(const DgDevice &d) { return d.gm1_f; }
  static __device__ __forceinline__ float igm1(const DgDevice &d) { return d.igm1_f; }
  static __device__ __forceinline__ float iR(const DgDevice &d) { return d.iR_f; }
  static __device__ __forceinline__ float pref(const DgDevice &d) { return d.p_ref_f; }
  static __device__ __forceinline__ float href(const DgDevice &d) { return d.href_f; }
  static __device__ __forceinline__ float mu(const DgDevice &d) { return d.mu_f; }
  static __device__ __forceinline__ float kappa(const DgDevice &d) { return d.kappa_f; }
};

// per-stage buffers and metric copies in the arithmetic type
template <typename R> struct Buf;
template <> struct Buf<double> {
  static __device__ __forceinline__ double *Fsurf(const DgDevice &d) { return d.Fsurf; }
  static __device__ __forceinline__ double *Wsurf(const DgDevice &d) { return d.Wsurf; }
  static __device__ __forceinline__ double *Fv(const DgDevice &d) { return d.Fv; }
  static __device__ __forceinline__ double *Fwall(const DgDevice &d) { return d.Fwall; }
  static __device__ __forceinline__ const double *Ja(const DgDevice &d) { return d.Ja; }
  static __device__ __forceinline__ const double *nrm(const DgDevice &d) { return d.nrm; }
};
template <> struct Buf<float> {
  static __device__ __forceinline__ float *Fsurf(const DgDevice &d) { return d.Fsurf_f; }
  static __device__ __forceinline__ float *Wsurf(const DgDevice &d) { return d.Wsurf_f; }
  static __device__ __forceinline__ float *Fv(const DgDevice &d) { return d.Fv_f; }
  static __device__ __forceinline__ float *Fwall(const DgDevice &d) { return d.Fwall_f; }
  static __device__ __forceinline__ const float *Ja(const DgDevice &d) { return d.Jaf; }
  static __device__ __forceinline__ const float *nrm(const DgDevice &d) { return d.nrm_f; }
};

// whether the state is carried shifted by the reference pressure (FP32 only)
template <typename R> constexpr bool kShift = std::is_same<R, float>::value;

enum { VF_KG = 0, VF_PIR = 1, VF_EC = 2, VF_CEN = 3 };
enum { SF_LLF = 0, SF_ROE = 1, SF_EC = 2 };

__host__ __device__ constexpr int round32(int x) { return (x + 31) / 32 * 32; }
// elements per CTA of the volume kernel: make 3 n^2 line threads x EPB fill whole warps
__host__ __device__ constexpr int vol_epb() {
  return N == 1 ? 8 : N == 2 ? 4 : N == 3 ? 2 : N == 4 ? 3 : N == 5 ? 2 : 1;
}
constexpr int VOL_EPB = vol_epb();
constexpr int VOL_THREADS = round32(3 * nn * VOL_EPB);
template <typename R, bool SC> __host__ __device__ constexpr int vol_threads() { return VOL_THREADS; }
// minimum resident CTAs per SM the register budget must allow (FP32 uses half the shared memory)
template <typename R, bool SC> __host__ __device__ constexpr int vol_min_blocks() {
  return std::is_same<R, float>::value && !SC ? 3 : 2;
}
// staged quantities per node: rho, u, v, w, 4 p_m, X, Y (+ p' for the FV operator)
template <bool SC> __host__ __device__ constexpr int vol_np() { return SC ? 8 : 7; }
// lifting kernel: whole elements per CTA, a thread per node (looped above 256 threads)
__host__ __device__ constexpr int lift_epb() { return nnn >= 128 ? 1 : (128 + nnn - 1) / nnn; }
constexpr int LIFT_EPB = lift_epb();
constexpr int LIFT_THREADS = round32(LIFT_EPB * nnn) > 256 ? 256 : round32(LIFT_EPB * nnn);

__device__ __forceinline__ int pidx(int node) {  // padded staging index of node (i,j,k)
  const int i = node % n, j = (node / n) % n, k = node / nn;
  return i + (n + 1) * (j + n * k);
}

__device__ __forceinline__ int face_node(int f, int p, int q) {
  const int b = (f & 1) ? N : 0;
  switch (f >> 1) {
    case 0: return b + n * (p + n * q);
    case 1: return p + n * (b + n * q);
    default: return p + n * (q + n * b);
  }
}

// the wall-model exchange node: `k` nodes from face f along the element's line through face point (p, q)
__device__ __forceinline__ int exchange_node(int f, int p, int q, int k) {
  const int b = (f & 1) ? N - k : k;
  switch (f >> 1) {
    case 0: return b + n * (p + n * q);
    case 1: return p + n * (b + n * q);
    default: return p + n * (q + n * b);
  }
}

__device__ __forceinline__ void orient_map(int o, int p, int q, int &p2, int &q2) {
  int a = p, b = q;
  if (o & 4) { a = q; b = p; }
  if (o & 1) a = N - a;
  if (o & 2) b = N - b;
  p2 = a;
  q2 = b;
}

__device__ __forceinline__ void flag_set(int *flag, int bit) { atomicOr(flag, bit); }

// Programmatic dependent launch of the stage's kernels (launch_after): a kernel lets the next one be set up once all
// its blocks are in their last phase, and the next one's blocks load their tables and geometry, which no kernel
// writes, before they wait for its completion (and, each kernel having waited for its own predecessor, for all
// earlier ones). Not earlier: with three kernels' blocks on the SMs the block scheduler doubles some up (10 steps at
// N = 7, 4^3: 3.46 ms when every kernel signalled at its start, 2.77 ms without dependent launch). A kernel launched so may
// be running while its predecessor writes, so it reads what the chain writes (state, face and viscous fluxes, jumps) by
// plain loads: no __ldg and no __restrict__ on those, whose read-only path asks for data constant from the kernel's start.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ double to_double(float f) { return (double)f; }
__device__ __forceinline__ double to_double(double x) { return x; }

// five conservative values of node `node` of element e, in the arithmetic type: the FP64 state,
// or in FP32 its shadow copy (E' = E - p_ref/(gamma-1) already applied, rounded once)
template <typename R>
__device__ __forceinline__ void load_state(const DgDevice &d, const double *U, size_t e, int node,
                                           R out[5]) {
  if (kShift<R>) {
    const float *Ue = d.Uf + e * 5 * nnn + node;
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = (R)Ue[v * nnn];
  } else {
    const double *Ue = U + e * 5 * nnn + node;
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = (R)Ue[v * nnn];
  }
}

// (float)x with the common case, a normal float, on the integer pipes: the hardware converts 2 per clock and SM
__device__ __forceinline__ float shadow_float(double x) {
  return ((unsigned)__double2hiint(x) & 0x7FFFFFFFu) - (897u << 20) < (254u << 20) ? d2f_int(x) : (float)x;
}

// FP32 shadow of the state: Uf = float(U), with E' = E - p_ref/(gamma-1) formed in FP64 first. Bound by HBM; V values
// per thread and step (V divides an element's nodes, so they share their variable; V = 4 wants 16-byte aligned U).
// N = 7, 24^3: 135 us with one value and the hardware's conversion.
template <int V>
__global__ void __launch_bounds__(256) k_shadow(const DgDevice d, const double *__restrict__ U) {
  const long long total = (long long)d.nE * 5 * nnn / V;
  const double eref = d.eref;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int v = total < (1ll << 31) ? (int)((unsigned)t / (nnn / V) % 5u) : (int)((t / (nnn / V)) % 5);
    if constexpr (V == 4) {
      const double2 x = reinterpret_cast<const double2 *>(U)[2 * t], y = reinterpret_cast<const double2 *>(U)[2 * t + 1];
      reinterpret_cast<float4 *>(d.Uf)[t] = v == 4 ? float4{shadow_float(x.x - eref), shadow_float(x.y - eref),
                                                                    shadow_float(y.x - eref), shadow_float(y.y - eref)}
                                                   : float4{shadow_float(x.x), shadow_float(x.y), shadow_float(y.x), shadow_float(y.y)};
    } else {
      d.Uf[t] = shadow_float(v == 4 ? U[t] - eref : U[t]);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// pointwise physics (pressure p' = p - p_ref enters the momentum flux; p_ref = 0 in FP64)
// ---------------------------------------------------------------------------------------------

__device__ __forceinline__ double rsq(double x) { return rsq_int(x); }
__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
template <typename R> __device__ __forceinline__ R rcp(const R &x) { return R(1) / x; }
template <> __device__ __forceinline__ double rcp<double>(const double &x) { return rcp_int(x); }
template <typename R> __device__ __forceinline__ R root(const R &x) { return sqrt(x); }
template <> __device__ __forceinline__ double root<double>(const double &x) { return sqr_int(x); }

// one side of a Riemann problem: conservative state, velocity, p' and the true pressure, 1/sqrt(rho), 1/rho
template <typename R>
struct RSide {
  R U[5], u[3], pm, p, rs, ir;
};

// Euler flux of one side through the unit vector a; returns u.a
template <typename R>
__device__ __forceinline__ R euler_flux(const RSide<R> &s, R href, const R a[3], R F[5]) {
  const R un = s.u[0] * a[0] + s.u[1] * a[1] + s.u[2] * a[2];
  F[0] = s.U[0] * un;
  F[1] = s.U[1] * un + s.pm * a[0];
  F[2] = s.U[2] * un + s.pm * a[1];
  F[3] = s.U[3] * un + s.pm * a[2];
  // E + p = E' + p' + gamma p_ref/(gamma-1)
  F[4] = kShift<R> ? (s.U[4] + s.pm + href) * un : (s.U[4] + s.pm) * un;
  return un;
}

// F = ln(a/b) / (2 f) and its reciprocal, with f = (a - b)/(a + b): the logarithmic mean of a and b is
// (a + b)/(2 F). Series in u = f^2 where the ratio is close to 1 (Ismail and Roe), and the series of 1/F
template <typename R>
__device__ __forceinline__ void log_ratio(R a, R b, R f, R &F, R &G) {
  const R u = f * f;
  const R cut = kShift<R> ? R(1e-2) : R(1e-4);
  if (u < cut) {
    F = R(1) + u * (R(1.0 / 3.0) + u * (R(0.2) + u * R(1.0 / 7.0)));
    G = R(1) - u * (R(1.0 / 3.0) + u * (R(4.0 / 45.0) + u * R(44.0 / 945.0)));
  } else {
    F = log(a / b) / (f + f);
    G = R(1) / F;
  }
}

// Chandrashekar's entropy-conservative two-point flux through the vector a (true pressures), with each side's
// beta = rho / (2 p). Two reciprocals per pair, of the sums of rho and of beta, serve the logarithmic means, their
// inverses and p-hat; a division for each of these made seven (volume kernel N = 4, 23 x 19 x 17: 1.76 -> 1.02 ms).
template <typename R>
__device__ __forceinline__ void ec_flux(R rL, R uL, R vL, R wL, R bL, R rR, R uR, R vR, R wR, R bR, const R a[3], R igm1,
                                        R pref, R F[5]) {
  const R Sr = rL + rR, Sb = bL + bR, iSb = rcp<R>(Sb);
  R Fr, Gr, Fb, Gb;
  log_ratio<R>(rL, rR, (rL - rR) * rcp<R>(Sr), Fr, Gr);
  log_ratio<R>(bL, bR, (bL - bR) * iSb, Fb, Gb);
  const R um = R(0.5) * (uL + uR), vm = R(0.5) * (vL + vR), wm = R(0.5) * (wL + wR);
  const R h0 = R(0.5) * Sr * iSb, phat = h0 + (R(0.5) * Sr - h0 * Sb) * iSb - pref;  // the quotient to its last bit
  const R q2 = R(0.25) * (uL * uL + vL * vL + wL * wL + uR * uR + vR * vR + wR * wR);
  const R V = um * a[0] + vm * a[1] + wm * a[2];
  F[0] = R(0.5) * Sr * Gr * V;
  F[1] = F[0] * um + phat * a[0];
  F[2] = F[0] * vm + phat * a[1];
  F[3] = F[0] * wm + phat * a[2];
  // energy: 1/(2 (gamma - 1) beta_ln) = F_b / ((gamma - 1) S_beta), and the true p-hat
  F[4] = F[0] * (Fb * iSb * igm1 - q2) + um * F[1] + vm * F[2] + wm * F[3] + pref * V;
}

// the side's velocity and pressure from its conservative state. One reciprocal square root: 1/sqrt(rho);
// 1/rho is its square and sqrt(rho) = rho/sqrt(rho)
template <typename R>
__device__ __forceinline__ void side_from_cons(R gm1, R pref, RSide<R> &s) {
  s.rs = rsq(s.U[0]);
  s.ir = s.rs * s.rs;
#pragma unroll
  for (int c = 0; c < 3; ++c) s.u[c] = s.U[1 + c] * s.ir;
  s.pm = gm1 * (s.U[4] - R(0.5) * (s.U[1] * s.u[0] + s.U[2] * s.u[1] + s.U[3] * s.u[2]));  // p'
  s.p = kShift<R> ? s.pm + pref : s.pm;
}

// Riemann flux F*(L, R, nv) of two sides for a unit normal nv
template <typename R>
__device__ __forceinline__ void riemann_sides(int sf, const RSide<R> &L, const RSide<R> &Q, const R nv[3], R gam,
                                              R pref, R href, R F[5]) {
  const R gm1 = gam - R(1);
  const R *UL = L.U, *UR = Q.U;
  const R irL = L.ir, irR = Q.ir, rsL = L.rs, rsR = Q.rs, pL = L.p, pR = Q.p;
  const R uL = L.u[0], vL = L.u[1], wL = L.u[2], uR = Q.u[0], vR = Q.u[1], wR = Q.u[2];
  if (sf == SF_EC) {
    ec_flux<R>(UL[0], uL, vL, wL, R(0.5) * UL[0] * rcp<R>(pL), UR[0], uR, vR, wR, R(0.5) * UR[0] * rcp<R>(pR), nv,
               rcp<R>(gm1),
               kShift<R> ? pref : R(0), F);
    return;
  }
  R FL[5], FR[5];
  const R unL = euler_flux<R>(L, href, nv, FL), unR = euler_flux<R>(Q, href, nv, FR);
  if (sf == SF_LLF) {
    const R cL = root<R>(gam * pL * irL), cR = root<R>(gam * pR * irR);
    const R lam = fmax(fabs(unL) + cL, fabs(unR) + cR);
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = R(0.5) * (FL[v] + FR[v] - lam * (UR[v] - UL[v]));
    return;
  }
  // Roe: sqrt(rho)-weighted average state, three wave families, no entropy fix. With
  // s = sqrt(rho), the weight of side k is s_k / (s_L + s_R), so the averages of u and H are
  // sum_k (m_k / s_k) / (s_L + s_R) = sum_k a_k m_k with a_k = (1/sqrt(rho_k)) / (s_L + s_R).
  const R sL = UL[0] * rsL, sR = UR[0] * rsR;
  const R iw = rcp<R>(sL + sR);
  const R aL = rsL * iw, aR = rsR * iw;
  const R ut = aL * UL[1] + aR * UR[1], vt = aL * UL[2] + aR * UR[2], wt = aL * UL[3] + aR * UR[3];
  const R EpL = kShift<R> ? UL[4] + pL - pref + href : UL[4] + pL;  // E + p
  const R EpR = kShift<R> ? UR[4] + pR - pref + href : UR[4] + pR;
  const R Ht = aL * EpL + aR * EpR;
  const R q2 = ut * ut + vt * vt + wt * wt;
  const R c2 = gm1 * (Ht - R(0.5) * q2);
  const R rc = rsq(c2);  // 1/c; c = c^2/c and 1/c^2 = (1/c)^2
  const R ct = c2 * rc, ic2 = rc * rc;
  const R rt = sL * sR;
  const R unt = ut * nv[0] + vt * nv[1] + wt * nv[2];
  const R dr = UR[0] - UL[0], dp = pR - pL;
  const R du = uR - uL, dv = vR - vL, dw = wR - wL;
  const R dun = du * nv[0] + dv * nv[1] + dw * nv[2];
  const R a1 = R(0.5) * (dp - rt * ct * dun) * ic2;
  const R a5 = R(0.5) * (dp + rt * ct * dun) * ic2;
  const R a2 = dr - dp * ic2;
  const R dut = du - dun * nv[0], dvt = dv - dun * nv[1], dwt = dw - dun * nv[2];
  const R l1a1 = fabs(unt - ct) * a1, l5a5 = fabs(unt + ct) * a5, l2 = fabs(unt);
  const R l2a2 = l2 * a2, l2r = l2 * rt;
  // dissipation sum_k |lambda_k| alpha_k r_k, collected: with s15 = l1a1 + l5a5 and c15 = c (l5a5 - l1a1),
  // the two acoustic waves give s15 (u~, H~) + c15 (n, u~_n)
  const R s15 = l1a1 + l5a5, c15 = ct * (l5a5 - l1a1);
  R D[5];
  D[0] = s15 + l2a2;
  D[1] = D[0] * ut + c15 * nv[0] + l2r * dut;
  D[2] = D[0] * vt + c15 * nv[1] + l2r * dvt;
  D[3] = D[0] * wt + c15 * nv[2] + l2r * dwt;
  D[4] = s15 * Ht + c15 * unt + l2a2 * R(0.5) * q2 + l2r * (ut * dut + vt * dvt + wt * dwt);
#pragma unroll
  for (int v = 0; v < 5; ++v) F[v] = R(0.5) * (FL[v] + FR[v] - D[v]);
}

// the same from two conservative states; also returns each side's 1/rho and true pressure (the face kernel's BR1
// face values reuse them)
template <typename R>
__device__ __forceinline__ void riemann(int sf, const R UL[5], const R UR[5], const R nv[3], R gam, R pref, R href,
                                        R F[5], R &irL, R &irR, R &pL, R &pR) {
  RSide<R> L, Q;
#pragma unroll
  for (int v = 0; v < 5; ++v) { L.U[v] = UL[v]; Q.U[v] = UR[v]; }
  side_from_cons<R>(gam - R(1), pref, L);
  side_from_cons<R>(gam - R(1), pref, Q);
  irL = L.ir; irR = Q.ir; pL = L.p; pR = Q.p;
  riemann_sides<R>(sf, L, Q, nv, gam, pref, href, F);
}

template <typename R>
__device__ __forceinline__ void riemann(int sf, const R UL[5], const R UR[5], const R nv[3], R gam, R pref, R href,
                                        R F[5]) {
  R irL, irR, pL, pR;
  riemann<R>(sf, UL, UR, nv, gam, pref, href, F, irL, irR, pL, pR);
}

// ---------------------------------------------------------------------------------------------
// init: curl-form metrics, Jacobian, face normals (FP64), FP32 copies
// ---------------------------------------------------------------------------------------------

__device__ __forceinline__ double dsweep(const double *f, int node, int d) {
  const int i = node % n, j = (node / n) % n, k = node / nn;
  const int id = d == 0 ? i : d == 1 ? j : k;
  const int st = d == 0 ? 1 : d == 1 ? n : nn;
  const int base = node - id * st;
  double s = 0.0;
#pragma unroll
  for (int m = 0; m < n; ++m) s += c_D[id * n + m] * f[base + m * st];
  return s;
}

// One CTA per element. Ja^d_c = D_k(X_l D_j X_m) - D_j(X_l D_k X_m), (d,j,k), (c,m,l) cyclic;
// J = det(D-derivatives of X). X is taken relative to the element's first node: the metric
// terms are translation invariant, and absolute coordinates (|x| >> h) would make the
// products X_l D_j X_m cancel to O(|x|/h) of rounding.
__global__ void __launch_bounds__(256) k_metrics(const DgDevice d) {
  extern __shared__ double sm[];
  double *X = sm;              // [3][nnn]
  double *dX = X + 3 * nnn;    // [c][dd][nnn]
  double *T1 = dX + 9 * nnn;   // [nnn]
  double *T2 = T1 + nnn;       // [nnn]
  const int e = blockIdx.x;
  const double *xe = d.xyz + (size_t)e * 3 * nnn;
  for (int t = threadIdx.x; t < 3 * nnn; t += blockDim.x) X[t] = xe[t] - xe[(t / nnn) * nnn];
  __syncthreads();
  for (int t = threadIdx.x; t < 9 * nnn; t += blockDim.x) {
    const int node = t % nnn, cd = t / nnn, c = cd / 3, dd = cd % 3;
    dX[cd * nnn + node] = dsweep(X + c * nnn, node, dd);
  }
  __syncthreads();
  for (int dir = 0; dir < 3; ++dir) {
    const int j = (dir + 1) % 3, k = (dir + 2) % 3;
    for (int c = 0; c < 3; ++c) {
      const int m = (c + 1) % 3, l = (c + 2) % 3;
      for (int node = threadIdx.x; node < nnn; node += blockDim.x) {
        T1[node] = X[l * nnn + node] * dX[(m * 3 + j) * nnn + node];
        T2[node] = X[l * nnn + node] * dX[(m * 3 + k) * nnn + node];
      }
      __syncthreads();
      for (int node = threadIdx.x; node < nnn; node += blockDim.x)
        d.Ja[(((size_t)e * 3 + dir) * 3 + c) * nnn + node] = dsweep(T1, node, k) - dsweep(T2, node, j);
      __syncthreads();
    }
  }
  for (int node = threadIdx.x; node < nnn; node += blockDim.x) {
    double a[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) a[c][dd] = dX[(c * 3 + dd) * nnn + node];
    const double J = a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0]) +
                     a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]);
    d.J[(size_t)e * nnn + node] = J;
    d.invJ[(size_t)e * nnn + node] = 1.0 / J;
    if (!(J > 0.0) || !isfinite(J)) flag_set(d.flag, 2);
  }
}

// One thread per face point: unit normal and area factor from the L element's metric.
__global__ void __launch_bounds__(256) k_face_normals(const DgDevice d) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.nF * nn) return;
  const int f = (int)(t / nn), pq = (int)(t % nn), p = pq % n, q = pq / n;
  const int eL = d.face[5 * f + 0], fL = d.face[5 * f + 1];
  const int dL = fL >> 1;
  const double sg = (fL & 1) ? 1.0 : -1.0;
  const int node = face_node(fL, p, q);
  double a[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) a[c] = sg * d.Ja[(((size_t)eL * 3 + dL) * 3 + c) * nnn + node];
  const double s = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
  const double is = 1.0 / s;
  double *o = d.nrm + (size_t)f * 4 * nn + pq;
  o[0] = a[0] * is;
  o[nn] = a[1] * is;
  o[2 * nn] = a[2] * is;
  o[3 * nn] = s;
  if (d.face[5 * f + 2] < 0 && d.hwm) {  // wall face: distance of the wall-model exchange node
    const int xnode = exchange_node(fL, p, q, d.wm_index);
    double h2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double dx = d.xyz[((size_t)eL * 3 + c) * nnn + xnode] - d.xyz[((size_t)eL * 3 + c) * nnn + node];
      h2 += dx * dx;
    }
    d.hwm[(size_t)f * nn + pq] = sqrt(h2);
  }
}

// FP32 roundings of the FP64 metric terms and face normals (FP32-bulk path)
__global__ void __launch_bounds__(256) k_round_geometry(const DgDevice d) {
  const long long nja = (long long)d.nE * 9 * nnn, nnr = (long long)d.nF * 4 * nn, nij = (long long)d.nE * nnn;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nja + nnr + nij;
       t += (long long)gridDim.x * blockDim.x) {
    if (t < nja) d.Jaf[t] = (float)d.Ja[t];
    else if (t < nja + nnr) d.nrm_f[t - nja] = (float)d.nrm[t - nja];
    else d.invJf[t - nja - nnr] = (float)d.invJ[t - nja - nnr];
  }
}

// ---------------------------------------------------------------------------------------------
// wall-modelled wall face point (Sec. 3): advective flux against the mirror state, BR1 jump to the
// mirror state's face value, and the wall shear stress of the wall model as the viscous flux
// ---------------------------------------------------------------------------------------------
template <typename R, int SF>
__device__ __forceinline__ void wall_face(const DgDevice &d, const double *U, int f, int pq, int eL,
                                          int fL, R pref, R href, R gam) {
  const int p = pq % n, q = pq / n;
  const int node = face_node(fL, p, q);
  R UL[5], UG[5], nv[3], Fs[5];
  load_state<R>(d, U, eL, node, UL);
  const R *nr = Buf<R>::nrm(d) + (size_t)f * 4 * nn + pq;
  nv[0] = nr[0];
  nv[1] = nr[nn];
  nv[2] = nr[2 * nn];
  const R s = nr[3 * nn];
  const R mn = UL[1] * nv[0] + UL[2] * nv[1] + UL[3] * nv[2];
  UG[0] = UL[0];
  UG[4] = UL[4];
#pragma unroll
  for (int c = 0; c < 3; ++c) UG[1 + c] = UL[1 + c] - R(2) * mn * nv[c];
  riemann<R>(SF, UL, UG, nv, gam, pref, href, Fs);
  R *oL = Buf<R>::Fsurf(d) + ((size_t)eL * 6 + fL) * 5 * nn + pq;
#pragma unroll
  for (int v = 0; v < 5; ++v) oL[v * nn] = s * Fs[v];
  if (d.equations != 1) return;
  // BR1: w* - w = (w_ghost - w) / 2 = (-(u.n) n, 0)
  const R un = mn / UL[0];
  R *jL = Buf<R>::Wsurf(d) + ((size_t)eL * 6 + fL) * 4 * nn + pq;
#pragma unroll
  for (int c = 0; c < 3; ++c) jL[c * nn] = -un * nv[c];
  jL[3 * nn] = R(0);
  // wall model at the exchange node
  R Ux[5];
  load_state<R>(d, U, eL, exchange_node(fL, p, q, d.wm_index), Ux);
  const R irx = R(1) / Ux[0];
  const R ux[3] = {Ux[1] * irx, Ux[2] * irx, Ux[3] * irx};
  const R uxn = ux[0] * nv[0] + ux[1] * nv[1] + ux[2] * nv[2];
  const R ut[3] = {ux[0] - uxn * nv[0], ux[1] - uxn * nv[1], ux[2] - uxn * nv[2]};
  const R Ut = sqrt(ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2]);
  R *fw = Buf<R>::Fwall(d) + (size_t)f * 4 * nn + pq;
  R tw[3] = {R(0), R(0), R(0)};
  if (Ut > R(0)) {
    int it;
    const R utau = wall_utau<R, true>(Ut, (R)d.hwm[(size_t)f * nn + pq], Cst<R>::mu(d) * irx, (R)d.wm_uinf, (R)d.wm_b,
                                d.wm_vd, it);
    const R tau = Ux[0] * utau * utau;
#pragma unroll
    for (int c = 0; c < 3; ++c) tw[c] = -tau * ut[c] / Ut;  // outward viscous flux: the wall's drag
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) fw[c * nn] = s * tw[c];
  fw[3 * nn] = R(0);  // adiabatic wall at rest
}

// ---------------------------------------------------------------------------------------------
// face kernel: Riemann flux once per face point, stored outward for both sides
// ---------------------------------------------------------------------------------------------
// Threads per block: 64, so that small meshes spread over the SMs (each SM's FP64 pipe takes 2 lanes per clock, so a
// 256-thread block alone on its SM runs its ~200 FP64 instructions per point for 13 us). Per launch at N = 7, 4^3
// (192 faces): 18.5 us with 256 threads, 12.5 with 128, 64 or 32; at 24^3 817 / 824 / 812 / 812 us.
constexpr int FACE_THREADS = 64;
template <typename R, int SF>
__global__ void __launch_bounds__(FACE_THREADS) k_face(const DgDevice d, const double *U) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.nF * nn) return;
  const int f = (int)(t / nn), pq = (int)(t % nn), p = pq % n, q = pq / n;
  const int *F5 = d.face + 5 * f;
  const int eL = F5[0], fL = F5[1], eR = F5[2], fR = F5[3], o = F5[4];
  const R pref = Cst<R>::pref(d), href = Cst<R>::href(d), gam = Cst<R>::gam(d);
  const R *nr = Buf<R>::nrm(d) + (size_t)f * 4 * nn + pq;
  const R nv[3] = {nr[0], nr[nn], nr[2 * nn]}, s = nr[3 * nn];
  wait_for_previous();
  if (eR < 0) {  // wall-modelled wall
    wall_face<R, SF>(d, U, f, pq, eL, fL, pref, href, gam);
    return;
  }
  int p2, q2;
  orient_map(o, p, q, p2, q2);
  const int nodeL = face_node(fL, p, q), nodeR = face_node(fR, p2, q2);
  const int pqR = p2 + n * q2;
  R UL[5], UR[5];
  load_state<R>(d, U, eL, nodeL, UL);
  load_state<R>(d, U, eR, nodeR, UR);
  R Fs[5], irL, irR, pL, pR;
  riemann<R>(SF, UL, UR, nv, gam, pref, href, Fs, irL, irR, pL, pR);
  let_next_start();
  R *oL = Buf<R>::Fsurf(d) + ((size_t)eL * 6 + fL) * 5 * nn;
  R *oR = Buf<R>::Fsurf(d) + ((size_t)eR * 6 + fR) * 5 * nn;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    oL[v * nn + pq] = s * Fs[v];
    oR[v * nn + pqR] = -s * Fs[v];
  }
  if (d.equations == 1) {  // BR1 face values of (u, v, w, T), from the Riemann solver's 1/rho and p
    const R wL[3] = {UL[1] * irL, UL[2] * irL, UL[3] * irL};
    const R wR[3] = {UR[1] * irR, UR[2] * irR, UR[3] * irR};
    const R iR = Cst<R>::iR(d);
    const R jump[4] = {R(0.5) * (wR[0] - wL[0]), R(0.5) * (wR[1] - wL[1]), R(0.5) * (wR[2] - wL[2]),
                       R(0.5) * (pR * irR - pL * irL) * iR};
    R *jL = Buf<R>::Wsurf(d) + ((size_t)eL * 6 + fL) * 4 * nn;
    R *jR = Buf<R>::Wsurf(d) + ((size_t)eR * 6 + fR) * 4 * nn;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      jL[c * nn + pq] = jump[c];
      jR[c * nn + pqR] = -jump[c];
    }
  }
}

// ---------------------------------------------------------------------------------------------
// BR1 lifting + viscous flux: grad w = (1/J)[sum_d Ja^d D_d w + sum_faces (1/w_b) s n_out (w* - w)],
// then Fv^d = sum_c Ja^d_c Fv_c(U, grad w) stored per node (4 components: momentum, energy).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int fx_relative(double f, int unit);  // dg_fixed.cuh

// (u, v, w, T) of one node from its state values (lifted quantities of BR1)
template <typename R>
__device__ __forceinline__ void lift_prim(const R Uv[5], R gm1, R iR, R pref, R Wn[4]) {
  const R r = Uv[0], ir = rcp<R>(r);
  const R u = Uv[1] * ir, v = Uv[2] * ir, w = Uv[3] * ir;
  R p = gm1 * (Uv[4] - R(0.5) * r * (u * u + v * v + w * w));
  if (kShift<R>) p += pref;
  Wn[0] = u;
  Wn[1] = v;
  Wn[2] = w;
  Wn[3] = p * ir * iR;
}

// one node's BR1 gradients and contravariant viscous flux: W = the element's lifted quantities
// [4][nnn] (shared memory), Jae its metric terms [3 d][3 c][nnn], Wse its BR1 face jumps [6][4][nn],
// iJ this node's 1/J; writes the element's Fv [3 d][4][nnn] at `node` (out = the element's Fv).
// tau (FP64 only, optional): the element's viscous stress record [6][nnn] (xx, yy, zz, xy, xz, yz),
// which the adjoint's viscous kernel reads instead of forming the gradients again
template <typename R>
__device__ __forceinline__ void lift_node(const DgDevice &d, int node, const R *__restrict__ W,
                                          const R (*__restrict__ sD)[n + 1], const R *__restrict__ Jae,
                                          const R *Wse, R iJ, R mu, R kappa, R *__restrict__ out,
                                          double *__restrict__ tau = nullptr, const int *unit = nullptr,
                                          int *fvm = nullptr) {
  const int ijk[3] = {node % n, (node / n) % n, node / nn};
  R Ja[3][3];
#pragma unroll
  for (int dd = 0; dd < 3; ++dd)
#pragma unroll
    for (int c = 0; c < 3; ++c) Ja[dd][c] = Jae[(dd * 3 + c) * nnn + node];
  R g[4][3];
#pragma unroll
  for (int q = 0; q < 4; ++q) g[q][0] = g[q][1] = g[q][2] = R(0);
#pragma unroll
  for (int dd = 0; dd < 3; ++dd) {
    const int id = ijk[dd];
    const int st = dd == 0 ? 1 : dd == 1 ? n : nn;
    const int base = node - id * st;
    // the reference derivative along dd, plus the surface term (1/w_b)(+-)(w* - w) on the face of
    // direction dd through this node, before the one contraction with Ja^dd
    R s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[q] = R(0);
#pragma unroll
      for (int m = 0; m < n; ++m) s[q] += sD[id][m] * W[q * nnn + base + m * st];
    }
    if (id == 0 || id == N) {
      const int f = 2 * dd + (id == N ? 1 : 0);
      const R sc = (id == N ? R(1) : R(-1)) * Tab<R>::invw(id);
      const int pp = dd == 0 ? ijk[1] : ijk[0];
      const int qq = dd == 2 ? ijk[1] : ijk[2];
      const R *js = Wse + f * 4 * nn + pp + n * qq;
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] += sc * js[q * nn];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      g[q][0] += Ja[dd][0] * s[q];
      g[q][1] += Ja[dd][1] * s[q];
      g[q][2] += Ja[dd][2] * s[q];
    }
  }
  // g holds J grad w; the flux below is linear in grad w, so 1/J goes into mu and kappa (two
  // multiplies per node instead of twelve)
  mu *= iJ;
  kappa *= iJ;
  // Navier-Stokes-Fourier flux in Cartesian direction c: (tau_xc, tau_yc, tau_zc, u.tau_c + kappa dT/dx_c)
  const R u = W[node], v = W[nnn + node], w = W[2 * nnn + node];
  const R div = g[0][0] + g[1][1] + g[2][2];
  const R t23 = R(2.0 / 3.0) * mu * div;
  const R txx = R(2) * mu * g[0][0] - t23, tyy = R(2) * mu * g[1][1] - t23, tzz = R(2) * mu * g[2][2] - t23;
  const R txy = mu * (g[0][1] + g[1][0]), txz = mu * (g[0][2] + g[2][0]), tyz = mu * (g[1][2] + g[2][1]);
  if constexpr (std::is_same<R, double>::value) {
    if (tau) {
      tau[node] = txx; tau[nnn + node] = tyy; tau[2 * nnn + node] = tzz;
      tau[3 * nnn + node] = txy; tau[4 * nnn + node] = txz; tau[5 * nnn + node] = tyz;
    }
  }
  R Fc[3][4];
  Fc[0][0] = txx; Fc[0][1] = txy; Fc[0][2] = txz; Fc[0][3] = u * txx + v * txy + w * txz + kappa * g[3][0];
  Fc[1][0] = txy; Fc[1][1] = tyy; Fc[1][2] = tyz; Fc[1][3] = u * txy + v * tyy + w * tyz + kappa * g[3][1];
  Fc[2][0] = txz; Fc[2][1] = tyz; Fc[2][2] = tzz; Fc[2][3] = u * txz + v * tyz + w * tzz + kappa * g[3][2];
#pragma unroll
  for (int dd = 0; dd < 3; ++dd)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const R f = Ja[dd][0] * Fc[0][q] + Ja[dd][1] * Fc[1][q] + Ja[dd][2] * Fc[2][q];
      out[(dd * 4 + q) * nnn + node] = f;
      // FP64: high words of the largest momentum and energy components against the directions' metric scales (fvmax)
      if constexpr (std::is_same<R, double>::value) fvm[q / 3] = max(fvm[q / 3], fx_relative(f, unit[dd]));
    }
}

// FP32 lifting, a thread per node (the FP64 one is k_lift_fx)
__global__ void __launch_bounds__(LIFT_THREADS, 5) k_lift(const DgDevice d) {
  __shared__ float W[LIFT_EPB][4][nnn];
  __shared__ float sD[n][n + 1];  // D, rows padded: lanes read different rows without bank conflicts
  for (int t = threadIdx.x; t < nn; t += blockDim.x) sD[t / n][t % n] = f_D[t];
  const int e0 = blockIdx.x * LIFT_EPB;
  for (int t = threadIdx.x; t < LIFT_EPB * nnn; t += blockDim.x) {
    const int le = t / nnn, node = t % nnn, e = e0 + le;
    if (e >= d.nE) continue;
    float Uv[5], Wn[4];
    load_state<float>(d, nullptr, e, node, Uv);
    lift_prim<float>(Uv, d.gm1_f, d.iR_f, d.p_ref_f, Wn);
#pragma unroll
    for (int q = 0; q < 4; ++q) W[le][q][node] = Wn[q];
  }
  __syncthreads();
  // the thread's nodes unrolled, so that their metric loads are in flight together
#pragma unroll
  for (int rr = 0; rr < (LIFT_EPB * nnn + LIFT_THREADS - 1) / LIFT_THREADS; ++rr) {
    const int t = threadIdx.x + rr * LIFT_THREADS;
    if (t >= LIFT_EPB * nnn) continue;
    const int le = t / nnn, node = t % nnn, e = e0 + le;
    if (e >= d.nE) continue;
    lift_node<float>(d, node, &W[le][0][0], sD, d.Jaf + (size_t)e * 9 * nnn, d.Wsurf_f + (size_t)e * 6 * 4 * nn,
                     d.invJf[(size_t)e * nnn + node], d.mu_f, d.kappa_f, d.Fv_f + (size_t)e * 12 * nnn);
  }
}

// ---------------------------------------------------------------------------------------------
// volume kernel
// ---------------------------------------------------------------------------------------------

// Flux differencing along one line of n nodes: acc_i = sum_{m != i} 2 D_im F#(U_i, U_m) with
// the metric average {Ja}. For Kennedy-Gruber and Pirozzoli the flux is formed from plain sums
// S = x_i + x_m and the 1/2 factors are folded into the coefficients (D/4 for mass, D/8 otherwise).
// Node i's sums stay in registers while m runs over i+1..N; node m's share of each pair goes
// straight to the line's accumulator in shared memory (the line belongs to this thread alone).
// Ac points at the direction's accumulator [5][PS] of this element, indexed like P.
// Staged slots: 0 rho, 1 u, 2 v, 3 w, 4 4 p' (momentum pressure), 5 X, 6 Y with
// PIR: X = h; KG: X = e = E/rho, Y = 2p; EC: Y = rho/(2p); central: X = E + p.
template <typename R, int VF>
__device__ __forceinline__ void line_fluxdiff(const R *__restrict__ P, int pb, int ps, const R *__restrict__ Jd,
                                              int gb, int gs, R igm1, R pref, R *__restrict__ Ac) {
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const int ai = pb + i * ps, gi = gb + i * gs;
    const R ri = P[ai], ui = P[PS + ai], vi = P[2 * PS + ai], wi = P[3 * PS + ai];
    const R p4i = P[4 * PS + ai], xi_ = P[5 * PS + ai], yi = P[6 * PS + ai];
    const R jxi = __ldg(Jd + gi), jyi = __ldg(Jd + nnn + gi), jzi = __ldg(Jd + 2 * nnn + gi);
    R ac[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) ac[v] = (i == 0) ? R(0) : Ac[v * PS + ai];
#pragma unroll
    for (int m = i + 1; m < n; ++m) {
      const int am = pb + m * ps, gm = gb + m * gs;
      const R rm = P[am], um = P[PS + am], vm = P[2 * PS + am], wm = P[3 * PS + am];
      const R p4m = P[4 * PS + am], xm = P[5 * PS + am], ym = P[6 * PS + am];
      const R jxm = __ldg(Jd + gm), jym = __ldg(Jd + nnn + gm), jzm = __ldg(Jd + 2 * nnn + gm);
      R F[5], ci[5], cm[5];
      if (VF == VF_PIR || VF == VF_KG) {
        const R Sjx = jxi + jxm, Sjy = jyi + jym, Sjz = jzi + jzm;
        const R Su = ui + um, Sv = vi + vm, Sw = wi + wm;
        const R Vp = Su * Sjx + Sv * Sjy + Sw * Sjz;  // 4 {u}.{Ja}
        F[0] = (ri + rm) * Vp;                        // 8 F_rho
        const R Sp = p4i + p4m;                       // 4 (p'_i + p'_m)
        F[1] = F[0] * Su + Sp * Sjx;                  // 16 F_rho u
        F[2] = F[0] * Sv + Sp * Sjy;
        F[3] = F[0] * Sw + Sp * Sjz;
        if (VF == VF_PIR) F[4] = F[0] * (xi_ + xm);            // 16 {rho}V{h}
        else F[4] = F[0] * (xi_ + xm) + (yi + ym) * Vp;        // 16 ({rho}V{e} + {p}V)
        ci[0] = Tab<R>::Dq(i * n + m); cm[0] = Tab<R>::Dq(m * n + i);
#pragma unroll
        for (int v = 1; v < 5; ++v) { ci[v] = Tab<R>::De(i * n + m); cm[v] = Tab<R>::De(m * n + i); }
      } else {
        const R a[3] = {R(0.5) * (jxi + jxm), R(0.5) * (jyi + jym), R(0.5) * (jzi + jzm)};
        if (VF == VF_EC) {
          ec_flux<R>(ri, ui, vi, wi, yi, rm, um, vm, wm, ym, a, igm1, kShift<R> ? pref : R(0), F);
        } else {  // central: mean of the two Euler fluxes through {Ja}; slot 5 = E + p
          const R Vi = ui * a[0] + vi * a[1] + wi * a[2], Vm = um * a[0] + vm * a[1] + wm * a[2];
          const R pm2 = R(0.125) * (p4i + p4m);
          F[0] = R(0.5) * (ri * Vi + rm * Vm);
          F[1] = R(0.5) * (ri * ui * Vi + rm * um * Vm) + pm2 * a[0];
          F[2] = R(0.5) * (ri * vi * Vi + rm * vm * Vm) + pm2 * a[1];
          F[3] = R(0.5) * (ri * wi * Vi + rm * wm * Vm) + pm2 * a[2];
          F[4] = R(0.5) * (xi_ * Vi + xm * Vm);
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) { ci[v] = Tab<R>::D2(i * n + m); cm[v] = Tab<R>::D2(m * n + i); }
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        ac[v] += ci[v] * F[v];
        if (i == 0) Ac[v * PS + am] = cm[v] * F[v];
        else Ac[v * PS + am] += cm[v] * F[v];
      }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) Ac[v * PS + ai] = ac[v];
  }
}

// Viscous divergence along one line: Ac[1+q]_i -= sum_{m != i} D_im Fv^d_q(m) for the line's n
// nodes (the diagonal cancels against the surface term, see the file header). Fvd points at the
// element's contravariant viscous flux of this direction [4][nnn].
template <typename R>
__device__ __forceinline__ void line_viscous(const R *__restrict__ Fvd, int gb, int gs, int pb, int ps,
                                             R *__restrict__ Ac) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    R f[n];
#pragma unroll
    for (int m = 0; m < n; ++m) f[m] = __ldg(Fvd + q * nnn + gb + m * gs);
    if constexpr (n % 2 == 0) {  // even-odd: n^2/2 + 2n operations per line instead of n^2
      R ev[EO_H], od[EO_H];
#pragma unroll
      for (int m = 0; m < EO_H; ++m) { ev[m] = f[m] + f[N - m]; od[m] = f[m] - f[N - m]; }
#pragma unroll
      for (int i = 0; i < EO_H; ++i) {
        R a = R(0), b = R(0);
#pragma unroll
        for (int m = 0; m < EO_H; ++m) {
          a += Tab<R>::VP(i * EO_H + m) * ev[m];
          b += Tab<R>::VM(i * EO_H + m) * od[m];
        }
        Ac[(1 + q) * PS + pb + i * ps] -= a + b;
        Ac[(1 + q) * PS + pb + (N - i) * ps] -= b - a;
      }
    } else {
#pragma unroll
      for (int i = 0; i < n; ++i) {
        R s = R(0);
#pragma unroll
        for (int m = 0; m < n; ++m)
          if (m != i) s += Tab<R>::D(i * n + m) * f[m];
        Ac[(1 + q) * PS + pb + i * ps] -= s;
      }
    }
  }
}

// (rho, u, v, w, p') of staged node a for the FV operator (slot 7 holds p')
template <typename R>
__device__ __forceinline__ void staged_prim(const R *__restrict__ P, int a, R q[5]) {
  q[0] = P[a]; q[1] = P[PS + a]; q[2] = P[2 * PS + a]; q[3] = P[3 * PS + a]; q[4] = P[7 * PS + a];
}

// reconstructed left/right interface states of subcell i (minmod slopes in primitive variables;
// first order in the outer subcells and wherever the reconstruction loses positivity)
template <typename R>
__device__ __forceinline__ void subcell_states(const R *__restrict__ P, int pb, int ps, int i, R pref, R qL[5],
                                               R qR[5]) {
  R q[5];
  staged_prim<R>(P, pb + i * ps, q);
  R sg[5] = {R(0), R(0), R(0), R(0), R(0)};
  if (i > 0 && i < N) {
    R qb[5], qf[5];
    staged_prim<R>(P, pb + (i - 1) * ps, qb);
    staged_prim<R>(P, pb + (i + 1) * ps, qf);
    const R hb = Tab<R>::ihx(i), hf = Tab<R>::ihx(i + 1);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const R sb = (q[v] - qb[v]) * hb, sf_ = (qf[v] - q[v]) * hf;
      sg[v] = (sb * sf_ <= R(0)) ? R(0) : (fabs(sb) < fabs(sf_) ? sb : sf_);
    }
  }
  const R dl = Tab<R>::xh(i) - Tab<R>::xi(i), dr = Tab<R>::xh(i + 1) - Tab<R>::xi(i);
#pragma unroll
  for (int v = 0; v < 5; ++v) { qL[v] = q[v] + sg[v] * dl; qR[v] = q[v] + sg[v] * dr; }
  const R pad = kShift<R> ? pref : R(0);
  if (qL[0] <= R(0) || qL[4] + pad <= R(0) || qR[0] <= R(0) || qR[4] + pad <= R(0)) {
#pragma unroll
    for (int v = 0; v < 5; ++v) { qL[v] = q[v]; qR[v] = q[v]; }
  }
}

// conservative state from (rho, u, v, w, p') in the kernel's representation (E' in FP32)
template <typename R>
__device__ __forceinline__ void cons_of(const R q[5], R igm1, R U[5]) {
  U[0] = q[0]; U[1] = q[0] * q[1]; U[2] = q[0] * q[2]; U[3] = q[0] * q[3];
  U[4] = q[4] * igm1 + R(0.5) * q[0] * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
}

// FV subcell operator along one line (Sec. 4.1): Riemann fluxes at the N interior subcell
// interfaces with telescoped interface metrics a_{i+1/2} = a_{i-1/2} + w_i (D Ja)_i, the DG surface
// fluxes at the element faces, and Ac_i = (f_{i+1/2} - f_{i-1/2}) / w_i written to shared memory.
template <typename R>
__device__ __forceinline__ void line_fv(const R *__restrict__ P, int pb, int ps, const R *__restrict__ Jd, int gb,
                                        int gs, const R *Fm, const R *Fp, int sf, R gam, R igm1, R pref, R href,
                                        R *__restrict__ Ac) {
  R fl[5];  // flux at the left interface of the current subcell, +xi direction
#pragma unroll
  for (int v = 0; v < 5; ++v) fl[v] = -Fm[v * nn];
  R a[3] = {__ldg(Jd + gb), __ldg(Jd + nnn + gb), __ldg(Jd + 2 * nnn + gb)};
  R qLn[5], qRn[5];
  subcell_states<R>(P, pb, ps, 0, pref, qLn, qRn);
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    R fr[5];
    const R qRi[5] = {qRn[0], qRn[1], qRn[2], qRn[3], qRn[4]};
    if (i < N) {
      subcell_states<R>(P, pb, ps, i + 1, pref, qLn, qRn);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        R dj = R(0);
#pragma unroll
        for (int m = 0; m < n; ++m) dj += Tab<R>::D(i * n + m) * __ldg(Jd + c * nnn + gb + m * gs);
        a[c] += Tab<R>::w(i) * dj;
      }
      const R a2 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
      const R is = rsq(a2);  // 1/|a|; |a| = |a|^2 / |a|
      const R s = a2 * is;
      const R nv[3] = {a[0] * is, a[1] * is, a[2] * is};
      R UL[5], UR[5], Fs[5];
      cons_of<R>(qRi, igm1, UL);
      cons_of<R>(qLn, igm1, UR);
      riemann<R>(sf, UL, UR, nv, gam, pref, href, Fs);
#pragma unroll
      for (int v = 0; v < 5; ++v) fr[v] = s * Fs[v];
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) fr[v] = Fp[v * nn];
    }
    const R iw = Tab<R>::invw(i);
#pragma unroll
    for (int v = 0; v < 5; ++v) { Ac[v * PS + pb + i * ps] = (fr[v] - fl[v]) * iw; fl[v] = fr[v]; }
  }
}

// line geometry of line `line` of direction `dir`: staging base/stride (padded) and global base/stride
__device__ __forceinline__ void line_geom(int dir, int line, int &pb, int &ps, int &gb, int &gs, int &a, int &b) {
  a = line % n;
  b = line / n;
  if (dir == 0) { pb = (n + 1) * (a + n * b); ps = 1; gb = n * (a + n * b); gs = 1; }
  else if (dir == 1) { pb = a + (n + 1) * n * b; ps = n + 1; gb = a + nn * b; gs = n; }
  else { pb = a + (n + 1) * b; ps = (n + 1) * n; gb = a + n * b; gs = nn; }
}

template <typename R, int VF, bool SC>
__global__ void __launch_bounds__(vol_threads<R, SC>(), vol_min_blocks<R, SC>()) k_volume(const DgDevice d, const double *U, double *out,
                                                        double *__restrict__ g, int mode, int first, double dt,
                                                        double A, double B) {
  constexpr int NP = vol_np<SC>();
  extern __shared__ __align__(16) unsigned char sm_raw[];
  R *P = reinterpret_cast<R *>(sm_raw);  // [EPB][NP][PS]
  R *Acc = P + VOL_EPB * NP * PS;         // [EPB][3][5][PS]
  R *AccT = Acc + VOL_EPB * 15 * PS;      // [EPB][5][nnn] (SC only)
  const int e0 = blockIdx.x * VOL_EPB;
  const R gam = Cst<R>::gam(d), gm1 = Cst<R>::gm1(d);
  const R pref = Cst<R>::pref(d), href = Cst<R>::href(d);
  const double eref = d.eref;
  const R *Jab = Buf<R>::Ja(d);
  const int vf = VF;
  // phase A: stage primitive quantities
  for (int t = threadIdx.x; t < VOL_EPB * nnn; t += blockDim.x) {
    const int le = t / nnn, node = t % nnn, e = e0 + le;
    if (e >= d.nE) continue;
    R Uv[5];
    load_state<R>(d, U, e, node, Uv);
    const R r = Uv[0], m1 = Uv[1], m2 = Uv[2], m3 = Uv[3], E = Uv[4];
    const R ir = rcp<R>(r);
    const R u = m1 * ir, v = m2 * ir, w = m3 * ir;
    const R pm = gm1 * (E - R(0.5) * (m1 * u + m2 * v + m3 * w));  // p' (= p in FP64)
    const R p = kShift<R> ? pm + pref : pm;
    const R Et = kShift<R> ? E + (R)eref : E;
    if (!(r > R(0)) || !(p > R(0)) || !isfinite(E)) flag_set(d.flag, 1);
    R *Pe = P + le * NP * PS + pidx(node);
    Pe[0] = r; Pe[PS] = u; Pe[2 * PS] = v; Pe[3 * PS] = w; Pe[4 * PS] = R(4) * pm;
    if (vf == VF_PIR) Pe[5 * PS] = (Et + p) * ir;
    else if (vf == VF_KG) { Pe[5 * PS] = Et * ir; Pe[6 * PS] = R(2) * p; }
    else if (vf == VF_EC) Pe[6 * PS] = R(0.5) * r * rcp<R>(p);  // beta
    else Pe[5 * PS] = Et + p;
    if (SC) Pe[7 * PS] = pm;
  }
  __syncthreads();
  // phase B: flux differencing, one thread per line, the three line families at once
  for (int t = threadIdx.x; t < VOL_EPB * 3 * nn; t += blockDim.x) {
    const int le = t / (3 * nn), r = t % (3 * nn), dir = r / nn, line = r % nn, e = e0 + le;
    if (e >= d.nE) continue;
    int pb, ps, gb, gs, a, b;
    line_geom(dir, line, pb, ps, gb, gs, a, b);
    // viscous divergence joins the line sums, except under the blend (which must not weight it)
    const bool visc = !SC && d.equations == 1;
    line_fluxdiff<R, VF>(P + le * NP * PS, pb, ps, Jab + ((size_t)e * 3 + dir) * 3 * nnn, gb, gs, Cst<R>::igm1(d), pref,
                         Acc + (le * 3 + dir) * 5 * PS);
    if (visc)
      line_viscous<R>(Buf<R>::Fv(d) + ((size_t)e * 12 + dir * 4) * nnn, gb, gs, pb, ps, Acc + (le * 3 + dir) * 5 * PS);
  }
  __syncthreads();
  const R *Fsb = Buf<R>::Fsurf(d);
  if (SC) {
    // DG total (volume + surface) per node into AccT, then the FV operator into Acc
    for (int t = threadIdx.x; t < VOL_EPB * nnn; t += blockDim.x) {
      const int le = t / nnn, node = t % nnn, e = e0 + le;
      if (e >= d.nE) continue;
      const int ijk[3] = {node % n, (node / n) % n, node / nn};
      const int pn = pidx(node);
      R s[5];
#pragma unroll
      for (int v = 0; v < 5; ++v)
        s[v] = Acc[(le * 3 + 0) * 5 * PS + v * PS + pn] + Acc[(le * 3 + 1) * 5 * PS + v * PS + pn] +
               Acc[(le * 3 + 2) * 5 * PS + v * PS + pn];
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        const int id = ijk[dd];
        if (id != 0 && id != N) continue;
        const int f = 2 * dd + (id == N ? 1 : 0);
        const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
        const R *fs = Fsb + ((size_t)e * 6 + f) * 5 * nn + pp + n * qq;
#pragma unroll
        for (int v = 0; v < 5; ++v) s[v] += Tab<R>::invw(id) * fs[v * nn];
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) AccT[(le * 5 + v) * nnn + node] = s[v];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < VOL_EPB * 3 * nn; t += blockDim.x) {
      const int le = t / (3 * nn), r = t % (3 * nn), dir = r / nn, line = r % nn, e = e0 + le;
      if (e >= d.nE) continue;
      if (!(d.alpha[e] > 0.0)) continue;
      int pb, ps, gb, gs, a, b;
      line_geom(dir, line, pb, ps, gb, gs, a, b);
      const R *Fm = Fsb + ((size_t)e * 6 + 2 * dir) * 5 * nn + a + n * b;
      const R *Fp = Fsb + ((size_t)e * 6 + 2 * dir + 1) * 5 * nn + a + n * b;
      line_fv<R>(P + le * NP * PS, pb, ps, Jab + ((size_t)e * 3 + dir) * 3 * nnn, gb, gs, Fm, Fp, d.sflux, gam,
                 Cst<R>::igm1(d), pref, href, Acc + (le * 3 + dir) * 5 * PS);
    }
    __syncthreads();
  }
  // phase C: per node -- surface terms, viscous divergence, blend, Jacobian, output / LSERK
  const bool ns = d.equations == 1;
  const R *Fvb = Buf<R>::Fv(d);
  for (int t = threadIdx.x; t < VOL_EPB * nnn; t += blockDim.x) {
    const int le = t / nnn, node = t % nnn, e = e0 + le;
    if (e >= d.nE) continue;
    const int ijk[3] = {node % n, (node / n) % n, node / nn};
    const int pn = pidx(node);
    R s[5];
    if (SC) {
      const R al = (R)d.alpha[e];
#pragma unroll
      for (int v = 0; v < 5; ++v) s[v] = AccT[(le * 5 + v) * nnn + node];
      if (al > R(0)) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const R fv = Acc[(le * 3 + 0) * 5 * PS + v * PS + pn] + Acc[(le * 3 + 1) * 5 * PS + v * PS + pn] +
                       Acc[(le * 3 + 2) * 5 * PS + v * PS + pn];
          s[v] = al * fv + (R(1) - al) * s[v];
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v)
        s[v] = Acc[(le * 3 + 0) * 5 * PS + v * PS + pn] + Acc[(le * 3 + 1) * 5 * PS + v * PS + pn] +
               Acc[(le * 3 + 2) * 5 * PS + v * PS + pn];
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        const int id = ijk[dd];
        if (id != 0 && id != N) continue;
        const int f = 2 * dd + (id == N ? 1 : 0);
        const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
        const R *fs = Fsb + ((size_t)e * 6 + f) * 5 * nn + pp + n * qq;
#pragma unroll
        for (int v = 0; v < 5; ++v) s[v] += Tab<R>::invw(id) * fs[v * nn];
      }
    }
    if (ns) {
      const R *Fve = Fvb + (size_t)e * 12 * nnn;
      R vis[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        const int id = ijk[dd];
        if (SC) {  // (without the blend the line threads of phase B already added this part)
          const int st = dd == 0 ? 1 : dd == 1 ? n : nn;
          const int base = node - id * st;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            R acc = R(0);
#pragma unroll
            for (int m = 0; m < n; ++m)
              if (m != id) acc += Tab<R>::D(id * n + m) * Fve[(dd * 4 + q) * nnn + base + m * st];
            vis[q] += acc;
          }
        }
        if (id == 0 || id == N) {  // -(1/(2 w_b)) phi_nb, phi_nb = neighbour's outward normal viscous flux
          const int f = 2 * dd + (id == N ? 1 : 0);
          const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
          const int *ef = d.ef + ((size_t)e * 6 + f) * 4;
          const int nb = ef[0], fnb = ef[1], o = ef[2];
          if (nb < 0) {  // wall: (1/w_b) (F*_wall - (+-) Fv_own / 2), the wall-model flux F*_wall outward
            const R *fw = Buf<R>::Fwall(d) + (size_t)ef[3] * 4 * nn + pp + n * qq;
            const R hs = (id == N) ? R(0.5) : R(-0.5);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              vis[q] += Tab<R>::invw(id) * (fw[q * nn] - hs * Fve[(dd * 4 + q) * nnn + node]);
            continue;
          }
          int p2, q2;
          orient_map(o, pp, qq, p2, q2);
          const int nbnode = face_node(fnb, p2, q2);
          const R sg = (fnb & 1) ? R(0.5) : R(-0.5);
          const R *Fvn = Fvb + ((size_t)nb * 12 + (fnb >> 1) * 4) * nnn + nbnode;
#pragma unroll
          for (int q = 0; q < 4; ++q) vis[q] -= Tab<R>::invw(id) * sg * Fvn[q * nnn];
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) s[1 + q] -= vis[q];
    }
    const double miJ = -d.invJ[(size_t)e * nnn + node];
    const size_t gi = (size_t)e * 5 * nnn + node;
    if (mode == 0) {
#pragma unroll
      for (int v = 0; v < 5; ++v) out[gi + v * nnn] = miJ * to_double(s[v]);
    } else {
      const double fac = dt * miJ;  // the stage increment dt Ut = (dt (-1/J)) s: one multiply per node
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double du = fac * to_double(s[v]);
        const double gv = first ? du : A * g[gi + v * nnn] + du;
        g[gi + v * nnn] = gv;
        const double un = U[gi + v * nnn] + B * gv;
        out[gi + v * nnn] = un;
        if (kShift<R>) d.Uf[gi + v * nnn] = (float)(v == 4 ? un - eref : un);
      }
    }
  }
}

}  // namespace

#include "dg_fixed.cuh"  // the FP64 volume kernel in 64-bit fixed point (KG and Pirozzoli fluxes, no blend)
#include "dg_fixed_lift.cuh"  // the FP64 lifting in the same fixed point
#include "dg_fp32.cuh"   // the FP32-bulk volume and lifting kernels without the blend

namespace {

// ---------------------------------------------------------------------------------------------
// modified Persson indicator (Sec. 4.1, Eq. (7)) and the neighbour extension (FP64)
// ---------------------------------------------------------------------------------------------
// One warp per element (IND_WARPS elements per CTA): q = rho p = (gamma - 1)(rho E - |m|^2 / 2) in FP64, its modal
// coefficients by three tensor-product passes with the inverse Vandermonde in the 64-bit fixed point of
// dg_fixed.cuh (scale: the element's largest |q|), the shell energies in FP64, reduced with warp shuffles; no
// block-wide barrier after the table load. Each pass uses the parity of the Legendre modes on the symmetric
// LGL nodes, Vinv[a][N-i] = (-1)^a Vinv[a][i]: output a needs the first half of row a against q_i + q_(N-i)
// (a even) or q_i - q_(N-i) (a odd). Row sums of |Vinv| are below 1.5, so values stay below 2^59 x 1.5^3 and the
// lo sums below 2^63. The threshold T of Eq. (7) and -s/T are per-context constants from the host. Measured at
// N = 5, 32^3: 0.26 ms per launch, 0.61 with FP64 passes (FP64-bound).
constexpr int IND_WARPS = 4;
constexpr int IND_H = (n + 1) / 2;  // first half of a line, the middle node included when n is odd
__constant__ int2 c_VI[n * IND_H];  // first halves of the rows of Vinv, 2^61 (the middle node's halved when n is odd)

// one pass along a line of stride st starting at `base`: out[base + a st] = sum_i Vinv[a][i] in[base + i st]
__device__ __forceinline__ void ind_pass(const int2 *__restrict__ row, const fx_t *__restrict__ in,
                                         fx_t *__restrict__ out, int base, int st, int a) {
  FxSum s = fx_zero(3);
#pragma unroll
  for (int i = 0; i < IND_H; ++i) {
    const fx_t x = in[base + i * st], y = in[base + (N - i) * st];
    fx_acc(s, fx_const(row[i]), fx_split((a & 1) ? x - y : x + y));
  }
  out[base + a * st] = fx_value(s, 3);
}

__global__ void __launch_bounds__(32 * IND_WARPS) k_indicator(const DgDevice d, const double *__restrict__ U) {
  constexpr int IR = (nnn + 31) / 32;
  __shared__ int2 sV[n * IND_H];
  __shared__ fx_t q[IND_WARPS][nnn], t1[IND_WARPS][nnn];
  for (int t = threadIdx.x; t < n * IND_H; t += blockDim.x) sV[t] = c_VI[t];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * IND_WARPS + w;
  if (e >= d.nE) return;
  const double gm1 = d.gm1;
  fx_t *qw = q[w], *tw = t1[w];
  int hi = 0;
#pragma unroll 4
  for (int node = lane; node < nnn; node += 32) {
    const double *Ue = U + (size_t)e * 5 * nnn + node;
    const double r = Ue[0], m1 = Ue[nnn], m2 = Ue[2 * nnn], m3 = Ue[3 * nnn];
    const double x = gm1 * (r * Ue[4 * nnn] - 0.5 * (m1 * m1 + m2 * m2 + m3 * m3));
    hi = max(hi, fx_hi_abs(x));
    qw[node] = __double_as_longlong(x);
  }
  const int ex = fx_exponent(__reduce_max_sync(0xffffffffu, hi));
  double all = 0.0, shN = 0.0, shN1 = 0.0;
  if (ex >= 525 && ex < 2047) {  // (energy ratios do not depend on the scale; below 1e-150 a zero indicator)
    __syncwarp();
    for (int node = lane; node < nnn; node += 32) qw[node] = fx_from(__longlong_as_double(qw[node]), ex, 4);
    __syncwarp();
    for (int node = lane; node < nnn; node += 32) {  // xi: (i,j,k) -> (a,j,k)
      const int a = node % n;
      ind_pass(sV + a * IND_H, qw, tw, node - a, 1, a);
    }
    __syncwarp();
    for (int node = lane; node < nnn; node += 32) {  // eta
      const int b = (node / n) % n;
      ind_pass(sV + b * IND_H, tw, qw, node - b * n, n, b);
    }
    __syncwarp();
    for (int node = lane; node < IR * 32; node += 32) {  // zeta, then the shell energies
      if (node >= nnn) continue;
      const int c = node / nn;
      ind_pass(sV + c * IND_H, qw, tw, node - c * nn, nn, c);
    }
    __syncwarp();
    for (int node = lane; node < nnn; node += 32) {
      const int a = node % n, b = (node / n) % n, c = node / nn;
      const int M = max(a, max(b, c));
      const double m = (double)tw[node];
      all += m * m;
      if (M == N) shN += m * m;
      if (M == N - 1) shN1 += m * m;
    }
  } else if (ex >= 2047) {
    all = shN = shN1 = __longlong_as_double(0x7ff8000000000000ll);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    all += __shfl_down_sync(0xffffffffu, all, o);
    shN += __shfl_down_sync(0xffffffffu, shN, o);
    shN1 += __shfl_down_sync(0xffffffffu, shN1, o);
  }
  if (lane == 0) {
    const double tot = all, sN = shN, sN1 = shN1;
    double E = tot > 1e-300 ? sN / tot : 0.0;
    if (N >= 2) {
      const double tot1 = tot - sN;
      const double E1 = tot1 > 1e-300 ? sN1 / tot1 : 0.0;
      E = fmax(E, E1);
    }
    double al = 1.0 / (1.0 + exp(d.ind_k * (E - d.ind_T)));
    if (al < d.alpha_min) al = 0.0;
    if (al > d.alpha_max) al = d.alpha_max;
    d.alpha_raw[e] = al;
  }
}

__global__ void __launch_bounds__(256) k_spread(const DgDevice d, double *alpha_out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= d.nE) return;
  double a = d.alpha_raw[e];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int nb = d.ef[(e * 6 + f) * 4];
    if (nb >= 0) a = fmax(a, 0.5 * d.alpha_raw[nb]);
  }
  alpha_out[e] = a;
}

// ---------------------------------------------------------------------------------------------
// reductions: integral invariants and the time-step estimate (deterministic two-pass, FP64)
// ---------------------------------------------------------------------------------------------
__constant__ LogEntry c_log[LOG_TABLE];

__global__ void __launch_bounds__(256) k_invariants(const DgDevice d, const double *__restrict__ U,
                                                    const double *__restrict__ Ut) {
  __shared__ double red[8][256];
  __shared__ LogEntry s_log[LOG_TABLE];
  for (int t = threadIdx.x; t < LOG_TABLE; t += 256) s_log[t] = c_log[t];
  __syncthreads();
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const long long total = (long long)d.nE * nnn;
  const double gam = d.gamma;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int e = (int)(t / nnn), node = (int)(t % nnn);
    const int i = node % n, j = (node / n) % n, k = node / nn;
    const double wq = c_w[i] * c_w[j] * c_w[k] * d.J[t];
    const size_t b = (size_t)e * 5 * nnn + node;
    double Uv[5], Tv[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) { Uv[v] = U[b + v * nnn]; Tv[v] = Ut[b + v * nnn]; }
    invariants_node(gam, d.igm1, wq, Uv, Tv, acc, [&](double x) { return log_int(x, s_log); });
  }
#pragma unroll
  for (int m = 0; m < 8; ++m) red[m][threadIdx.x] = acc[m];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
#pragma unroll
      for (int m = 0; m < 8; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 8) d.red[blockIdx.x * 8 + threadIdx.x] = red[threadIdx.x][0];
}

// The partial results of the blocks, one warp per output column: lane l takes rows l, l + 32, ... in order, then a
// shuffle tree (a fixed order: deterministic). One thread per column, 1024 dependent FP64 adds, took ~100 us.
__global__ void __launch_bounds__(256) k_reduce_partials(const double *__restrict__ part, int nblocks, int width,
                                                         int op_min, double *out) {
  const int c = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (c >= width) return;
  double s = op_min ? part[c] : 0.0;
  for (int b = lane; b < nblocks; b += 32) {
    const double x = part[b * width + c];
    s = op_min ? fmin(s, x) : s + x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double x = __shfl_down_sync(0xffffffffu, s, o);
    s = op_min ? fmin(s, x) : s + x;
  }
  if (lane == 0) out[c] = s;
}

// float(x 2^(1023 - e)) for a double whose biased exponent is at most e (zero where that is below 2^-126)
__device__ __forceinline__ float scaled_float(double x, int e) {
  const int h = __double2hiint(x), ex = (h >> 20) & 0x7ff, k = ex + 1023 - e;
  const unsigned m = ((unsigned)h << 3 & 0x7fffffu) | ((unsigned)__double2loint(x) >> 29);
  return k > 897 ? __uint_as_float(((unsigned)h & 0x80000000u) | (unsigned)(k - 896) << 23 | m) : 0.0f;
}

// cfl-free time step: min over nodes of 2J / ((2N+1) sum_d (|u.Ja^d| + c|Ja^d|)). The wave speed sum takes four FP64
// square roots and a division (~75 FP64 instructions); it is estimated in FP32 first, from values scaled by their own
// exponents (to 2e-6, the products' rounding added), and evaluated in FP64 only where the estimate, with 8 units of a
// double's high word on top (at least 3.3e-6 after the estimate's truncation to one), reaches the block's largest
// sum / J so far. The node with the smallest step is never skipped, so the result is the minimum of
// the same FP64 expression. N = 5, 24^3: 210 us, 477 with every node in FP64.
__global__ void __launch_bounds__(256) k_max_dt(const DgDevice d, const double *__restrict__ U) {
  __shared__ double red[256];
  __shared__ int s_top;  // high word of the block's largest sum / J
  if (threadIdx.x == 0) s_top = 0;
  __syncthreads();
  double best = 1e300;
  const long long total = (long long)d.nE * nnn;
  const double gam = d.gamma;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int e = (int)(t / nnn), node = (int)(t % nnn);
    const size_t b = (size_t)e * 5 * nnn + node;
    const double r = U[b], ir = 1.0 / r;
    const double u = U[b + nnn] * ir, v = U[b + 2 * nnn] * ir, w = U[b + 3 * nnn] * ir;
    const double p = (gam - 1.0) * (U[b + 4 * nnn] - 0.5 * r * (u * u + v * v + w * w));
    const double c2 = gam * p * ir;
    double J[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) J[k] = d.Ja[((size_t)e * 9 + k) * nnn + node];
    const double ij = d.invJ[t];
    // the estimate: velocities scaled by 2^-(eu - 1023), c^2 by its square, Ja by 2^-(ej - 1023)
    const int hc = __double2hiint(c2) >> 20, hu = max(max(fx_hi_abs(u), fx_hi_abs(v)), fx_hi_abs(w)) >> 20;
    const int eu = max(hu, ((hc + 1023) >> 1) + 1);
    int hj = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) hj = max(hj, fx_hi_abs(J[k]));
    const int ej = hj >> 20, eij = __double2hiint(ij) >> 20;
    const float fu = scaled_float(u, eu), fv = scaled_float(v, eu), fw = scaled_float(w, eu);
    const float fc = sqrtf(scaled_float(c2, 2 * eu - 1023));
    float lam = 0.0f;
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const float x = scaled_float(J[3 * dd], ej), y = scaled_float(J[3 * dd + 1], ej), z = scaled_float(J[3 * dd + 2], ej);
      lam += fabsf(fu * x + fv * y + fw * z) + fc * sqrtf(x * x + y * y + z * z) +
             1e-6f * (fabsf(fu * x) + fabsf(fv * y) + fabsf(fw * z));  // the products may cancel
    }
    lam *= scaled_float(ij, eij);
    // its high word as a double's, with the exponents put back (a value outside FP64's range counts as large)
    const int eh = eu + ej + eij - 3 * 1023, fl = (int)__float_as_uint(lam);
    const int h = (fl >> 3) + (896 << 20), top = *(volatile int *)&s_top;
    const bool odd = hc < 0 || hc >= 2047 || hu >= 2047 || fl <= 0 || fl >= 0x7f000000 || abs(eh) > 900;
    if (odd || h + (eh << 20) + 8 >= top) {
      const double c = sqrt(c2);
      double sum = 0.0;
#pragma unroll
      for (int dd = 0; dd < 3; ++dd)
        sum += fabs(u * J[3 * dd] + v * J[3 * dd + 1] + w * J[3 * dd + 2]) +
               c * sqrt(J[3 * dd] * J[3 * dd] + J[3 * dd + 1] * J[3 * dd + 1] + J[3 * dd + 2] * J[3 * dd + 2]);
      const double x = 2.0 * d.J[t] / ((2.0 * N + 1.0) * sum);
      best = fmin(best, x);
      const int hs = __double2hiint(sum * ij);
      if (!odd && hs > top) atomicMax(&s_top, hs);
    }
  }
  red[threadIdx.x] = best;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) d.red[blockIdx.x] = red[0];
}

// ---------------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------------
cudaError_t upload(const DgTables &t) {
  if (t.N != N) return cudaErrorInvalidValue;
  double D2[nn], Dq[nn], De[nn], Dr[nn];
  float fD[nn], fD2[nn], fDq[nn], fDe[nn], fw[n], finvw[n], fxi[n], fxh[n + 1];
  for (int i = 0; i < n; ++i)
    for (int m = 0; m < n; ++m) {
      const double v = (i == m) ? 0.0 : t.D[i * n + m];
      D2[i * n + m] = 2.0 * v;
      Dq[i * n + m] = 0.25 * v;
      De[i * n + m] = 0.125 * v;
      Dr[i * n + m] = (i == m) ? 0.0 : t.D[m * n + i] / t.D[i * n + m];
      fD[i * n + m] = (float)t.D[i * n + m];
      fD2[i * n + m] = (float)D2[i * n + m];
      fDq[i * n + m] = (float)Dq[i * n + m];
      fDe[i * n + m] = (float)De[i * n + m];
    }
  for (int i = 0; i < n; ++i) { fw[i] = (float)t.w[i]; finvw[i] = (float)t.invw[i]; fxi[i] = (float)t.xi[i]; }
  for (int i = 0; i <= n; ++i) fxh[i] = (float)t.xh[i];
  double vp[EO_H * EO_H] = {0.0}, vm[EO_H * EO_H] = {0.0};
  float fvp[EO_H * EO_H] = {0.0f}, fvm[EO_H * EO_H] = {0.0f};
  if (n % 2 == 0)
    for (int i = 0; i < EO_H; ++i)
      for (int m = 0; m < EO_H; ++m) {
        const double a = (i == m) ? 0.0 : t.D[i * n + m], b = (i == N - m) ? 0.0 : t.D[i * n + (N - m)];
        vp[i * EO_H + m] = 0.5 * (a + b);
        vm[i * EO_H + m] = 0.5 * (a - b);
        fvp[i * EO_H + m] = (float)vp[i * EO_H + m];
        fvm[i * EO_H + m] = (float)vm[i * EO_H + m];
      }
  int2 VI[n * IND_H];
  for (int i = 0; i < n; ++i)
    for (int m = 0; m < IND_H; ++m)
      VI[i * IND_H + m] = fx_halves((n % 2 && m == N / 2 ? 0.5L : 1.0L) * t.Vinv[i * n + m], 61);
  double ihx[n];
  float fihx[n];
  ihx[0] = 0.0;
  for (int i = 1; i < n; ++i) ihx[i] = 1.0 / (t.xi[i] - t.xi[i - 1]);
  for (int i = 0; i < n; ++i) fihx[i] = (float)ihx[i];
  LogEntry lt[LOG_TABLE];
  log_table(lt);
  cudaError_t err = fx_upload(t);
  err = err ? err : cudaMemcpyToSymbol(c_log, lt, sizeof(lt));
  err = err ? err : fx_lift_upload(t);
  err = err ? err : cudaMemcpyToSymbol(c_ihx, ihx, sizeof(double) * n);
  err = err ? err : cudaMemcpyToSymbol(c_VP, vp, sizeof(vp));
  err = err ? err : cudaMemcpyToSymbol(c_VM, vm, sizeof(vm));
  err = err ? err : cudaMemcpyToSymbol(f_VP, fvp, sizeof(fvp));
  err = err ? err : cudaMemcpyToSymbol(f_VM, fvm, sizeof(fvm));
  err = err ? err : cudaMemcpyToSymbol(f_ihx, fihx, sizeof(float) * n);
  err = err ? err : cudaMemcpyToSymbol(c_D, t.D, sizeof(double) * nn);
  err = err ? err : cudaMemcpyToSymbol(c_D2, D2, sizeof(double) * nn);
  err = err ? err : cudaMemcpyToSymbol(c_Dq, Dq, sizeof(double) * nn);
  err = err ? err : cudaMemcpyToSymbol(c_De, De, sizeof(double) * nn);
  err = err ? err : cudaMemcpyToSymbol(c_Dr, Dr, sizeof(double) * nn);
  err = err ? err : cudaMemcpyToSymbol(c_w, t.w, sizeof(double) * n);
  err = err ? err : cudaMemcpyToSymbol(c_invw, t.invw, sizeof(double) * n);
  err = err ? err : cudaMemcpyToSymbol(c_xi, t.xi, sizeof(double) * n);
  err = err ? err : cudaMemcpyToSymbol(c_xh, t.xh, sizeof(double) * (n + 1));
  err = err ? err : cudaMemcpyToSymbol(c_VI, VI, sizeof(VI));
  err = err ? err : cudaMemcpyToSymbol(f_D, fD, sizeof(float) * nn);
  err = err ? err : cudaMemcpyToSymbol(f_D2, fD2, sizeof(float) * nn);
  err = err ? err : cudaMemcpyToSymbol(f_Dq, fDq, sizeof(float) * nn);
  err = err ? err : cudaMemcpyToSymbol(f_De, fDe, sizeof(float) * nn);
  err = err ? err : cudaMemcpyToSymbol(f_w, fw, sizeof(float) * n);
  err = err ? err : cudaMemcpyToSymbol(f_invw, finvw, sizeof(float) * n);
  err = err ? err : cudaMemcpyToSymbol(f_xi, fxi, sizeof(float) * n);
  err = err ? err : cudaMemcpyToSymbol(f_xh, fxh, sizeof(float) * (n + 1));
  return err;
}

void launch_metrics(const DgDevice &d, cudaStream_t s) {
  const size_t smem = sizeof(double) * 14 * nnn;
  cudaFuncSetAttribute(k_metrics, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_metrics<<<d.nE, 256, smem, s>>>(d);
}

void launch_face_normals(const DgDevice &d, cudaStream_t s) {
  const long long pts = (long long)d.nF * nn;
  k_face_normals<<<(unsigned)((pts + 255) / 256), 256, 0, s>>>(d);
  if (d.precision == 1) k_round_geometry<<<4 * 152, 256, 0, s>>>(d);
  else k_metric_max<<<(d.nE + 3) / 4, 128, 0, s>>>(d);
}

// launch that may be set up before the previous kernel of the stream has completed (see let_next_start); the kernel
// calls wait_for_previous before it touches anything a kernel writes
template <typename... P, typename... T>
void launch_after(void (*k)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s, T... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k, static_cast<P>(args)...);
}

template <typename R>
void launch_face_t(const DgDevice &d, const double *U, cudaStream_t s) {
  const long long pts = (long long)d.nF * nn;
  const unsigned grid = (unsigned)((pts + FACE_THREADS - 1) / FACE_THREADS);
  switch (d.sflux) {
    case SF_LLF: launch_after(k_face<R, SF_LLF>, grid, FACE_THREADS, 0, s, d, U); break;
    case SF_ROE: launch_after(k_face<R, SF_ROE>, grid, FACE_THREADS, 0, s, d, U); break;
    default: launch_after(k_face<R, SF_EC>, grid, FACE_THREADS, 0, s, d, U); break;
  }
}

void launch_face(const DgDevice &d, const double *U, cudaStream_t s) {
  if (d.precision == 1) launch_face_t<float>(d, U, s);
  else launch_face_t<double>(d, U, s);
}

void launch_lift(const DgDevice &d, const double *U, double *tau, cudaStream_t s) {
  if (TMA_OK && d.precision == 1 && d.use_tma) {  // FP32-bulk: the TMA-fed persistent form
    static int grid_lt = 0;
    if (!grid_lt) {
      cudaFuncSetAttribute(k_lift_f32_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LT_SMEM);
      int dev = 0, sms = 0, per_sm = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lift_f32_tma, LT_THREADS, LT_SMEM);
      grid_lt = sms * (per_sm > 0 ? per_sm : 1);
    }
    const int blocks = d.nE < grid_lt ? d.nE : grid_lt;
    k_lift_f32_tma<<<blocks, LT_THREADS, LT_SMEM, s>>>(d);
    return;
  }
  if (d.precision == 1) {
    k_lift<<<(d.nE + LIFT_EPB - 1) / LIFT_EPB, LIFT_THREADS, 0, s>>>(d);
    return;
  }
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_lift_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FXL_SMEM);
    attr_set = true;
  }
  launch_after(k_lift_fx, (d.nE + FX_EPB - 1) / FX_EPB, FX_THREADS, FXL_SMEM, s, d, U, tau);
}

template <typename R, int VF, bool SC>
void launch_volume_t(const DgDevice &d, const double *U, double *out, double *g, int mode, int first, double dt,
                     double A, double B, cudaStream_t s) {
  const size_t smem =
      sizeof(R) * (VOL_EPB * vol_np<SC>() * PS + VOL_EPB * 15 * PS + (SC ? VOL_EPB * 5 * nnn : 0));
  static bool attr_set = false;  // per instantiation; setting it twice is harmless
  if (!attr_set) {
    cudaFuncSetAttribute(k_volume<R, VF, SC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  k_volume<R, VF, SC><<<(d.nE + VOL_EPB - 1) / VOL_EPB, vol_threads<R, SC>(), smem, s>>>(d, U, out, g, mode, first, dt, A,
                                                                                    B);
}

template <int VF, bool SC>
void launch_volume_fx(const DgDevice &d, const double *U, double *out, double *g, int mode, int first, double dt,
                      double A, double B, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_volume_fx<VF, SC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_SMEM);
    attr_set = true;
  }
  launch_after(k_volume_fx<VF, SC>, (d.nE + FX_EPB - 1) / FX_EPB, FX_THREADS, FX_SMEM, s, d, U, out, g, mode, first, dt, A, B);
}

template <int VF>
void launch_volume_f32(const DgDevice &d, const double *U, double *out, double *g, int mode, int first, double dt,
                       double A, double B, cudaStream_t s) {
  const bool aligned = !(((uintptr_t)U | (uintptr_t)out | (uintptr_t)g) & 15u);
  // pair-symmetric line kernel, warp-specialised. Its warp groups trade registers (setmaxnreg), which
  // is only safe if the block is launched with exactly the registers the split assumes; any other
  // compiled count takes the plain node kernel instead.
  static int grid_ln = 0;  // > 0: usable, < 0: not usable
  if (LN_OK && d.use_tma == 3 && aligned && grid_ln == 0) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, k_volume_f32_line<VF>) == cudaSuccess && fa.numRegs == LN_REG_LAUNCH) {
      cudaFuncSetAttribute(k_volume_f32_line<VF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LN_SMEM);
      int dev = 0, sms = 0, per_sm = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_volume_f32_line<VF>, LN_THREADS, LN_SMEM);
      grid_ln = per_sm == 1 ? sms : -1;  // one block per SM: the register split needs the whole file
    } else {
      grid_ln = -1;
    }
  }
  if (LN_OK && d.use_tma == 3 && aligned && grid_ln > 0) {
    const int blocks = d.nE < grid_ln ? d.nE : grid_ln;
    k_volume_f32_line<VF><<<blocks, LN_THREADS, LN_SMEM, s>>>(d, U, out, g, mode, first, dt, A, B);
    return;
  }
  // warp-specialised persistent kernel, on request: its few warps per SM leave it behind another form at every degree, with
  // the same bits. At N = 3 and 5 that is the TMA-fed node kernel below (right-hand side / LSERK stage: N = 5,
  // 17 x 13 x 11: 69.6 / 74 against 45.2 / 54 us; 32^3: 903 / 945 against 529 / 641 us; N = 3, 32^3: 373 / 380 against
  // 128 / 163 us); at N = 7, where the line kernel cannot run, the plain one (stage at 32^3: 1470 against 1363 us, TMA-fed
  // 1679, line kernel 1017)
  if (TMA_OK && d.use_tma == 2 && aligned) {
    static int grid_ws = 0;
    if (!grid_ws) {
      cudaFuncSetAttribute(k_volume_f32_ws<VF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WS_SMEM);
      int dev = 0, sms = 0, per_sm = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_volume_f32_ws<VF>, WS_THREADS, WS_SMEM);
      grid_ws = sms * (per_sm > 0 ? per_sm : 1);
    }
    const int blocks = d.nE < grid_ws ? d.nE : grid_ws;
    k_volume_f32_ws<VF><<<blocks, WS_THREADS, WS_SMEM, s>>>(d, U, out, g, mode, first, dt, A, B);
    return;
  }
  if (TMA_OK && (d.use_tma == 1 || (d.use_tma == 3 && !LN_OK)) && aligned) {
    static int grid = 0;  // persistent: CTAs resident on all SMs at once
    if (!grid) {
      cudaFuncSetAttribute(k_volume_f32_tma<VF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TB_SMEM);
      int dev = 0, sms = 0, per_sm = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_volume_f32_tma<VF>, TMA_THREADS, TB_SMEM);
      grid = sms * (per_sm > 0 ? per_sm : 1);
    }
    const int blocks = d.nE < grid ? d.nE : grid;
    k_volume_f32_tma<VF><<<blocks, TMA_THREADS, TB_SMEM, s>>>(d, U, out, g, mode, first, dt, A, B);
    return;
  }
  const size_t smem = sizeof(float) * NODE_EPB * NODE_SLOTS * nnn;
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_volume_f32<VF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  k_volume_f32<VF><<<(d.nE + NODE_EPB - 1) / NODE_EPB, NODE_THREADS, smem, s>>>(d, U, out, g, mode, first, dt, A, B);
}

// k_volume: FP32 under the blend (any flux), and in FP64 the fluxes that have no fixed-point form (EC, central)
template <typename R, bool SC>
void launch_volume_lines(const DgDevice &d, const double *U, double *out, double *g, int mode, int first, double dt,
                         double A, double B, cudaStream_t s) {
  if constexpr (std::is_same<R, float>::value) {
    if (d.vflux == VF_KG) { launch_volume_t<R, VF_KG, SC>(d, U, out, g, mode, first, dt, A, B, s); return; }
    if (d.vflux == VF_PIR) { launch_volume_t<R, VF_PIR, SC>(d, U, out, g, mode, first, dt, A, B, s); return; }
  }
  if (d.vflux == VF_EC) launch_volume_t<R, VF_EC, SC>(d, U, out, g, mode, first, dt, A, B, s);
  else launch_volume_t<R, VF_CEN, SC>(d, U, out, g, mode, first, dt, A, B, s);
}

void launch_volume(const DgDevice &d, const double *U, double *out, double *g, int mode, int first, double dt,
                   double A, double B, cudaStream_t s) {
  const bool sc = d.shock_capturing != 0;
  if (d.precision == 1 && sc) {
    launch_volume_lines<float, true>(d, U, out, g, mode, first, dt, A, B, s);
  } else if (d.precision == 1) {
    switch (d.vflux) {
      case VF_KG: launch_volume_f32<VF_KG>(d, U, out, g, mode, first, dt, A, B, s); break;
      case VF_PIR: launch_volume_f32<VF_PIR>(d, U, out, g, mode, first, dt, A, B, s); break;
      case VF_EC: launch_volume_f32<VF_EC>(d, U, out, g, mode, first, dt, A, B, s); break;
      default: launch_volume_f32<VF_CEN>(d, U, out, g, mode, first, dt, A, B, s); break;
    }
  } else if (d.vflux == VF_KG) {
    if (sc) launch_volume_fx<VF_KG, true>(d, U, out, g, mode, first, dt, A, B, s);
    else launch_volume_fx<VF_KG, false>(d, U, out, g, mode, first, dt, A, B, s);
  } else if (d.vflux == VF_PIR) {
    if (sc) launch_volume_fx<VF_PIR, true>(d, U, out, g, mode, first, dt, A, B, s);
    else launch_volume_fx<VF_PIR, false>(d, U, out, g, mode, first, dt, A, B, s);
  } else {
    if (sc) launch_volume_lines<double, true>(d, U, out, g, mode, first, dt, A, B, s);
    else launch_volume_lines<double, false>(d, U, out, g, mode, first, dt, A, B, s);
  }
}

void launch_indicator(const DgDevice &d, const double *U, cudaStream_t s) {
  k_indicator<<<(d.nE + IND_WARPS - 1) / IND_WARPS, 32 * IND_WARPS, 0, s>>>(d, U);
}

void launch_shadow(const DgDevice &d, const double *U, cudaStream_t s) {
  constexpr int V = nnn % 4 == 0 ? 4 : 1;
  if (((uintptr_t)U & 15u) == 0) k_shadow<V><<<8 * 152, 256, 0, s>>>(d, U);
  else k_shadow<1><<<8 * 152, 256, 0, s>>>(d, U);
}

void launch_spread(const DgDevice &d, double *alpha_out, cudaStream_t s) {
  k_spread<<<(d.nE + 255) / 256, 256, 0, s>>>(d, alpha_out);
}

void launch_invariants(const DgDevice &d, const double *U, const double *Ut, double *out8, cudaStream_t s) {
  const long long total = (long long)d.nE * nnn;
  int blocks = (int)((total + 255) / 256);
  if (blocks > DG_RED_BLOCKS) blocks = DG_RED_BLOCKS;
  k_invariants<<<blocks, 256, 0, s>>>(d, U, Ut);
  k_reduce_partials<<<1, 256, 0, s>>>(d.red, blocks, 8, 0, out8);
}

void launch_max_dt(const DgDevice &d, const double *U, double *out, cudaStream_t s) {
  const long long total = (long long)d.nE * nnn;
  int blocks = (int)((total + 255) / 256);
  if (blocks > DG_RED_BLOCKS) blocks = DG_RED_BLOCKS;
  k_max_dt<<<blocks, 256, 0, s>>>(d, U);
  k_reduce_partials<<<1, 32, 0, s>>>(d.red, blocks, 1, 1, out);
}

}  // namespace
