// dg_fixed_lift.cuh -- the FP64 BR1 lifting (reference derivatives of u, v, w, T, their contraction with the
// metric terms, the viscous flux and its contravariant projection) in the 64-bit fixed point of
// dg_fixed.cuh. Part of dg_kernels.cuh (same unnamed namespace).
//
// Per node the lifting is 24 products of the derivative sums (even-odd halves), 48 of the metric contraction,
// 22 of the stress and the heat flux and 36 of the projection: ~200 FP64 instructions (~100 clocks per
// lane and SM) or 130 x 3 IMAD.WIDE (~16 clocks). The derivatives are those of Q = W D, D's diagonal
// (-1/2 and 1/2 at the ends) included; the BR1 face jump w* - w of a direction adds to its end nodes' sums
// with weight -1 and 1, and the weights 1 / w_d of the three directions enter as ratios to the largest.
// A derivative is a sum with cancellation: FP64 forms it to 2^-53 of sum |D_im w_m|, this form to 2^-59 of
// the element's largest value, and later products keep that absolute resolution: FP64's accuracy in the norm of the
// stress over the element, not for each of its components (see fx_lift_exponents).
#pragma once

namespace {

// rows of the derivative sums: n even, row i < n/2 the even half of Q, row N - i the odd half, 2^62; n odd,
// the whole rows, 2^61
__constant__ int2 c_QD[n * FX_QV];
constexpr int FX_DA = n % 2 == 0 ? 1 : 2;  // their window: the sums carry one bit less than the values

struct FxLift {
  int ok;
  int eu, et, ej, em, ek;  // exponents of velocity and T (jumps included), metric terms, mu/(J w), kappa/(J w)
  int bu, bt;              // left shifts that bring the element's largest reference derivatives to full size
  int he, hk;              // right shifts of u.tau and of the heat flux to their common scale
  int kt, km, ke;          // stress, momentum and energy fluxes are fixed value x 2^k
  int e[3];                // 2^20 times the metric terms' e_d (for fvmax)
};

// exponents, before the derivative sums. The three directions' terms of J grad w are added at the scale of the largest metric
// term, so on a stretched element the stress between two small velocity components is resolved at 2^-59 of the largest
// one's. That stays below the rounding of the pressure flux in FP64 unless the element is dominated by viscosity:
// tested where the directions' metric terms differ by more than 4, from bounds of the viscous flux
// (mu/J) max|Ja|^2 max|w| / w_0 and of the smallest pressure flux, with the pressure of the element's first node.
__device__ __forceinline__ FxLift fx_lift_exponents(const DgDevice &d, const double *U, int e, int mu_, int mt) {
  FxLift s;
  const int4 mj = d.jmax[e];
  const double ij = d.ijmax[e] * c_invw[0], muj = d.mu * ij, kaj = d.kappa * ij;
  const int h = max(mj.x, max(mj.y, mj.z)), hs = min(mj.x, min(mj.y, mj.z));
  s.e[0] = fx_unit(mj.x) << 20; s.e[1] = fx_unit(mj.y) << 20; s.e[2] = fx_unit(mj.z) << 20;
  s.eu = fx_exponent(mu_); s.et = fx_exponent(mt); s.ej = fx_exponent(h);
  s.em = fx_exponent(__double2hiint(muj)); s.ek = fx_exponent(__double2hiint(kaj));
  const int lo = min(min(s.et, s.ej), min(s.em, s.ek)), hi = max(max(s.et, s.ej), max(max(s.em, s.ek), s.eu));
  s.ok = lo >= 800 && hi <= 1150;
  if (h - hs > (2 << 20)) {
    double Uv[5];
    load_state<double>(d, U, e, 0, Uv);
    const int p = __double2hiint(d.gm1 * (Uv[4] - 0.5 * (Uv[1] * Uv[1] + Uv[2] * Uv[2] + Uv[3] * Uv[3]) / Uv[0]));
    s.ok = s.ok && p > 0 && s.em + 2 * s.ej + s.eu - 2046 <= 1 + (p >> 20) + (hs >> 20);
  }
  // a fluid at rest has no scale of its own; the floor is 2^-32 sqrt(kappa T / mu)
  s.eu = max(s.eu, (959 - s.em + s.et + s.ek) >> 1);
  s.ok = s.ok && s.eu <= 1150;
  return s;
}

// Scales, from the high words of the largest derivative sums times w_0 / w (the reference derivatives times w_0). Bounds (value x scale, log2): u, v, w, T, Ja < 60,
// jumps < 59; derivative sums < 61.3, times w_0 / w shifted left to at most that; J grad w < 59.9; tau < 61.3, u.tau and heat
// flux < 61.9 before their shifts, energy flux < 61.9; contravariant fluxes < 62.5
__device__ __forceinline__ void fx_lift_scales(FxLift &s, int yu, int yt) {
  s.bu = min(max(__clz(yu + 1) - 3, 0), 24);
  s.bt = min(max(__clz(yt + 1) - 3, 0), 24);
  const int sj = 1082 - s.ej, sw = 1082 - s.eu, sT = 1082 - s.et;
  const int st = (sw - 1 + s.bu) + sj - 63 + (1084 - s.em) - 62;
  const int se = st + sw - 61, sk = (sT - 1 + s.bt) + sj - 63 + (1084 - s.ek) - 60;
  const int sE = min(se, sk) - 1;
  s.he = min(se - sE, 62);  // (a share that far below the other rounds away)
  s.hk = min(sk - sE, 62);
  s.kt = -st; s.km = -(st + sj - 61); s.ke = -(sE + sj - 61);
}

__device__ __forceinline__ double fx_to(fx_t x, int k) {  // x 2^k (k keeps the exponent in range)
  const double v = (double)x;
  return x == 0 ? 0.0 : __hiloint2double(__double2hiint(v) + (int)((unsigned)k << 20), __double2loint(v));
}

__device__ __noinline__ void fx_general_lift(const DgDevice &d, size_t e, int node, const double *W,
                                             const double (*sD)[n + 1], double *tau, const int *unit, int *fvm) {
  lift_node<double>(d, node, W, sD, d.Ja + e * 9 * nnn, d.Wsurf + e * 24 * nn, d.invJ[e * nnn + node], d.mu, d.kappa,
                    d.Fv + e * 12 * nnn, tau ? tau + e * 6 * nnn : nullptr, unit, fvm);
}

// element slots: 0-3 u, v, w, T; 4 + 4 dir + q derivative sums; then the face jumps [6][4][nn]
constexpr int FXL_SLOTS = 16;
constexpr int FXL_ELEM = FXL_SLOTS * FX_PS + 24 * nn;
constexpr size_t FXL_SMEM = sizeof(fx_t) * FX_EPB * FXL_ELEM;

// One thread per node, phases as in k_volume_fx. What bounds it: instruction issue (49 % of the slots) and the
// latencies between its four barriers; FMA-heavy 41 %, ALU 48 %, FP64 pipe 35 %, DRAM 20 %. Measured per launch
// at N = 7, 24^3: 1.00 ms (the FP64 line sweeps with a node-wise contraction 2.57 ms); N = 5, 24 x 12 x 12: 0.123
// against 0.277 ms.
__global__ void __launch_bounds__(FX_THREADS, FX_MINB) k_lift_fx(const DgDevice d, const double *U, double *tau) {
  constexpr int JR = (FX_EPB * 24 * nn + FX_THREADS - 1) / FX_THREADS;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  fx_t *S = reinterpret_cast<fx_t *>(sm_raw);  // [EPB][FXL_ELEM]
  __shared__ int s_mx[FX_EPB][2], s_my[FX_EPB][2], s_fv[FX_EPB][2];
  __shared__ FxLift s_sc[FX_EPB];
  __shared__ int2 s_rho[FX_H], s_QD[n * FX_QV];
  const int e0 = blockIdx.x * FX_EPB, tid = threadIdx.x;
  if (tid < 2 * FX_EPB) s_mx[tid >> 1][tid & 1] = s_my[tid >> 1][tid & 1] = s_fv[tid >> 1][tid & 1] = 0;
  for (int t = tid; t < FX_H; t += FX_THREADS) s_rho[t] = c_rho[t * FX_H];  // w_0 / w
  for (int t = tid; t < n * FX_QV; t += FX_THREADS) s_QD[t] = c_QD[t];
  wait_for_previous();
  __syncthreads();
  const int le = tid / nnn, node = tid % nnn, e = e0 + le;
  const bool on = tid < FX_EPB * nnn && e < d.nE;
  // phase A: (u, v, w, T) of the thread's node, the element's face jumps, and their maxima
  double wv[4], jv[JR];
  int mu_ = 0, mt = 0;
  if (on) {
    double Uv[5];
    load_state<double>(d, U, e, node, Uv);
    lift_prim<double>(Uv, d.gm1, d.iR, 0.0, wv);
    mu_ = max(max(fx_hi_abs(wv[0]), fx_hi_abs(wv[1])), fx_hi_abs(wv[2]));
    mt = fx_hi_abs(wv[3]);
  }
#pragma unroll
  for (int k = 0; k < JR; ++k) {
    const int t = tid + k * FX_THREADS, lj = t / (24 * nn);
    if (t >= FX_EPB * 24 * nn || e0 + lj >= d.nE) continue;
    jv[k] = d.Wsurf[(size_t)e0 * 24 * nn + t];
    const int h = fx_hi_abs(jv[k]);
    if (FX_EPB > 1) atomicMax(&s_mx[lj][(t / nn) % 4 == 3 ? 1 : 0], h);
    else if ((t / nn) % 4 == 3) mt = max(mt, h);
    else mu_ = max(mu_, h);
  }
  if (FX_EPB == 1) {
    mu_ = __reduce_max_sync(0xffffffffu, mu_);
    mt = __reduce_max_sync(0xffffffffu, mt);
  }
  if (FX_EPB == 1 ? (tid & 31) == 0 : on) {
    atomicMax(&s_mx[le][0], mu_);
    atomicMax(&s_mx[le][1], mt);
  }
  __syncthreads();
  int good = 1;
  if (tid < FX_EPB && e0 + tid < d.nE) {
    s_sc[tid] = fx_lift_exponents(d, U, e0 + tid, s_mx[tid][0], s_mx[tid][1]);
    good = s_sc[tid].ok;
  }
  const bool ok = __syncthreads_and(good);
  fx_t *Se = S + le * FXL_ELEM;
  int fvm[2] = {0, 0};
  if (ok) {
    if (on) {
      const int eu = s_sc[le].eu, et = s_sc[le].et;
#pragma unroll
      for (int q = 0; q < 4; ++q) Se[q * FX_PS + fx_idx(node)] = fx_from(wv[q], q < 3 ? eu : et, 3);
    }
#pragma unroll
    for (int k = 0; k < JR; ++k) {
      const int t = tid + k * FX_THREADS, lj = t / (24 * nn), r = t % (24 * nn);
      if (t >= FX_EPB * 24 * nn || e0 + lj >= d.nE) continue;
      S[lj * FXL_ELEM + FXL_SLOTS * FX_PS + r] = fx_from(jv[k], (r / nn) % 4 == 3 ? s_sc[lj].et : s_sc[lj].eu, 4);
    }
    __syncthreads();
    // phase B: derivative sums along the three directions, one lane per node of a line
    constexpr int GROUPS = (FX_EPB * nn + FX_LPW - 1) / FX_LPW;
    const int lane = tid & 31, idx = lane % n, l0 = (lane / n) % FX_LPW * n;
    const bool low = idx < EO_H;
    const int rw = s_rho[min(idx, N - idx)].x;
    int yu = 0, yt = 0;  // high words of the largest sums times w_0 / w
    for (int gr = tid >> 5; gr < 3 * GROUPS; gr += FX_THREADS / 32) {
      const int dir = gr / GROUPS, g0 = (gr % GROUPS) * FX_LPW;
      const bool own = lane < FX_LPW * n && g0 + lane / n < FX_EPB * nn;
      const int ln = own ? g0 + lane / n : g0;  // lanes without a line of their own repeat the group's first one
      const int lel = ln / nn, ll = ln % nn, la = ll % n, lb = ll / n;
      const int ps = dir == 0 ? 1 : dir == 1 ? FX_SJ : FX_SK;
      const int pb = dir == 0 ? FX_SJ * la + FX_SK * lb : dir == 1 ? la + FX_SK * lb : la + FX_SJ * lb;
      fx_t *Sl = S + lel * FXL_ELEM;
      const fx_t *jp = Sl + FXL_SLOTS * FX_PS + (2 * dir + (idx == N ? 1 : 0)) * 4 * nn + la + n * lb;
      const int2 *row = s_QD + idx * FX_QV;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const fx_t f = Sl[q * FX_PS + pb + idx * ps];
        FxSum s = fx_zero(FX_DA);
        fx_t y;
        if constexpr (n % 2 == 0) {
          const fx_t g = __shfl_sync(0xffffffffu, f, l0 + N - idx);
          const FxD h = fx_split(low ? f + g : g - f);
#pragma unroll
          for (int m = 0; m < EO_H; ++m) {
            const int src = l0 + (low ? m : N - m);
            fx_acc(s, fx_const(row[m]),
                   FxD{__shfl_sync(0xffffffffu, h.h, src), __shfl_sync(0xffffffffu, h.l, src)});
          }
          y = fx_value(s, FX_DA);
          const fx_t z = __shfl_sync(0xffffffffu, y, l0 + N - idx);
          y = low ? y + z : y - z;
        } else {
          const FxD h = fx_split(f);
#pragma unroll
          for (int m = 0; m < n; ++m)
            fx_acc(s, fx_const(row[m]),
                   FxD{__shfl_sync(0xffffffffu, h.h, l0 + m), __shfl_sync(0xffffffffu, h.l, l0 + m)});
          y = fx_value(s, FX_DA);
        }
        if (idx == 0) y -= jp[q * nn];
        if (idx == N) y += jp[q * nn];
        if (own) Sl[(4 + 4 * dir + q) * FX_PS + pb + idx * ps] = y;
        const int h = __mulhi((int)((y ^ (y >> 63)) >> 32), rw) * 4 + 4;
        if (FX_EPB > 1) atomicMax(&s_my[lel][q / 3], h);
        else if (q < 3) yu = max(yu, h);
        else yt = max(yt, h);
      }
    }
    if (FX_EPB == 1) {
      yu = __reduce_max_sync(0xffffffffu, yu);
      yt = __reduce_max_sync(0xffffffffu, yt);
      if (lane == 0) {
        atomicMax(&s_my[0][0], yu);
        atomicMax(&s_my[0][1], yt);
      }
    }
    __syncthreads();
    if (tid < FX_EPB) fx_lift_scales(s_sc[tid], s_my[tid][0], s_my[tid][1]);
    __syncthreads();
    let_next_start();
    // phase C: per node -- metric contraction, stress, heat flux, contravariant viscous flux
    if (on) {
      const FxLift &c = s_sc[le];
      const double *Je = d.Ja + (size_t)e * 9 * nnn + node;
      const double ij = d.invJ[(size_t)e * nnn + node];
      FxD J[3][3];
#pragma unroll
      for (int k = 0; k < 9; ++k) J[k / 3][k % 3] = fx_split(fx_from(__ldg(Je + k * nnn), c.ej, 3));
      const int ijk[3] = {node % n, (node / n) % n, node / nn};
      FxD r[3];
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) r[dd] = fx_const(s_rho[min(ijk[dd], N - ijk[dd])]);
      const double ijw = ij * c_invw[0];
      const fx_t *Sn = Se + fx_idx(node);
      auto grad = [&](int q, fx_t g[3]) {  // J grad w_q times w_0
        const int aw = 2 + (q < 3 ? c.bu : c.bt);
        FxD y[3];
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) {
          FxSum s = fx_zero_biased(aw);
          fx_acc(s, r[dd], fx_split(Sn[(4 + 4 * dd + q) * FX_PS]));
          y[dd] = fx_biased(fx_value(s, aw));
        }
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
          FxSum s = fx_zero(1);
#pragma unroll
          for (int dd = 0; dd < 3; ++dd) fx_acc(s, J[dd][cc], y[dd]);
          g[cc] = fx_value(s, 1);
        }
      };
      fx_t gu[3], gv[3], gw[3];
      grad(0, gu);
      grad(1, gv);
      grad(2, gw);
      const FxD M = fx_split(fx_from(d.mu * ijw, c.em, 1));
      const FxD third{0x2AAAAAAB, (int)0xAAAAAAABu};  // 2/3, 2^62
      auto scaled = [&](fx_t x) {                    // x mu / (J w_0)
        FxSum s = fx_zero_biased(2);
        fx_acc(s, M, fx_split(x));
        return fx_value(s, 2);
      };
      auto normal = [&](fx_t x) {  // two thirds of x, scaled
        FxSum s = fx_zero(2);
        fx_acc(s, third, fx_split(x));
        return scaled(fx_value(s, 2));
      };
      FxD t[6];  // xx, yy, zz, xy, xz, yz
      {
        const fx_t b[6] = {normal(2 * gu[0] - gv[1] - gw[2]), normal(2 * gv[1] - gu[0] - gw[2]),
                           normal(2 * gw[2] - gu[0] - gv[1]), scaled(gu[1] + gv[0]), scaled(gu[2] + gw[0]),
                           scaled(gv[2] + gw[1])};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          t[k] = fx_biased(b[k]);
          if (tau) tau[((size_t)e * 6 + k) * nnn + node] = fx_to(b[k] - FX_BIAS, c.kt);
        }
      }
      double *out = d.Fv + (size_t)e * 12 * nnn + node;
      int fm[3] = {0, 0, 0};
      auto project = [&](int q, FxD f0, FxD f1, FxD f2) {
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) {
          FxSum s = fx_zero(3);
          fx_acc(s, J[dd][0], f0);
          fx_acc(s, J[dd][1], f1);
          fx_acc(s, J[dd][2], f2);
          const double f = fx_to(fx_value(s, 3), q < 3 ? c.km : c.ke);
          out[(dd * 4 + q) * nnn] = f;
          fm[dd] = max(fm[dd], fx_hi_abs(f));  // (finite, below 2^700)
        }
      };
      project(0, t[0], t[3], t[4]);
      project(1, t[3], t[1], t[5]);
      project(2, t[4], t[5], t[2]);
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) {
        fvm[0] = max(fvm[0], fm[dd] - c.e[dd]);
        fm[dd] = 0;
      }
      fx_t gt[3];
      grad(3, gt);
      const FxD K = fx_split(fx_from(d.kappa * ijw, c.ek, 1));
      const FxD u = fx_split(Sn[0]), v = fx_split(Sn[FX_PS]), w = fx_split(Sn[2 * FX_PS]);
      auto energy = [&](FxD tx, FxD ty, FxD tz, fx_t g) {
        FxSum s = fx_zero(3), k = fx_zero(4);
        fx_acc(s, u, tx);
        fx_acc(s, v, ty);
        fx_acc(s, w, tz);
        fx_acc(k, K, fx_split(g));
        return fx_split(fx_shr(fx_value(s, 3), c.he) + fx_shr(fx_value(k, 4), c.hk));
      };
      project(3, energy(t[0], t[3], t[4], gt[0]), energy(t[3], t[1], t[5], gt[1]), energy(t[4], t[5], t[2], gt[2]));
#pragma unroll
      for (int dd = 0; dd < 3; ++dd) fvm[1] = max(fvm[1], fm[dd] - c.e[dd]);
    }
  } else {  // general path: FP64
    double *W = reinterpret_cast<double *>(S);  // [EPB][4][nnn], then D padded
    double(*sD)[n + 1] = reinterpret_cast<double(*)[n + 1]>(W + FX_EPB * 4 * nnn);
    if (on) {
#pragma unroll
      for (int q = 0; q < 4; ++q) W[(le * 4 + q) * nnn + node] = wv[q];
    }
    for (int t = tid; t < nn; t += FX_THREADS) sD[t / n][t % n] = c_D[t];
    __syncthreads();
    if (on) {
      int m[2] = {0, 0};
      fx_general_lift(d, e, node, W + le * 4 * nnn, sD, tau, s_sc[le].e, m);
      fvm[0] = m[0];
      fvm[1] = m[1];
    }
  }
  // the element's largest viscous flux components, for the volume kernel's scales
  if (FX_EPB == 1) {
    fvm[0] = __reduce_max_sync(0xffffffffu, fvm[0]);
    fvm[1] = __reduce_max_sync(0xffffffffu, fvm[1]);
  }
  if (FX_EPB == 1 ? (tid & 31) == 0 : on) {
    atomicMax(&s_fv[le][0], fvm[0]);
    atomicMax(&s_fv[le][1], fvm[1]);
  }
  __syncthreads();
  if (tid < 2 * FX_EPB && e0 + (tid >> 1) < d.nE) d.fvmax[2 * e0 + tid] = s_fv[tid >> 1][tid & 1];
}

cudaError_t fx_lift_upload(const DgTables &t) {
  int2 QD[n * FX_QV];
  for (int i = 0; i < n; ++i)
    for (int m = 0; m < FX_QV; ++m) {
      auto q = [&](int a, int b) { return a != b ? t.Q[a * n + b] : a == 0 ? -0.5L : a == N ? 0.5L : 0.0L; };
      long double v = q(i, m);
      if (n % 2 == 0 && i < n / 2) v = (v + q(i, N - m)) / 2;
      else if (n % 2 == 0) v = (q(N - i, m) - q(N - i, N - m)) / 2;
      QD[i * FX_QV + m] = fx_halves(v, n % 2 == 0 ? 62 : 61);
    }
  return cudaMemcpyToSymbol(c_QD, QD, sizeof(QD));
}

}  // namespace
