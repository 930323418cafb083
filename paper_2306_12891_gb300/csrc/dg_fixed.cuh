// dg_fixed.cuh -- the FP64 volume kernel for the Kennedy-Gruber and Pirozzoli fluxes, its two-point fluxes and viscous divergence evaluated in 64-bit fixed point on the integer pipes. Part
// of dg_kernels.cuh (same unnamed namespace); works on the degree constants defined there.
//
// Why: GB300 issues FP64 arithmetic at 2 lanes per clock and SM, IMAD.WIDE at 25 and 64-bit integer adds
// at 55 (measured). A pair flux is 30 FP64 instructions (~16 clocks per lane and SM); in fixed point it is
// 13 products of three IMAD.WIDE each and ~40 adds and shifts (~2 clocks).
//
// Format: per element every quantity (the metric terms: per direction) is scaled by a power of two taken from the
// element's largest value of it, X = x 2^s with |X| < 2^62 (rho, p) or 2^60 (the rest): an FP64 significand has 53 bits, so an input
// is exact down to 2^-7 of the element's maximum. A product keeps the high 64 of 128 bits: with X = 2^32 h +
// l, h and l signed 32-bit halves, it is h h' + (h l' + l h') / 2^32; the dropped l l' is below a quarter
// unit. Every product is rounded to nearest in a window chosen per element (FxScale), so that the largest
// value it can take fills the word. Pair sums and sums over a line are exact integer adds, so with the pair symmetry
// Q_im = -Q_mi of the SBP operator Q = W D the two shares of a pair, formed once and handed on, cancel exactly (the pairs
// half a line apart at even n are formed at both nodes, with opposite factors, and cancel to a unit: products round half up).
// Precision: all rounding happens at about 2^-61 of the largest flux sum the element can have, where FP64
// rounds each flux and each partial sum at 2^-53 of itself, and values are held to 2^-60 of the element's largest of
// their kind. So the results are those of FP64 normwise, per element and variable; what is small beside the rest of its
// element (a velocity component far below the largest, say) is not held to 53 bits of its own. An element takes the general FP64 path of the
// same kernel (fx_general_lines) instead when a value is not finite, rho, p or h (e) is not positive or
// spans more than 2^8 within the element, the exponents of its metric terms differ by more than FX_JSPAN (a stretch beyond 8 to
// 16), or the exponents leave a safe range.
#pragma once

namespace {

typedef long long fx_t;

__constant__ int2 c_Qx[nn];                       // Q_im = w_i D_im, zero diagonal, 2^63, halves (h, l)
// rows of the viscous divergence, 2^62: n even, row i < n/2 the even half of Q, row N - i the odd half (n/2 each);
// n odd, Q itself
constexpr int FX_QV = n % 2 == 0 ? EO_H : n;
__constant__ int2 c_QV[n * FX_QV];
constexpr int FX_H = (n + 1) / 2;                 // distinct node weights
__constant__ int2 c_DT[nn];                       // [i][m] = D_mi / 32, zero diagonal, 2^62 (the adjoint's sweeps)
__constant__ int2 c_rho[FX_H * FX_H];             // min(w_a, w_b) / w_a, 2^62: [a][b], a, b = distance to the face

__device__ __forceinline__ fx_t fx_mad(int a, int b, fx_t c) {
  fx_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// balanced halves of X = 2^32 h + l, l in [-2^31, 2^31), from X + 2^31
struct FxD {
  int h, l;
};
constexpr fx_t FX_BIAS = 0x80000000ll;
__device__ __forceinline__ FxD fx_biased(fx_t x) { return FxD{(int)(x >> 32), (int)x ^ (int)0x80000000}; }
__device__ __forceinline__ FxD fx_split(fx_t x) { return fx_biased(x + FX_BIAS); }
__device__ __forceinline__ FxD fx_const(int2 q) { return FxD{q.x, q.y}; }
// one sum of products: hi collects h h', lo collects h l' + l h'
struct FxSum {
  fx_t hi, lo;
};
__device__ __forceinline__ void fx_acc(FxSum &s, FxD a, FxD b) {
  s.lo = fx_mad(a.h, b.l, s.lo);
  s.lo = fx_mad(a.l, b.h, s.lo);
  s.hi = fx_mad(a.h, b.h, s.hi);
}
// the sum / 2^64 times 2^a (0 <= a < 32): lo starts at half a unit of that window, which rounds; with hi
// starting at the same number the value comes out with the bias that fx_biased takes
__device__ __forceinline__ FxSum fx_zero(int a) { return FxSum{0, (fx_t)(0x80000000u >> a)}; }
__device__ __forceinline__ FxSum fx_zero_biased(int a) { return FxSum{(fx_t)(0x80000000u >> a), (fx_t)(0x80000000u >> a)}; }
__device__ __forceinline__ fx_t fx_value(const FxSum &s, int a) { return (s.hi << a) + (s.lo >> (32 - a)); }
__device__ __forceinline__ FxD fx_mul(FxD a, FxD b) {
  FxSum s = fx_zero_biased(0);
  fx_acc(s, a, b);
  return fx_biased(fx_value(s, 0));
}
__device__ __forceinline__ fx_t fx_shr(fx_t x, int k) {  // x / 2^k rounded, 0 <= k <= 62
  return (x + ((1ll << k) >> 1)) >> k;
}

// |x| 2^(...) truncated, with x's sign: the leading significand bit of a double with biased exponent E
// lands on bit 62 - drop (E >= the exponent of x)
__device__ __forceinline__ fx_t fx_from(double x, int E, int drop) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long M = (((unsigned long long)mh << 32) | lo) << 10;
  const int s = min(E - ex + drop, 63);
  const fx_t X = (fx_t)(M >> s);
  return hi < 0 ? -X : X;
}
// biased exponent that bounds a magnitude whose high word is at most `hi` (with 2^-16 to spare, so that a
// sum of two values at the bound still splits into signed halves)
__device__ __forceinline__ int fx_exponent(int hi) { return (hi + 0x10) >> 20; }
__device__ __forceinline__ int fx_hi_abs(double x) { return __double2hiint(x) & 0x7fffffff; }

// Metric terms: each direction d has its own scale 2^-e_d, e_d the exponent of its largest |Ja^d_c| in the element (jmax).
// All products of a direction's lines carry Ja^d once, so the windows below are those of metric terms below 2, and a
// direction's sums come out in units of 2^e_d. Even so the wide directions' sums are rounded in windows made for the thin
// one's pressure and velocity: the error of the right-hand side against that of FP64 (rms per variable, shear layers across
// the thin direction, N = 3, 5, 7) is 0.59 to 0.68 on cubes, 0.64 to 0.85 at aspect ratio 8, 0.64 to 1.13 at 16 and up to 4
// at 64 (one scale for all directions: 1.4 at 16, 4 at 64, 37 at 1024). Elements whose metric terms span more than FX_JSPAN
// take the general path.
constexpr int FX_JSPAN = 3;         // largest span of max_c |Ja^d_c| over the element's nodes and directions, log2
constexpr int FX_FAR = 1 << 28;     // jmax.w of an element beyond it
constexpr int FX_NEAR = 2;          // directions' exponents this close: sums added as integers
__device__ __forceinline__ int fx_unit(int h) {  // e_d
  return max(-340, min(340, fx_exponent(h) - 1023));
}

// |f| of direction d against 2^e_d, as a high word (unit: e_d 2^20); what is not finite, or beyond 2^477, counts as such
__device__ __forceinline__ int fx_relative(double f, int unit) {
  const int h = fx_hi_abs(f);
  return h < (1500 << 20) ? h - unit : 0x7ff00000;
}

// per-element scales, from the maxima (high words) of the staged quantities, the metric terms and the
// viscous flux
struct FxScale {
  int ok;
  int er, eu, ep, ex;      // exponents E of rho, velocity, p, h (or e)
  int e[3];                // e_d; Ja^d is taken with the exponent 1023 + e_d
  int top;                 // largest e_d, or -1000 where they differ by more than FX_NEAR
  int dp, dx;              // extra bits dropped from p and h (e)
  int av, ag;              // windows of V and G
  int kg, kv;              // right shifts of G before the momentum product, of V before p V (KG)
  int vm, ve;              // fx_from exponents of the viscous flux (momentum, energy), e_d to be added
  int k0, km, ke;          // results are fixed value x 2^(k + e_d) x (1/w)
};
constexpr int FX_AM = 3;  // window of the momentum and energy products

// upper bound of log2 of a magnitude whose high word is at most hi, in 2^-20: log2 m <= (m - 1) + 0.0861
__device__ __forceinline__ int fx_lg(int hi) { return hi - (1023 << 20) + 0x16200; }
// largest row sum R of |Q|: 0.5, 1.34, 1.87, 2.44, 2.79, 3.15, 3.41 (N = 1..7): its log2 in 2^-20, and ceil(log2 R)
constexpr int FX_LGR = N == 1 ? -1048576 : N == 2 ? 443000 : N == 3 ? 947000 : N == 4 ? 1350000 : N == 5 ? 1552000
                     : N == 6 ? 1736000 : 1856000;
constexpr int FX_RB = N == 1 ? 0 : N <= 3 ? 1 : 2;

// Bounds (value x scale, log2): S_rho < 63, S_u, S_Ja, S_h < 61, S_p < 63; T = Q S_rho < 62; V = u.Ja <=
// max|u| max_d sum_c |Ja^d_c| fills 62.9, G = T V fills 62.3; momentum and energy operands are shifted
// right until a line's sum of advective terms stays below 61.7; the viscous share adds at most 59.8. The
// halved sum of three directions then stays below 62.9, and the cross sums h l' + l h' of every product
// group below 63.
template <int VF>
__device__ __forceinline__ FxScale fx_scales(const int *mx, int4 mj, int mvm, int mve, bool ns) {
  // mx: high words: rho max, rho min, |u| max, p max, p min, x max, x min (minima signed); mj: jmax; mvm, mve: fvmax
  FxScale s;
  const int j0 = fx_exponent(mj.x), j1 = fx_exponent(mj.y), j2 = fx_exponent(mj.z);
  s.e[0] = fx_unit(mj.x); s.e[1] = fx_unit(mj.y); s.e[2] = fx_unit(mj.z);
  const int jt = max(s.e[0], max(s.e[1], s.e[2])), jb = min(s.e[0], min(s.e[1], s.e[2]));
  s.top = jt - jb <= FX_NEAR ? jt : -1000;
  s.er = fx_exponent(mx[0]); s.ep = fx_exponent(mx[3]); s.ex = fx_exponent(mx[5]);
  constexpr int ej = 1023;
  s.eu = max(fx_exponent(mx[2]), (1996 - s.er + s.ep) >> 1);  // floor 2^-26 sqrt(p / rho): kg stays within 62
  const int lo = min(min(s.er, s.ep), min(min(s.ex, s.eu), min(j0, min(j1, j2))));
  const int hi = max(max(s.er, s.ep), max(max(s.ex, s.eu), max(j0, max(j1, j2))));
  const int lr = fx_lg(mx[0]), lu = max(fx_lg(mx[2]), (s.eu - 1023) << 20), lp = fx_lg(mx[3]), lx = fx_lg(mx[5]), lj = mj.w;
  const int lv = lu + lj;                                      // log2 of the V bound
  constexpr int L = 1 << 20, LIM = (int)(61.7 * L);
  // scales: fixed = value 2^s
  const int st = 1084 - s.er, sv0 = 2102 - s.eu - ej;
  s.av = min((((int)(62.9 * L) - lv) >> 20) - sv0, 6);
  const int sv = sv0 + s.av;
  s.ag = min((((int)(62.3 * L) - lr - lv) >> 20) - (st + sv - 64), 4);
  const int sg = st + sv - 64 + s.ag;
  const int xa = sg + 1022 - s.eu, xp = 2106 - s.ep - ej;    // momentum from G u, from p Ja
  int xm = min(min(xa, xp), (LIM - (FX_LGR + L + max(lr + lv + lu, lp + lj))) >> 20);
  const int evm = fx_exponent(mvm), eve = fx_exponent(mve);
  if (ns) xm = min(xm, 1081 - evm);
  s.kg = xa - xm;
  s.dp = xp - xm;
  const int xe0 = sg + 1022 - s.ex;                            // energy from G h (G e)
  int be = lr + lv + lx, xe = xe0, xq = 0;
  if (VF == VF_KG) {  // and from (Q S_p) V
    xq = 3123 - s.dp - s.ep - s.eu - ej + s.av;
    xe = min(xe, xq);
    be = max(be, lp + lv) + L;
  }
  xe = min(xe, (LIM - (FX_LGR + be)) >> 20);
  if (ns) xe = min(xe, 1081 - eve);
  s.dx = xe0 - xe;
  s.kv = VF == VF_KG ? 2 + xq - xe : 0;
  s.vm = 1084 - xm;  // (the rows c_QV carry one bit less than Q)
  s.ve = 1084 - xe;
  s.k0 = 2 - (sg - FX_RB); s.km = 2 - xm; s.ke = 2 - xe;  // 2 D F, and the halved sum of directions
  const int kmax = max(max(abs(s.k0), abs(s.km)), abs(s.ke));
  s.ok = mx[1] > 0 && mx[4] > 0 && mx[6] > 0 && s.er - (mx[1] >> 20) <= 8 && s.ep - (mx[4] >> 20) <= 8 &&
         s.ex - (mx[6] >> 20) <= 8 && lo >= 700 && hi <= 1350 && kmax <= 560 && mj.w < FX_FAR && s.av >= 0 && s.ag >= 0 &&
         s.kg >= 0 && s.kg <= 62 && s.dp >= 0 && s.dx >= 0 && s.kv <= 62 && (!ns || (evm < 1500 && eve < 1500));
  return s;
}

// staging index of node (i, j, k): strides chosen so that the lanes of a half warp (two lines' nodes along any
// direction) meet few bank conflicts (n = 8: strides 10 and 82, 2 mod 4: none along eta and zeta)
constexpr int FX_SJ = n == 8 ? 10 : n + 1, FX_SK = n == 8 ? 82 : n * (n + 1) + 1;
constexpr int FX_PS = N * (1 + FX_SJ + FX_SK) + 1;
__device__ __forceinline__ int fx_idx(int node) { return node % n + FX_SJ * ((node / n) % n) + FX_SK * (node / nn); }

// element slots (fx_t, FX_PS each): 0-5 rho, u, v, w, p, h|e; 6 + 3 dir + c metric terms; after a line thread
// has finished node i, its direction's sums (5) replace the three metric slots of (dir, i) and slots
// 15 + 2 dir, 16 + 2 dir
constexpr int FX_SLOTS = 21;
__device__ __forceinline__ int fx_slot(int dir, int v) { return v < 3 ? 6 + 3 * dir + v : 12 + 2 * dir + v; }

struct FxNode {
  fx_t r, u, v, w, p, x, jx, jy, jz;
};
__device__ __forceinline__ FxNode fx_load(const fx_t *__restrict__ S, int a, int dir) {
  const fx_t *J = S + (6 + 3 * dir) * FX_PS + a;
  return FxNode{S[a], S[FX_PS + a], S[2 * FX_PS + a], S[3 * FX_PS + a], S[4 * FX_PS + a], S[5 * FX_PS + a], J[0], J[FX_PS], J[2 * FX_PS]};
}

// the five fluxes of one pair, weighted with Q_im (see fx_scales for the scales); the staged values carry half
// the bias each, so a pair sum splits without an add
template <int VF>
__device__ __forceinline__ void fx_pair(const FxNode &a, const FxNode &b, FxD q, int av, int ag, int kg, int kv,
                                        fx_t F[5]) {
  const FxD Sjx = fx_biased(a.jx + b.jx), Sjy = fx_biased(a.jy + b.jy), Sjz = fx_biased(a.jz + b.jz);
  const FxD Su = fx_biased(a.u + b.u), Sv = fx_biased(a.v + b.v), Sw = fx_biased(a.w + b.w);
  FxSum s = fx_zero_biased(av);
  fx_acc(s, Su, Sjx);
  fx_acc(s, Sv, Sjy);
  fx_acc(s, Sw, Sjz);
  const fx_t Vb = fx_value(s, av);
  s = fx_zero_biased(ag);
  fx_acc(s, fx_mul(q, fx_biased(a.r + b.r)), fx_biased(Vb));
  const fx_t Gb = fx_value(s, ag), G = Gb - FX_BIAS;
  const FxD P = fx_mul(q, fx_biased(a.p + b.p));
  F[0] = (Gb + (((1 << FX_RB) >> 1) - FX_BIAS)) >> FX_RB;
  const FxD Gm = fx_split(fx_shr(G, kg));
  s = fx_zero(FX_AM);
  fx_acc(s, Gm, Su); fx_acc(s, P, Sjx);
  F[1] = fx_value(s, FX_AM);
  s = fx_zero(FX_AM);
  fx_acc(s, Gm, Sv); fx_acc(s, P, Sjy);
  F[2] = fx_value(s, FX_AM);
  s = fx_zero(FX_AM);
  fx_acc(s, Gm, Sw); fx_acc(s, P, Sjz);
  F[3] = fx_value(s, FX_AM);
  s = fx_zero(FX_AM);
  fx_acc(s, fx_biased(Gb), fx_biased(a.x + b.x));
  if (VF == VF_KG) fx_acc(s, P, fx_split(fx_shr(Vb - FX_BIAS, kv)));
  F[4] = fx_value(s, FX_AM);
}

// Lanes of the pair phase: a warp takes FX_LPW lines of one direction, one lane per node, a line's nodes in
// neighbouring lanes
constexpr int FX_LPW = 32 / n;

// viscous divergence of the lane's node along its line: -sum_m Q_im Fv_m / 2 for the four quantities.
// n even: lane i < n/2 forms the sum with the even half of Q, lane N - i that with the odd half
// (n^2/2 products per line and quantity instead of n^2)
__device__ __forceinline__ void fx_viscous(const double *Fn, const int2 *__restrict__ sQ, int idx, int l0,
                                           int vm, int ve, fx_t acc[5]) {
  const int2 *row = sQ + idx * FX_QV;
  double f64[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) f64[q] = Fn[q * nnn];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const fx_t f = fx_from(f64[q], q < 3 ? vm : ve, 0);
    FxSum s = fx_zero(0);
    if constexpr (n % 2 == 0) {
      const bool low = idx < EO_H;
      const int opp = l0 + N - idx;
      const fx_t g = __shfl_sync(0xffffffffu, f, opp);
      const fx_t h = low ? f + g : g - f;  // the even sum, or the odd difference of the low node
#pragma unroll
      for (int m = 0; m < EO_H; ++m)
        fx_acc(s, fx_const(row[m]), fx_split(__shfl_sync(0xffffffffu, h, l0 + (low ? m : N - m))));
      const fx_t y = fx_value(s, 0), z = __shfl_sync(0xffffffffu, y, opp);
      acc[1 + q] = low ? -(y + z) : z - y;
    } else {
#pragma unroll
      for (int m = 0; m < n; ++m)  // (the diagonal of Q is zero)
        fx_acc(s, fx_const(row[m]), fx_split(__shfl_sync(0xffffffffu, f, l0 + m)));
      acc[1 + q] = -fx_value(s, 0);
    }
  }
}

// Elements per CTA: one; CTAs of one or two warps at the lowest degrees, so that small meshes spread over the SMs
constexpr int FX_EPB = N == 1 ? 8 : N == 2 ? 2 : 1;
constexpr int FX_THREADS = round32(FX_EPB * nnn);
// the line of the lane's node in group gr of the pair phase (lanes without a line of their own repeat the group's
// first one): direction, node on the line, lane of node 0, element of the block, node 0 and stride in the element's
// arrays (gb, gs) and in the staged ones (pb, ps)
constexpr int FX_GROUPS = (FX_EPB * nn + FX_LPW - 1) / FX_LPW;  // warps' worth of lines per direction
struct FxLine {
  bool own;
  int dir, idx, l0, lel, gb, gs, pb, ps;
};
__device__ __forceinline__ FxLine fx_line(int gr, int lane) {
  FxLine q;
  q.dir = gr / FX_GROUPS;
  const int g0 = (gr % FX_GROUPS) * FX_LPW, l = (lane / n) % FX_LPW;
  q.idx = lane % n;
  q.l0 = l * n;
  q.own = lane < FX_LPW * n && g0 + l < FX_EPB * nn;
  const int ln = q.own ? g0 + l : g0;
  q.lel = ln / nn;
  const int ll = ln % nn, la = ll % n, lb = ll / n;
  q.gb = q.dir == 0 ? n * (la + n * lb) : q.dir == 1 ? la + nn * lb : la + n * lb;
  q.gs = q.dir == 0 ? 1 : q.dir == 1 ? n : nn;
  q.ps = q.dir == 0 ? 1 : q.dir == 1 ? FX_SJ : FX_SK;
  q.pb = q.dir == 0 ? FX_SJ * la + FX_SK * lb : q.dir == 1 ? la + FX_SK * lb : la + FX_SJ * lb;
  return q;
}

// general path: the pair phase in FP64 on the staged doubles (slots as in the fixed-point phase, 4 p), each pair formed once
// and its flux handed to the partner by shuffles. Bound by the FP64 pipe. Right-hand side with every element general, N = 7,
// 12^3, Euler: 754 us, 1159 with a thread per node that formed all its pairs itself, 734 with the former FP64 line
// kernel (n / 2 of the n (n - 1) / 2 pairs of a line are formed twice here); N = 3, 21 x 18 x 15: 229, 330 and 224 us.
template <int VF>
__device__ __noinline__ void fx_general_lines(const DgDevice &d, double *S, int e0) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int gr = threadIdx.x >> 5; gr < 3 * FX_GROUPS; gr += FX_THREADS / 32) {
    const FxLine q = fx_line(gr, lane);
    double *Se = S + q.lel * FX_SLOTS * FX_PS, *Pi = Se + q.pb + q.idx * q.ps;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (d.equations == 1) {
      const double *Fn = d.Fv + ((size_t)min(e0 + q.lel, d.nE - 1) * 12 + q.dir * 4) * nnn + q.gb + q.idx * q.gs;
      double f[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) f[v] = 8.0 * Fn[v * nnn];
#pragma unroll 1
      for (int m = 0; m < n; ++m) {
        const double c = c_De[q.idx * n + m];
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[1 + v] -= c * __shfl_sync(0xffffffffu, f[v], q.l0 + m);
      }
    }
#pragma unroll 1
    for (int s = n / 2; s > 0; --s) {  // the smaller factors first
      const int m = q.idx + s < n ? q.idx + s : q.idx + s - n, j = q.idx >= s ? q.idx - s : q.idx - s + n;
      const double *Pm = Se + q.pb + m * q.ps, *Ji = Pi + (6 + 3 * q.dir) * FX_PS, *Jm = Pm + (6 + 3 * q.dir) * FX_PS;
      const double Sj[3] = {Ji[0] + Jm[0], Ji[FX_PS] + Jm[FX_PS], Ji[2 * FX_PS] + Jm[2 * FX_PS]};
      const double Su[3] = {Pi[FX_PS] + Pm[FX_PS], Pi[2 * FX_PS] + Pm[2 * FX_PS], Pi[3 * FX_PS] + Pm[3 * FX_PS]};
      const double Vp = Su[0] * Sj[0] + Su[1] * Sj[1] + Su[2] * Sj[2], Sp = Pi[4 * FX_PS] + Pm[4 * FX_PS];
      double F[5];
      F[0] = (Pi[0] + Pm[0]) * Vp;
#pragma unroll
      for (int k = 0; k < 3; ++k) F[1 + k] = F[0] * Su[k] + Sp * Sj[k];
      F[4] = F[0] * (Pi[5 * FX_PS] + Pm[5 * FX_PS]);
      if (VF == VF_KG) F[4] += 0.5 * Sp * Vp;
      const double ci = c_De[q.idx * n + m], cj = c_De[q.idx * n + j];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        acc[v] += ci * F[v];
        if (2 * s != n) acc[v] += cj * __shfl_sync(0xffffffffu, F[v], q.l0 + j);
      }
    }
    acc[0] *= 2.0;  // (the mass flux's factor is D / 4)
    __syncwarp();
    if (q.own) {
#pragma unroll
      for (int v = 0; v < 5; ++v) Pi[fx_slot(q.dir, v) * FX_PS] = acc[v];
    }
  }
}

// FV subcell operator of the blend (Sec. 4.1), in FP64 (see line_fv for the operator). It is bound by the FP64 pipe
// (~280 instructions per interface with LLF); one thread per interface keeps a troubled element's critical path at
// three solves per thread, where a thread per line ran N of them in a row on half the threads. Right-hand side's
// volume part per launch, N = 5, 24^3, LLF, blend on every element: 4.74 (FP64 line kernel) -> 3.51 ms; N = 3, 32^3:
// 2.57 -> 2.40 ms; without troubled elements (blast, N = 5, 32^3): 3.91 -> 1.35 ms.
// Staged slots of an
// element under the blend, after the pair phase: 0-4 rho, u, v, w, p; from slot 6 on the interface fluxes
// [3 dir][N interfaces][5][nn lines].
__constant__ double c_Ct[N * n];  // interface metric i + 1/2 = sum_m c_Ct[i][m] Ja_m = Ja_0 + sum_{k <= i} w_k (D Ja)_k

// minmod of two slopes; signs and magnitudes compared as integers, which keeps it off the FP64 pipe
__device__ __forceinline__ double fv_minmod(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b), m = 0x7fffffffffffffffll;
  return (x ^ y) < 0 || (x & m) == 0 || (y & m) == 0 ? 0.0 : ((x & m) < (y & m) ? a : b);
}

// a Riemann side from (rho, u, v, w, p)
__device__ __forceinline__ void fv_side(const double q[5], double igm1, RSide<double> &s) {
  s.rs = rsq(q[0]);
  s.ir = s.rs * s.rs;
  s.U[0] = q[0];
#pragma unroll
  for (int c = 0; c < 3; ++c) { s.u[c] = q[1 + c]; s.U[1 + c] = q[0] * q[1 + c]; }
  s.pm = s.p = q[4];
  s.U[4] = q[4] * igm1 + 0.5 * (s.U[1] * q[1] + s.U[2] * q[2] + s.U[3] * q[3]);
}

// flux through interface i + 1/2 of one line, into out [5][nn]: the states of subcells i and i + 1 there (minmod
// slopes inside, first order in the outer subcells and where a reconstruction loses positivity), each slope's
// difference formed once
__device__ __noinline__ void fv_interface(const DgDevice &d, const double *__restrict__ P, int pb, int ps,
                                          const double *__restrict__ Jd, int gs, int i, double *__restrict__ out) {
  double qL[5], qR[5], a[3], F[5];
  {
    const int p0 = pb + i * ps, bk = i > 0 ? -ps : 0, fw = i + 1 < N ? 2 * ps : ps;
    const double hb = c_ihx[i], hc = c_ihx[i + 1], hf = i + 1 < N ? c_ihx[i + 2] : 0.0;
    const double xL = c_xi[i], xR = c_xi[i + 1], lm = c_xh[i] - xL, lp = c_xh[i + 1] - xL, rm = c_xh[i + 1] - xR,
                 rp = c_xh[i + 2] - xR;
    double l0[5], r0[5];
    bool okL = true, okR = true;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double *Pv = P + v * FX_PS + p0;
      const double q0 = Pv[0], q1 = Pv[ps], dc = (q1 - q0) * hc;
      const double sL = fv_minmod((q0 - Pv[bk]) * hb, dc), sR = fv_minmod(dc, (Pv[fw] - q1) * hf);
      l0[v] = q0;
      r0[v] = q1;
      qL[v] = q0 + sL * lp;
      qR[v] = q1 + sR * rm;
      if (v == 0 || v == 4) {
        okL = okL && qL[v] > 0.0 && q0 + sL * lm > 0.0;
        okR = okR && qR[v] > 0.0 && q1 + sR * rp > 0.0;
      }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if (!okL) qL[v] = l0[v];
      if (!okR) qR[v] = r0[v];
    }
  }
  RSide<double> L, R;
  fv_side(qL, d.igm1, L);
  fv_side(qR, d.igm1, R);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a[c] = 0.0;
#pragma unroll
    for (int m = 0; m < n; ++m) a[c] += c_Ct[i * n + m] * __ldg(Jd + c * nnn + m * gs);
  }
  const double a2 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2], is = rsq(a2), s = a2 * is;
  const double nv[3] = {a[0] * is, a[1] * is, a[2] * is};
  riemann_sides<double>(d.sflux, L, R, nv, d.gamma, 0.0, 0.0, F);
#pragma unroll
  for (int v = 0; v < 5; ++v) out[v * nn] = s * F[v];
}

// One thread per node. What bounds it: instruction issue (55 % of the slots) with the FP64 pipe at 36 %, FMA-heavy
// (IMAD.WIDE) at 44 %, ALU at 52 % and DRAM at 15 %; 64 registers and 21 slots of shared memory keep two CTAs
// (32 warps) per SM at N = 7. A thread per line (half the pair evaluations' overhead, sums in 80 registers,
// 168 in all) held 12 warps and measured 2.43 ms per launch at N = 7, 24^3, Navier-Stokes, Pirozzoli; this form
// 1.74 ms, the FP64 line kernel before it 6.21 ms (N = 5, 24 x 12 x 12 channel: 0.197 against 0.586 ms).
constexpr size_t FX_SMEM = sizeof(fx_t) * FX_EPB * FX_SLOTS * FX_PS;
constexpr int FX_MINB = 1024 / FX_THREADS < 32 ? 1024 / FX_THREADS : 32;  // 64 registers per thread

template <int VF, bool SC>
__global__ void __launch_bounds__(FX_THREADS, FX_MINB)
    k_volume_fx(const DgDevice d, const double *U, double *out, double *__restrict__ g, int mode, int first, double dt,
                double A, double B) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  fx_t *S = reinterpret_cast<fx_t *>(sm_raw);  // [EPB][FX_SLOTS][FX_PS]
  __shared__ int s_mx[FX_EPB][8];
  __shared__ FxScale s_sc[FX_EPB];
  __shared__ int2 s_rho[FX_H * FX_H], s_Q[nn], s_QV[n * FX_QV];
  const int e0 = blockIdx.x * FX_EPB, tid = threadIdx.x;
  const bool ns = d.equations == 1;
  const double gm1 = d.gm1;
  for (int t = tid; t < FX_EPB * 8; t += FX_THREADS) {
    const int k = t & 7;
    s_mx[t >> 3][k] = (k == 1 || k == 4 || k == 6) ? 0x7fffffff : 0;
  }
  for (int t = tid; t < FX_H * FX_H; t += FX_THREADS) s_rho[t] = c_rho[t];
  for (int t = tid; t < nn; t += FX_THREADS) s_Q[t] = c_Qx[t];
  for (int t = tid; t < n * FX_QV; t += FX_THREADS) s_QV[t] = c_QV[t];
  wait_for_previous();
  __syncthreads();
  // phase A: primitive quantities of the thread's node and the element maxima
  const int le = tid / nnn, node = tid % nnn, e = e0 + le;
  const bool on = tid < FX_EPB * nnn && e < d.nE;
  double q[6], J[9];
  {
    int m0 = 0, n0 = 0x7fffffff, mu_ = 0, m3 = 0, n3 = 0x7fffffff, m5 = 0, n5 = 0x7fffffff;
    if (on) {
      double Uv[5];
      load_state<double>(d, U, e, node, Uv);
      const double *Je = d.Ja + (size_t)e * 9 * nnn + node;
#pragma unroll
      for (int k = 0; k < 9; ++k) J[k] = __ldg(Je + k * nnn);
      const double r = Uv[0], ir = rcp_int(r);
      const double u = Uv[1] * ir, v = Uv[2] * ir, w = Uv[3] * ir;
      const double p = gm1 * (Uv[4] - 0.5 * (Uv[1] * u + Uv[2] * v + Uv[3] * w));
      const double x = VF == VF_PIR ? (Uv[4] + p) * ir : Uv[4] * ir;
      q[0] = r; q[1] = u; q[2] = v; q[3] = w; q[4] = p; q[5] = x;
      if (!(r > 0.0) || !(p > 0.0) || !isfinite(Uv[4])) flag_set(d.flag, 1);
      // minima keep the sign (a negative high word fails the scale test), maxima are of magnitudes
      m0 = fx_hi_abs(r); n0 = __double2hiint(r);
      mu_ = max(max(fx_hi_abs(u), fx_hi_abs(v)), fx_hi_abs(w));
      m3 = fx_hi_abs(p); n3 = __double2hiint(p);
      m5 = fx_hi_abs(x); n5 = __double2hiint(x);
    }
    bool each = on;  // whether this lane adds its own maxima
    if (FX_EPB == 1) {
      m0 = __reduce_max_sync(0xffffffffu, m0); n0 = __reduce_min_sync(0xffffffffu, n0);
      mu_ = __reduce_max_sync(0xffffffffu, mu_);
      m3 = __reduce_max_sync(0xffffffffu, m3); n3 = __reduce_min_sync(0xffffffffu, n3);
      m5 = __reduce_max_sync(0xffffffffu, m5); n5 = __reduce_min_sync(0xffffffffu, n5);
      each = (tid & 31) == 0 && on;
    }
    if (each) {
      atomicMax(&s_mx[le][0], m0); atomicMin(&s_mx[le][1], n0); atomicMax(&s_mx[le][2], mu_);
      atomicMax(&s_mx[le][3], m3); atomicMin(&s_mx[le][4], n3);
      atomicMax(&s_mx[le][5], m5); atomicMin(&s_mx[le][6], n5);
    }
  }
  __syncthreads();
  int good = 1;
  if (tid < FX_EPB && e0 + tid < d.nE) {
    const int et = e0 + tid;
    s_sc[tid] = fx_scales<VF>(s_mx[tid], d.jmax[et], ns ? d.fvmax[2 * et] : 0, ns ? d.fvmax[2 * et + 1] : 0, ns);
    good = s_sc[tid].ok;
  }
  const bool ok = __syncthreads_and(good);
  if (ok) {
    if (on) {
      const FxScale &c = s_sc[le];
      fx_t *Se = S + le * FX_SLOTS * FX_PS + fx_idx(node);
      constexpr fx_t HB = FX_BIAS / 2;
      Se[0] = fx_from(q[0], c.er, 1) + HB;
      Se[FX_PS] = fx_from(q[1], c.eu, 3) + HB;
      Se[2 * FX_PS] = fx_from(q[2], c.eu, 3) + HB;
      Se[3 * FX_PS] = fx_from(q[3], c.eu, 3) + HB;
      Se[4 * FX_PS] = fx_from(q[4], c.ep, 1 + c.dp) + HB;
      Se[5 * FX_PS] = fx_from(q[5], c.ex, 3 + c.dx) + HB;
#pragma unroll
      for (int k = 0; k < 9; ++k) Se[(6 + k) * FX_PS] = fx_from(J[k], 1023 + c.e[k / 3], 3) + HB;
    }
    __syncthreads();
    // phase B: one lane per node of a line. Lane i forms the pairs (i, i + s mod n), s <= (n - 1) / 2, adds its
    // share and hands the partner's on by a shuffle; at s = n / 2 (n even) both nodes form the pair.
    const int lane = tid & 31;
    for (int gr = tid >> 5; gr < 3 * FX_GROUPS; gr += FX_THREADS / 32) {
      const int dir = gr / FX_GROUPS, g0 = (gr % FX_GROUPS) * FX_LPW;
      const int idx = lane % n, l = (lane / n) % FX_LPW, l0 = l * n;
      // lanes without a line of their own repeat the group's first one
      const bool own = lane < FX_LPW * n && g0 + l < FX_EPB * nn;
      const int ln = own ? g0 + l : g0;
      const int lel = ln / nn, ll = ln % nn;
      const int la = ll % n, lb = ll / n;
      const int gb = dir == 0 ? n * (la + n * lb) : dir == 1 ? la + nn * lb : la + n * lb;
      const int gs = dir == 0 ? 1 : dir == 1 ? n : nn, ps = dir == 0 ? 1 : dir == 1 ? FX_SJ : FX_SK;
      const int pb = dir == 0 ? FX_SJ * la + FX_SK * lb : dir == 1 ? la + FX_SK * lb : la + FX_SJ * lb;
      const FxScale &c = s_sc[lel];
      fx_t *Se = S + lel * FX_SLOTS * FX_PS;
      const int ai = pb + idx * ps;
      fx_t acc[5] = {0, 0, 0, 0, 0};
      if (ns) {
        const size_t el = min(e0 + lel, d.nE - 1);
        fx_viscous(d.Fv + (el * 12 + dir * 4) * nnn + gb + idx * gs, s_QV, idx, l0, c.vm + c.e[dir], c.ve + c.e[dir], acc);
      }
      const int av = c.av, ag = c.ag, kg = c.kg, kv = c.kv;
      const FxNode ni = fx_load(Se, ai, dir);
#pragma unroll 1
      for (int s = 1; s <= n / 2; ++s) {
        const int m = idx + s < n ? idx + s : idx + s - n;
        const FxNode nm = fx_load(Se, pb + m * ps, dir);
        fx_t F[5];
        fx_pair<VF>(ni, nm, fx_const(s_Q[idx * n + m]), av, ag, kg, kv, F);
        const bool both = 2 * s == n;
        const int src = l0 + (idx >= s ? idx - s : idx - s + n);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          acc[v] += F[v];
          if (!both) acc[v] -= __shfl_sync(0xffffffffu, F[v], src);
        }
      }
      __syncwarp();
      if (own) {
#pragma unroll
        for (int v = 0; v < 5; ++v) Se[fx_slot(dir, v) * FX_PS + ai] = acc[v];
      }
    }
  } else if (on) {
    double *Se = reinterpret_cast<double *>(S) + le * FX_SLOTS * FX_PS + fx_idx(node);
#pragma unroll
    for (int k = 0; k < 6; ++k) Se[k * FX_PS] = k == 4 ? 4.0 * q[k] : q[k];
#pragma unroll
    for (int k = 0; k < 9; ++k) Se[(6 + k) * FX_PS] = J[k];
  }
  if (!ok) {
    __syncthreads();
    fx_general_lines<VF>(d, reinterpret_cast<double *>(S), e0);
  }
  __syncthreads();
  let_next_start();
  // phase C: per node -- directions summed, surface terms, neighbour's viscous flux, blend, Jacobian, output / LSERK
  const int ijk[3] = {node % n, (node / n) % n, node / nn};
  double s[5];
  if (on) {
    if (ok) {
      const fx_t *Se = S + le * FX_SLOTS * FX_PS + fx_idx(node);
      const int a0 = min(ijk[0], N - ijk[0]), a1 = min(ijk[1], N - ijk[1]), a2 = min(ijk[2], N - ijk[2]);
      const int am = min(a0, min(a1, a2));  // the direction with the smallest weight
      const FxD r0 = fx_const(s_rho[a0 * FX_H + am]), r1 = fx_const(s_rho[a1 * FX_H + am]),
                r2 = fx_const(s_rho[a2 * FX_H + am]);
      const double iw = c_invw[am];
      const int iwh = __double2hiint(iw), iwl = __double2loint(iw);
      const FxScale &c = s_sc[le];
      const int k0 = c.k0, km = c.km, ke = c.ke, e0 = c.e[0], e1 = c.e[1], e2 = c.e[2], top = c.top;
      if (top != -1000) {
        auto scaled = [](FxD r, int h) { return fx_split((((fx_t)r.h << 32) + r.l) >> h); };
        const FxD q0 = scaled(r0, top - e0), q1 = scaled(r1, top - e1), q2 = scaled(r2, top - e2);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          FxSum f0{0, 0x40000000ll}, f1 = f0, f2 = f0;  // the three lo sums do not fit one
          fx_acc(f0, q0, fx_split(Se[fx_slot(0, v) * FX_PS]));
          fx_acc(f1, q1, fx_split(Se[fx_slot(1, v) * FX_PS]));
          fx_acc(f2, q2, fx_split(Se[fx_slot(2, v) * FX_PS]));
          // half the sum of the three directions (the factors carry 2^62)
          const fx_t sum = ((f0.hi + f1.hi + f2.hi) << 1) + (f0.lo >> 31) + (f1.lo >> 31) + (f2.lo >> 31);
          s[v] = (double)sum * __hiloint2double(iwh + (int)((unsigned)((v == 0 ? k0 : v < 4 ? km : ke) + top) << 20), iwl);
        }
      } else {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const int k = v == 0 ? k0 : v < 4 ? km : ke;
          auto part = [&](FxD r, int dir, int e) {
            FxSum f{0, 0x40000000ll};
            fx_acc(f, r, fx_split(Se[fx_slot(dir, v) * FX_PS]));
            return (double)((f.hi << 1) + (f.lo >> 31)) * __hiloint2double(iwh + (int)((unsigned)(k + e) << 20), iwl);
          };
          s[v] = part(r0, 0, e0) + part(r1, 1, e1) + part(r2, 2, e2);
        }
      }
    } else {
      const double *Se = reinterpret_cast<const double *>(S) + le * FX_SLOTS * FX_PS + fx_idx(node);
#pragma unroll
      for (int v = 0; v < 5; ++v) s[v] = Se[fx_slot(0, v) * FX_PS] + Se[fx_slot(1, v) * FX_PS] + Se[fx_slot(2, v) * FX_PS];
    }
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const int id = ijk[dd];
      if (id != 0 && id != N) continue;
      const int f = 2 * dd + (id == N ? 1 : 0);
      const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
      const double *fs = d.Fsurf + ((size_t)e * 6 + f) * 5 * nn + pp + n * qq;
#pragma unroll
      for (int v = 0; v < 5; ++v) s[v] += c_invw[0] * fs[v * nn];
    }
  }
  if constexpr (SC) {  // blend with the FV subcell operator where alpha > 0
    const double al = on ? d.alpha[e] : 0.0;
    if (__syncthreads_or(al > 0.0)) {
      double *P0 = reinterpret_cast<double *>(S);
      if (al > 0.0) {
        double Uv[5];
        load_state<double>(d, U, e, node, Uv);
        const double ir = rcp_int(Uv[0]);
        const double u = Uv[1] * ir, v = Uv[2] * ir, w = Uv[3] * ir;
        double *P = P0 + le * FX_SLOTS * FX_PS + fx_idx(node);
        P[0] = Uv[0]; P[FX_PS] = u; P[2 * FX_PS] = v; P[3 * FX_PS] = w;
        P[4 * FX_PS] = gm1 * (Uv[4] - 0.5 * (Uv[1] * u + Uv[2] * v + Uv[3] * w));
      }
      __syncthreads();
      // one thread per interface of a line
      for (int t = tid; t < FX_EPB * 3 * N * nn; t += FX_THREADS) {
        const int lt = t / (3 * N * nn), r = t % (3 * N * nn), dir = r / (N * nn), i = (r / nn) % N, line = r % nn;
        const int et = e0 + lt;
        if (et >= d.nE || !(d.alpha[et] > 0.0)) continue;
        const int la = line % n, lb = line / n;
        const int ps = dir == 0 ? 1 : dir == 1 ? FX_SJ : FX_SK, gs = dir == 0 ? 1 : dir == 1 ? n : nn;
        const int pb = dir == 0 ? FX_SJ * la + FX_SK * lb : dir == 1 ? la + FX_SK * lb : la + FX_SJ * lb;
        const int gb = dir == 0 ? n * (la + n * lb) : dir == 1 ? la + nn * lb : la + n * lb;
        double *P = P0 + lt * FX_SLOTS * FX_PS;
        fv_interface(d, P, pb, ps, d.Ja + ((size_t)et * 3 + dir) * 3 * nnn + gb, gs, i,
                     P + 6 * FX_PS + (dir * N + i) * 5 * nn + line);
      }
      __syncthreads();
      if (al > 0.0) {
        const double *Fi = P0 + le * FX_SLOTS * FX_PS + 6 * FX_PS;
        double fv[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) {
          const int id = ijk[dd];
          const int line = (dd == 0 ? ijk[1] : ijk[0]) + n * (dd == 2 ? ijk[1] : ijk[2]);  // = the faces' point
          const double *fl = id > 0 ? Fi + (dd * N + id - 1) * 5 * nn + line
                                    : d.Fsurf + ((size_t)e * 6 + 2 * dd) * 5 * nn + line;
          const double *fr = id < N ? Fi + (dd * N + id) * 5 * nn + line
                                    : d.Fsurf + ((size_t)e * 6 + 2 * dd + 1) * 5 * nn + line;
          const double iw = c_invw[min(id, N - id)];
#pragma unroll
          for (int v = 0; v < 5; ++v) fv[v] += iw * (id > 0 ? fr[v * nn] - fl[v * nn] : fr[v * nn] + fl[v * nn]);
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) s[v] = al * fv[v] + (1.0 - al) * s[v];
        if (ns)  // the line sums hold the viscous divergence too, which the blend must not weight
          for (int dd = 0; dd < 3; ++dd) {
            const int id = ijk[dd], st = dd == 0 ? 1 : dd == 1 ? n : nn;
            const double *Fv = d.Fv + ((size_t)e * 12 + dd * 4) * nnn + node - id * st;
            for (int m = 0; m < n; ++m)
              if (m != id)
#pragma unroll
                for (int v = 0; v < 4; ++v) s[1 + v] -= al * c_D[id * n + m] * Fv[v * nnn + m * st];
          }
      }
    }
  }
  if (!on) return;
  if (ns) {  // -(1/(2 w_b)) phi_nb, phi_nb = neighbour's outward normal viscous flux; or the wall's
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const int id = ijk[dd];
      if (id != 0 && id != N) continue;
      const int f = 2 * dd + (id == N ? 1 : 0);
      const int pp = dd == 0 ? ijk[1] : ijk[0], qq = dd == 2 ? ijk[1] : ijk[2];
      const int *ef = d.ef + ((size_t)e * 6 + f) * 4;
      const int nb = ef[0], fnb = ef[1], o = ef[2];
      if (nb < 0) {
        const double *fw = d.Fwall + (size_t)ef[3] * 4 * nn + pp + n * qq;
        const double hs = (id == N) ? 0.5 : -0.5;
        const double *Fve = d.Fv + ((size_t)e * 12 + dd * 4) * nnn + node;
#pragma unroll
        for (int v = 0; v < 4; ++v) s[1 + v] -= c_invw[0] * (fw[v * nn] - hs * Fve[v * nnn]);
      } else {
        int p2, q2;
        orient_map(o, pp, qq, p2, q2);
        const double sg = (fnb & 1) ? 0.5 * c_invw[0] : -0.5 * c_invw[0];
        const double *Fvn = d.Fv + ((size_t)nb * 12 + (fnb >> 1) * 4) * nnn + face_node(fnb, p2, q2);
#pragma unroll
        for (int v = 0; v < 4; ++v) s[1 + v] += sg * Fvn[v * nnn];
      }
    }
  }
  const double miJ = -d.invJ[(size_t)e * nnn + node];
  const size_t gi = (size_t)e * 5 * nnn + node;
  if (mode == 0) {
#pragma unroll
    for (int v = 0; v < 5; ++v) out[gi + v * nnn] = miJ * s[v];
  } else {
    const double fac = dt * miJ;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double du = fac * s[v];
      const double gv = first ? du : A * g[gi + v * nnn] + du;
      g[gi + v * nnn] = gv;
      out[gi + v * nnn] = U[gi + v * nnn] + B * gv;
    }
  }
}

// per element: jmax (see DgDevice) and the largest 1/J, for the fixed-point scales (1/J: zero where it spans more than 2^8
// in the element, which sends the lifting to its general path)
__global__ void __launch_bounds__(128) k_metric_max(const DgDevice d) {  // one warp per element
  const int e = blockIdx.x * 4 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (e >= d.nE) return;
  int h[3] = {0, 0, 0}, h1[3] = {0, 0, 0}, small = 0x7fffffff;
  double lo = 1e300, hi = 0.0;
  for (int t = lane; t < nnn; t += 32) {
    const double ij = d.invJ[(size_t)e * nnn + t];
    lo = fmin(lo, ij);
    hi = fmax(hi, ij);
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      const double *J = d.Ja + ((size_t)e * 3 + dd) * 3 * nnn + t;
      const double a = fabs(J[0]), b = fabs(J[nnn]), c = fabs(J[2 * nnn]);
      const int m = max(fx_hi_abs(a), max(fx_hi_abs(b), fx_hi_abs(c)));
      h[dd] = max(h[dd], m);
      small = min(small, m);
      h1[dd] = max(h1[dd], fx_hi_abs(a + b + c));
    }
  }
  small = __reduce_min_sync(0xffffffffu, small);
  int lg = 0, top = 0;
#pragma unroll
  for (int dd = 0; dd < 3; ++dd) {
    h[dd] = __reduce_max_sync(0xffffffffu, h[dd]);
    lg = max(lg, fx_lg(__reduce_max_sync(0xffffffffu, h1[dd])) - (fx_unit(h[dd]) << 20));
    top = max(top, fx_exponent(h[dd]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    d.jmax[e] = int4{h[0], h[1], h[2], top - fx_exponent(small) > FX_JSPAN ? FX_FAR : lg};
    d.ijmax[e] = hi <= 256.0 * lo ? hi : 0.0;
  }
}

int2 fx_halves(long double v, int bits) {  // v 2^bits rounded to nearest, balanced halves (host)
  const long long x = std::llrint(std::ldexp(v, bits));
  const int l = (int)(unsigned)(x & 0xffffffffll);
  return int2{(int)((x - l) >> 32), l};
}

// fixed-point tables from the extended-precision Q = W D and weights (host)
cudaError_t fx_upload(const DgTables &t) {
  int2 Q[nn], DT[nn], QV[n * FX_QV], rho[FX_H * FX_H];
  for (int i = 0; i < nn; ++i) Q[i] = fx_halves(t.Q[i], 63);
  for (int i = 0; i < nn; ++i) DT[i] = fx_halves(t.Q[i % n * n + i / n] / t.wl[i % n] / 32, 62);
  for (int i = 0; i < n; ++i)
    for (int m = 0; m < FX_QV; ++m) {
      long double v = t.Q[i * n + m];
      if (n % 2 == 0 && i < n / 2) v = (v + t.Q[i * n + N - m]) / 2;
      else if (n % 2 == 0) v = (t.Q[(N - i) * n + m] - t.Q[(N - i) * n + N - m]) / 2;
      QV[i * FX_QV + m] = fx_halves(v, 62);
    }
  for (int a = 0; a < FX_H; ++a)
    for (int b = 0; b < FX_H; ++b) rho[a * FX_H + b] = fx_halves(t.wl[a < b ? a : b] / t.wl[a], 62);
  double Ct[N * n];
  for (int m = 0; m < n; ++m) {
    long double acc = m == 0 ? 1.0L : 0.0L;
    for (int i = 0; i < N; ++i) {
      acc += t.Q[i * n + m] + (i == m && i == 0 ? -0.5L : 0.0L);  // (D_ii = 0 inside, w_0 D_00 = -1/2)
      Ct[i * n + m] = (double)acc;
    }
  }
  cudaError_t err = cudaMemcpyToSymbol(c_Qx, Q, sizeof(Q));
  err = err ? err : cudaMemcpyToSymbol(c_DT, DT, sizeof(DT));
  err = err ? err : cudaMemcpyToSymbol(c_Ct, Ct, sizeof(Ct));
  err = err ? err : cudaMemcpyToSymbol(c_QV, QV, sizeof(QV));
  return err ? err : cudaMemcpyToSymbol(c_rho, rho, sizeof(rho));
}

}  // namespace
