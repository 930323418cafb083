// dg_recip.cuh -- reciprocal and reciprocal square root of a double on the integer pipes.
//
// GB300 issues FP64 instructions at 2 lanes per clock and SM, so a division or a reciprocal square root (8 to 10 of
// them) takes ~5 clocks per lane and SM; these take ~45 integer instructions (~0.5 clocks). Roe face kernel at N = 7,
// 24^3: 812 -> 728 us per launch, LLF faces at N = 5, 32^3: 678 -> 563 us, EC volume kernel at N = 4, 23 x 19 x 17:
// 997 -> 864 us. Method: an FP32
// approximation y0 of the significand's (reciprocal) root, exact in 24 bits, then one step of the third-order
// iteration that truncates the binomial series of 1 / (1 - e) or (1 - e)^(-1/2) after e^2, in 64-bit fixed point:
//   1/m:        e = 1 - m y0,    y = y0 (1 + e + e^2)
//   1/sqrt(m):  e = 1 - m y0^2,  y = y0 (1 + e/2 + 3/8 e^2)
// |e| < 2^-20.5, so the truncated e^3 is below 2^-61; with the fixed point's rounding the relative error before the
// final rounding to 53 bits is below 2^-59, i.e. the result is within 0.51 ulp. Arguments that are not positive
// normal numbers, and results that would not be normal, take CUDA's own division and rsqrt.
#pragma once
#include <cuda_runtime.h>

// 2^63 y from y0 = Y / 2^32 and d = D / 2^63: y0 (1 + d), rounded to the 53-bit significand of a number in [1/2, 1]
static __device__ __forceinline__ double recip_pack(unsigned Y, long long D, int exponent) {
  const long long c = (long long)(int)(D >> 32) * (long long)Y + (long long)(((unsigned long long)(unsigned)D * Y) >> 32);
  const unsigned long long R = ((unsigned long long)Y << 31) + (unsigned long long)c;
  const unsigned long long q = (R + 512) >> 10;
  return __longlong_as_double((long long)(((unsigned long long)(unsigned)(exponent - 1) << 52) + q));
}

// y0 2^32 of a float that approximates a number in (1/2, 1]
static __device__ __forceinline__ unsigned recip_seed(float y) {
  const unsigned b = min(max(__float_as_uint(y), 0x3f000000u), 0x3f7fffffu);
  return (b << 8) | 0x80000000u;
}

static __device__ __forceinline__ double rcp_int(double x) {  // 1 / x
  const int h = __double2hiint(x);
  if ((unsigned)(h - 0x00100000) >= 0x7fb00000u) return 1.0 / x;  // exponents 1 to 2043
  const unsigned lo = (unsigned)__double2loint(x);
  const int ex = h >> 20;
  const unsigned mh = ((unsigned)h & 0xfffffu) << 11 | lo >> 21 | 0x80000000u, ml = lo << 11;  // m 2^63
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(0x3f800000u | (mh >> 8 & 0x7fffffu))));
  const unsigned Y = recip_seed(y);
  const unsigned long long p = (unsigned long long)mh * Y + (((unsigned long long)ml * Y) >> 32);  // m y0 2^63
  const long long E = (long long)(0x8000000000000000ull - p);
  const int eh = (int)(E >> 20);  // e 2^43
  return recip_pack(Y, E + (((long long)eh * eh) >> 23), 2045 - ex);
}

static __device__ __forceinline__ double rsq_int(double x) {  // 1 / sqrt(x)
  const int h = __double2hiint(x);
  if ((unsigned)(h - 0x00100000) >= 0x7fe00000u) return rsqrt(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int ex = (h >> 20) - 1023, odd = ex & 1;
  const unsigned sh = 10 + odd;  // m in [1, 4), m 2^62
  const unsigned mh = (((unsigned)h & 0xfffffu) | 0x100000u) << sh | lo >> (32 - sh), ml = lo << sh;
  float y;
  const unsigned mf = (((unsigned)h & 0xfffffu) << 3 | lo >> 29) + (odd ? 0x40000000u : 0x3f800000u);
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(mf)));
  const unsigned Y = recip_seed(y);
  const unsigned long long P = (unsigned long long)Y * Y;  // y0^2 2^64
  const unsigned ph = (unsigned)(P >> 32), pl = (unsigned)P;
  // m y0^2 2^62
  const unsigned long long c = ((unsigned long long)mh * pl >> 1) + ((unsigned long long)ml * ph >> 1);
  const unsigned long long t = (unsigned long long)mh * ph + (c >> 31);
  const long long E = (long long)(0x4000000000000000ull - t);
  const int eh = (int)(E >> 19);  // e 2^43
  // d 2^63 = e 2^62 + 3/8 e^2 2^63
  return recip_pack(Y, E + ((3 * (long long)eh * eh) >> 26), 1022 - ((ex - odd) >> 1));
}

static __device__ __forceinline__ double sqr_int(double x) {  // sqrt(x): x / sqrt(x), and one Heron step
  if ((unsigned)(__double2hiint(x) - 0x00100000) >= 0x7fe00000u) return sqrt(x);
  const double y = rsq_int(x), s = x * y;
  return fma(fma(-s, s, x), 0.5 * y, s);
}
