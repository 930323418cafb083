// dg_log.cuh -- natural logarithm of a positive normal double on the integer pipes, to an absolute error of
// 2^-58 + 2^-54 + 2.4e-17 |k| (ln m in fixed point, its conversion, the rounded ln 2 times the exponent k below) and half an
// ulp of the result, for sums in which it meets numbers of order one (the entropy of the integral
// diagnostics; CUDA's log is ~25 FP64 instructions, on a pipe of 2 lanes per clock and SM: two of them per node were
// most of k_invariants, N = 5, 24^3 644 -> 330 us).
//
// x = 2^k m, m in [1, 2). The leading seven bits of m's fraction select c, 1/m rounded to 32 bits at the middle of
// that interval, so that m c = 1 + r with |r| < 2^-8 exactly in 64-bit fixed point, and
//   ln x = k ln 2 - ln c + ln(1 + r),   ln(1 + r) = r - r^2/2 + r^3/3 - ... + r^7/7   (r^8/8 < 2^-67),
// by Horner's rule: the terms from r^4 on in 32 bits, the others in 64. The table holds c 2^32 and -ln c 2^62.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

struct LogEntry {
  unsigned c;
  unsigned lo, hi;  // -ln c 2^62
};
constexpr int LOG_TABLE = 128;

static inline void log_table(LogEntry *t) {  // (host)
  for (int i = 0; i < LOG_TABLE; ++i) {
    const long double mid = 1.0L + (i + 0.5L) / LOG_TABLE;
    t[i].c = (unsigned)std::llrint(std::ldexp(1.0L / mid, 32));
    const unsigned long long l = (unsigned long long)std::llrint(std::ldexp(-std::log(std::ldexp((long double)t[i].c, -32)), 62));
    t[i].lo = (unsigned)l;
    t[i].hi = (unsigned)(l >> 32);
  }
}

// high 64 bits of the product of two signed numbers below 2^62 (to a unit)
static __device__ __forceinline__ long long log_mulhi(long long a, long long b) {
  const int ah = (int)(a >> 32), bh = (int)(b >> 32);
  const unsigned al = (unsigned)a, bl = (unsigned)b;
  const long long lo = (((long long)ah * (long long)(bl >> 1)) >> 31) + (((long long)bh * (long long)(al >> 1)) >> 31);
  return (long long)ah * bh + lo;
}

static __device__ __forceinline__ double log_int(double x, const LogEntry *__restrict__ t) {
  const int h = __double2hiint(x);
  if ((unsigned)(h - 0x00100000) >= 0x7fe00000u) return log(x);
  const unsigned w = (unsigned)__double2loint(x);
  const unsigned mh = ((unsigned)h & 0xfffffu) << 11 | w >> 21 | 0x80000000u, ml = w << 11;  // m 2^63
  const LogEntry e = t[mh >> 24 & 0x7fu];
  const unsigned long long p = (unsigned long long)mh * e.c + (((unsigned long long)ml * e.c) >> 32);
  const long long z = (long long)(p - 0x8000000000000000ull) << 7;  // r 2^70
  const int zh = (int)(z >> 32);                                    // r 2^38
  int a = 357913941 - (__mulhi(zh, 306783378) >> 6);                // 2^31 (1/6 - r/7)
  a = 429496730 - (__mulhi(zh, a) >> 6);
  a = 536870912 - (__mulhi(zh, a) >> 6);
  long long s = 768614336404564651ll - (((long long)zh * a) >> 8);  // 2^61 (1/3 - r (1/4 - ...))
  s = (1ll << 60) - (log_mulhi(z, s) >> 6);
  s = (1ll << 61) - (log_mulhi(z, s) >> 6);
  const long long y = (log_mulhi(z, s) >> 5) + (long long)((unsigned long long)e.hi << 32 | e.lo);  // 2^62
  return fma((double)((h >> 20) - 1023), 0.69314718055994530942, (double)y * 0x1p-62);
}
