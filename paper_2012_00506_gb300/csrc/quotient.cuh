// quotient.cuh -- FP64 division for latency-bound chains.
#pragma once
#include "common.cuh"

namespace pdeshep {

// a / d rounded to nearest, in integers: the FP64 division is a chain of FP64 instructions of 64 clocks each
// (about 600 clocks for a warp, and its quadrant's pipe is taken meanwhile), the division of two 53-bit
// integers about 200 clocks of the integer pipes, and the reciprocal serves all entries of a column.
// The reciprocal of the divisor's significand comes from one Newton step on a 23-bit estimate (relative error e:
// e <= 2^-23 for the estimate plus 2^-24 for its argument, e^2 < 2^-44.8 after the step); the quotient to 54
// bits follows from it and one correction by the remainder, which is exact modulo 2^64 and below 2^62.3; a last
// comparison makes it the floor.  A quotient of two 53-bit numbers is never half-way between two of them, so its
// 54th bit rounds it.  Zero, subnormal, infinite and NaN operands and results outside the normal range go
// to the FP64 division (zero numerators, common in a band, give their zero at once).
struct Divisor {
  double d;
  unsigned long long md, r1;  // significand (53 bits); 2^62 / (md / 2^53)
  unsigned r0;                // 2^30 / (md / 2^53)
};
__device__ __forceinline__ Divisor divisor(double d) {
  Divisor v;
  v.d = d;
  v.md = ((unsigned long long)__double_as_longlong(d) & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned dh = (unsigned)(v.md >> 21), dl = (unsigned)(v.md << 11);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint2float_rn(dh)));
  v.r0 = min(__float2uint_rz(r * 4611686018427387904.0f), 0x7FFFFFFFu);
  // 1 - x r0 in units of 2^-52
  const unsigned long long p = (unsigned long long)dh * v.r0 + (((unsigned long long)dl * v.r0) >> 32);
  const int e = (int)((long long)((1ull << 62) - p) >> 10);
  v.r1 = ((unsigned long long)v.r0 << 32) + (unsigned long long)(((long long)e * (int)v.r0) >> 20);
  return v;
}
// (out of line: inlined, its instructions were issued for all lanes of a column, 500 clocks)
static __device__ __noinline__ double quotient_special(double a, double d) { return __ddiv_rn(a, d); }
__device__ __forceinline__ double quotient(double a, const Divisor& v) {
  const unsigned long long ab = (unsigned long long)__double_as_longlong(a),
                           db = (unsigned long long)__double_as_longlong(v.d);
  const int ea = (int)(ab >> 52) & 0x7FF, ed = (int)(db >> 52) & 0x7FF;
  const unsigned long long ma = (ab & 0xFFFFFFFFFFFFFull) | (1ull << 52), sign = (ab ^ db) & (1ull << 63);
  const int less = ma < v.md;
  const int e = ea - ed + 1023 - less;
  const unsigned long long n = ma << less;  // n / md in [1, 2)
  unsigned long long q = __umul64hi(n << 10, v.r1) >> 8;
  long long rem = (long long)((n << 53) - q * v.md);
  const int c = (int)(((long long)(int)(rem >> 32) * (int)v.r0) >> 51);
  q += (long long)c;
  rem -= (long long)((unsigned long long)(long long)c * v.md);
  if (rem < 0)
    --q;
  else if ((unsigned long long)rem >= v.md)
    ++q;
  double x = __longlong_as_double((long long)(sign | (((unsigned long long)(e - 1) << 52) + ((q + 1) >> 1))));
  const bool dnormal = (unsigned)(ed - 1) < 2046u;
  if (dnormal && (ab << 1) == 0)
    x = __longlong_as_double((long long)sign);
  else if (!(dnormal && (unsigned)(ea - 1) < 2046u && e >= 1 && e <= 2046))
    x = quotient_special(a, v.d);
  return x;
}
__device__ __forceinline__ double divide(double a, double d) { return quotient(a, divisor(d)); }
__device__ __forceinline__ float divide(float a, float d) { return a / d; }

}  // namespace pdeshep
