// Fixed-point forms of binary64 values and back, on the integer pipe (the solves of
// solve_digits.cu and solve_limbs.cu).  On GB300 the FP64 unit, which also executes the
// hardware's 64-bit conversions, issues one warp instruction per 64 cycles and scheduler; each
// conversion here takes 10 to 30 integer instructions of one cycle.
#pragma once

#include <cuda_runtime.h>

namespace rexi {
namespace fixed {

constexpr int kNotFinite = 1 << 20;  // exponent of a group that holds an Inf or NaN
// Bits by which a pole's couplings may differ in scale from the middle pole's, and reciprocals of the
// shifts from the largest: |alpha| up to some 2^8.
constexpr int kMaxSpread = 8;

__device__ __forceinline__ int bexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x as a fixed-point number of 61 bits below its group's leading bit, d = that bit's exponent
// less x's own (truncated at 2^-61 of the leading bit; zero and subnormal x give zero)
__device__ __forceinline__ long long to_fixed(double x, int d) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  m = (m << 9) >> (d & 63);
  if (d > 63 || !(hi & 0x7ff00000u)) m = 0;
  return (int)hi < 0 ? -(long long)m : (long long)m;
}

// t 2^e in binary64 (round half away from zero), on the integer pipe; results below 2^-1022
// are zero, e of a group that is not finite gives NaN
__device__ __forceinline__ double fixed_to_double(long long t, int e) {
  const int sign = (int)(t >> 63);
  const unsigned long long m = (unsigned long long)((t ^ (long long)sign) - (long long)sign);
  unsigned h = (unsigned)(m >> 32), l = (unsigned)m;
  int be = 1023 + 62 + e;  // the biased exponent less one of a number with bit 63 set
  if (h == 0) {
    h = l;
    l = 0;
    be -= 32;
  }
  const int lz = __clz((int)h);  // 32 where t is zero: the shifts take it as 0
  const unsigned fh = __funnelshift_l(l, h, lz), fl = l << (lz & 31);
  be -= lz;
  const unsigned long long r =
      ((unsigned long long)(fh >> 11) << 32 | __funnelshift_r(fl, fh, 11)) + ((fl >> 10) & 1);
  unsigned hi = (unsigned)(r >> 32) + ((unsigned)be << 20), lo = (unsigned)r;
  if ((unsigned)be >= 2046u || fh == 0) {
    const bool nan = e >= kNotFinite / 2;
    hi = nan ? 0x7ff80000u : (be >= 2046 && fh != 0 ? 0x7ff00000u : 0u);
    lo = 0;
  }
  return __hiloint2double((int)(hi | ((unsigned)sign & 0x80000000u)), (int)lo);
}

__device__ __forceinline__ double2 cfms(double2 acc, double2 a, double2 b) {
  double re = fma(-a.x, b.x, acc.x), im = fma(-a.x, b.y, acc.y);
  return make_double2(fma(a.y, b.y, re), fma(-a.y, b.x, im));
}
__device__ __forceinline__ double2 cfma(double2 acc, double2 a, double2 b) {
  double re = fma(a.x, b.x, acc.x), im = fma(a.x, b.y, acc.y);
  return make_double2(fma(-a.y, b.y, re), fma(a.y, b.x, im));
}

}  // namespace fixed
}  // namespace rexi
