// Several quotients by one binary64 divisor.
#pragma once

#include <cuda_runtime.h>

namespace rexi {

// a / d as the product by 1/d, corrected by its remainder (Markstein, IBM J. Res. Dev. 34, 1990: with
// 1/d correctly rounded the corrected quotient is), three FP64 instructions each after the one
// division.  Where the reciprocal, the quotient or the remainder could leave the normal range (biased
// exponents outside [200, 1800], or a's and d's more than 900 apart), a is divided.
struct Recip {
  double d, r;
  int least, most;  // exponents of a for the product
  __device__ __forceinline__ explicit Recip(double d_) : d(d_), r(1.0 / d_) {
    const int e = (__double2hiint(d_) >> 20) & 0x7ff;
    const bool plain = e < 200 || e > 1800;
    least = plain ? 2048 : (e > 1100 ? e - 900 : 200);
    most = e < 900 ? e + 900 : 1800;
  }
  __device__ __forceinline__ double of(double a) const {
    const int e = (__double2hiint(a) >> 20) & 0x7ff;
    if (e < least || e > most) return a / d;
    const double q = a * r;
    return fma(fma(-q, d, a), r, q);
  }
};

// complex quotients by one divisor
struct ComplexRecip {
  double2 b;
  Recip d;
  __device__ __forceinline__ explicit ComplexRecip(double2 b_) : b(b_), d(b_.x * b_.x + b_.y * b_.y) {}
  __device__ __forceinline__ double2 of(double2 a) const {
    return make_double2(d.of(a.x * b.x + a.y * b.y), d.of(a.y * b.x - a.x * b.y));
  }
};

}  // namespace rexi
