// Several quotients by one binary64 divisor.
#pragma once

#include <cuda_runtime.h>

namespace rexi {

// a / d as the product by 1/d, corrected by its remainder (Markstein, IBM J. Res. Dev. 34, 1990: with
// 1/d correctly rounded the corrected quotient is), three FP64 instructions each after the one
// division.  Divisors whose reciprocal or remainders leave the normal range are divided by.
struct Recip {
  double d, r;
  bool plain;
  __device__ __forceinline__ explicit Recip(double d_) : d(d_), r(1.0 / d_) {
    const int e = (__double2hiint(d_) >> 20) & 0x7ff;
    plain = e < 200 || e > 1800;
  }
  __device__ __forceinline__ double of(double a) const {
    const int e = (__double2hiint(a) >> 20) & 0x7ff;
    if (plain || e < 200 || e > 1800) return a / d;
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
