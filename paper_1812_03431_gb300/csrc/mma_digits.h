// Digits of fixed-point numbers as fp16 pairs and their products on the tensor cores
// (solve_digits.cu, legendre_digits.cu).
#pragma once

#include <cuda_runtime.h>

#include "fixed.h"

namespace rexi {
namespace fixed {

__device__ __forceinline__ unsigned half2_sub(unsigned a, unsigned b) {
  unsigned r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// the eight balanced digits of (re, im), most significant first, as fp16 pairs: bytes of the
// biased number under the fp16 exponent of 1024, less 1024 + 128
__device__ __forceinline__ void digits(long long re, long long im, unsigned (&w)[8]) {
  const unsigned long long ur = (unsigned long long)re + 0x8080808080808080ull;
  const unsigned long long ui = (unsigned long long)im + 0x8080808080808080ull;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned r = h == 0 ? (unsigned)(ur >> 32) : (unsigned)ur, i = h == 0 ? (unsigned)(ui >> 32) : (unsigned)ui;
    const unsigned top = __byte_perm(r, i, 0x7362), low = __byte_perm(r, i, 0x5140);
    w[4 * h + 0] = half2_sub(__byte_perm(top, 0x64646464u, 0x4342), 0x64806480u);
    w[4 * h + 1] = half2_sub(__byte_perm(top, 0x64646464u, 0x4140), 0x64806480u);
    w[4 * h + 2] = half2_sub(__byte_perm(low, 0x64646464u, 0x4342), 0x64806480u);
    w[4 * h + 3] = half2_sub(__byte_perm(low, 0x64646464u, 0x4140), 0x64806480u);
  }
}

// the same digits as stored: biased bytes, each place's pair (re, im) side by side, most
// significant first
__device__ __forceinline__ uint4 packed_digits(long long re, long long im) {
  const unsigned long long ur = (unsigned long long)re + 0x8080808080808080ull;
  const unsigned long long ui = (unsigned long long)im + 0x8080808080808080ull;
  const unsigned rh = (unsigned)(ur >> 32), rl = (unsigned)ur, ih = (unsigned)(ui >> 32), il = (unsigned)ui;
  return make_uint4(__byte_perm(rh, ih, 0x6273), __byte_perm(rh, ih, 0x4051), __byte_perm(rl, il, 0x6273),
                    __byte_perm(rl, il, 0x4051));
}

__device__ __forceinline__ unsigned half2_fma(unsigned a, unsigned b, unsigned c) {
  unsigned r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// stored digits as fp16 pairs, times `one` (+-1 each, less = -+1152)
__device__ __forceinline__ void unpack(uint4 d, unsigned one, unsigned less, unsigned (&w)[8]) {
  const unsigned v[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    w[2 * j] = half2_fma(__byte_perm(v[j], 0x64646464u, 0x4140), one, less);
    w[2 * j + 1] = half2_fma(__byte_perm(v[j], 0x64646464u, 0x4342), one, less);
  }
}

// An accumulator's bits are kMagicBits + its sum (kEvenBits for those that start at kEven), so
// that of two neighbouring sums 256 bits(even) + bits(odd) = 256 s_c + s_{c+1} + 2^31.
constexpr float kMagic = 12582912.0f;  // 1.5 2^23
constexpr float kEven = 11845632.0f;
constexpr unsigned kMagicBits = 0x4B400000u, kEvenBits = 0x4B34C000u;
static_assert(kEvenBits * 256u + kMagicBits == 0x80000000u, "the pair's offset");

__device__ __forceinline__ unsigned bits(float x) { return (unsigned)__float_as_int(x); }

// sum of s_c 2^(-8c), c = 0..7, in units of 2^-46; the pairs (s_0, s_1) ... (s_6, s_7) come as
// 256 s_c + s_{c+1} + 2^31
__device__ __forceinline__ long long weigh(unsigned h, unsigned m, unsigned l, unsigned q) {
  unsigned long long t = (unsigned long long)h << 32 | l;
  asm("mad.wide.u32 %0, %1, 65536, %0;" : "+l"(t) : "r"(m));
  return (long long)((t << 6) + (q >> 10) - ((1ull << 53) + (1ull << 37) + (1ull << 21)));
}

__device__ __forceinline__ void mma_first(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                          unsigned b1, float start = kMagic) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(start));
}
__device__ __forceinline__ void mma_add(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                        unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

}  // namespace fixed
}  // namespace rexi
