// The sweeps of solve_digits.cu, shared with the ragged launch.
#pragma once

#include <cuda_runtime.h>

#include "fixed.h"
#include "mma_digits.h"
#include "rexi_internal.h"

namespace rexi {
namespace digit_solve {

using namespace fixed;

constexpr int kTile = 8;                   // states per warp
constexpr int kWin = 8;                    // poles per window
constexpr int kLOff = 512, kEOff = 640, kFwdRec = 672;  // per (row, window): coupling digits, l, exponents
constexpr int kCOff = 512, kBwdRec = 576;  // per (row, window): weight digits and exponents, |Chat| of the row before
constexpr int kStateRec = 1024;            // per (row, tile): input digits

struct DigitSweep {
  const char *fwd, *bwd, *dig;
  const int *uexp;
  const int4 *sys, *items;  // {system, tile, first window | windows << 16, slot}
  double *part;             // [slots][nrows][tiles][4 streams][re, im][8 states]
  double2 *ybuf;            // per resident warp: [lmax][2][32]
  unsigned *counter;
  int64_t nrows;
  int nitems, tiles, nwin, lmax;
};

__device__ __forceinline__ void load_words(const char *p, unsigned (&w)[8]) {
  const uint4 x = reinterpret_cast<const uint4 *>(p)[0], y = reinterpret_cast<const uint4 *>(p)[1];
  w[0] = x.x, w[1] = x.y, w[2] = x.z, w[3] = x.w, w[4] = y.x, w[5] = y.y, w[6] = y.z, w[7] = y.w;
}

// Staging: a warp's next rows are copied into shared memory while it works on one (three forward
// stages: the record, the inputs' digits and exponents; two backward ones), so that no row
// waits for L2.
constexpr int kSIn = kFwdRec, kSU = kSIn + kStateRec, kStage = kSU + 32;
constexpr int kFwdStages = 3;
constexpr int kSmemWarp = kFwdStages * kStage;
static_assert(kStage % 16 == 0 && kSmemWarp >= 2 * kBwdRec, "stages");

__device__ __forceinline__ void copy_async(unsigned to, const void *from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" : : "r"(to), "l"(from) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" : : : "memory"); }
template <int PENDING>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" : : "n"(PENDING) : "memory"); }

// |x| as to_fixed gives it, E the exponent (biased) of its group's leading bit
__device__ __forceinline__ unsigned long long magnitude(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int d = min(E - (int)((hi >> 20) & 0x7ff), 63);
  unsigned h = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 9), l = lo << 9;
  if (d >= 32) {
    l = h;
    h = 0;
  }
  return (unsigned long long)(h >> (d & 31)) << 32 | __funnelshift_r(l, h, d & 31);
}

// the eight digits of two numbers of one group, as fp16 pairs
__device__ __forceinline__ void digits_of(double a, double b, int E, unsigned (&w)[8]) {
  const unsigned long long ua = magnitude(a, E) + 0x8080808080808080ull, ub = magnitude(b, E) + 0x8080808080808080ull;
  const unsigned sign = __byte_perm((unsigned)__double2hiint(a), (unsigned)__double2hiint(b), 0x7632) & 0x80008000u;
  const unsigned one = sign | 0x3c003c00u, less = sign ^ 0xe480e480u;  // +-1 and -+1152
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned x = h == 0 ? (unsigned)(ua >> 32) : (unsigned)ua, y = h == 0 ? (unsigned)(ub >> 32) : (unsigned)ub;
    const unsigned top = __byte_perm(x, y, 0x7362), low = __byte_perm(x, y, 0x5140);
    w[4 * h + 0] = half2_fma(__byte_perm(top, 0x64646464u, 0x4342), one, less);
    w[4 * h + 1] = half2_fma(__byte_perm(top, 0x64646464u, 0x4140), one, less);
    w[4 * h + 2] = half2_fma(__byte_perm(low, 0x64646464u, 0x4342), one, less);
    w[4 * h + 3] = half2_fma(__byte_perm(low, 0x64646464u, 0x4140), one, less);
  }
}

// The right-hand sides of one row for the lane's two poles: digits of the inputs (rows of the
// product: states, real rows above imaginary ones) times those of the couplings (columns:
// poles), one accumulator per sum of digit places, two digit pairs per MMA.
__device__ __forceinline__ void right_hand_sides(const char *f, int lane, double2 (&r)[2]) {
  unsigned p[8], v[8], z[8];
  load_words(f + kSIn + lane * 32, p);
  unpack(reinterpret_cast<const uint4 *>(f)[lane], 0x3c003c00u, 0xe480e480u, v);
  const int U = reinterpret_cast<const int *>(f + kSU)[lane >> 2] - 56;
  const int2 e = reinterpret_cast<const int2 *>(f + kEOff)[lane & 3];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    z[j] = __byte_perm(p[j], 0, 0x1032);  // (im, re): imaginary rows
    p[j] ^= 0x80000000u;                  // (re, -im): real rows
  }
  unsigned pair[4][4];
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    float s[2][4];
#pragma unroll
    for (int o = 0; o < 2; ++o)
#pragma unroll
      for (int i = 0; i <= c + o; i += 2) {
        const int j = c + o - i;
        const unsigned a2 = j > 0 ? p[i < 7 ? i + 1 : 7] : 0u, a3 = j > 0 ? z[i < 7 ? i + 1 : 7] : 0u, b1 = j > 0 ? v[j > 0 ? j - 1 : 0] : 0u;
        if (i == 0) mma_first(s[o], p[i], z[i], a2, a3, v[j], b1, o == 0 ? kEven : kMagic);
        else mma_add(s[o], p[i], z[i], a2, a3, v[j], b1);
      }
#pragma unroll
    for (int k = 0; k < 4; ++k) pair[c / 2][k] = bits(s[0][k]) * 256u + bits(s[1][k]);
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int ee = U + (g ? e.y : e.x);
    r[g] = make_double2(fixed_to_double(weigh(pair[0][g], pair[1][g], pair[2][g], pair[3][g]), ee),
                        fixed_to_double(weigh(pair[0][g + 2], pair[1][g + 2], pair[2][g + 2], pair[3][g + 2]), ee));
  }
}

// Adds to the lane's two running sums (states 2 q and 2 q + 1 of one stream's real or
// imaginary part) the weighted sums over the window's eight poles of x, a row's solutions:
// digits of the weights (rows: streams) times those of x (columns: states).
__device__ __forceinline__ double2 weighted_sums(const char *f, const double2 (&x)[2], int lane, double2 sum) {
  const int q = lane & 3;
  const bool im_row = (lane >> 2) & 1;
  // a real row takes (re, -im) of the weights against (re, im) of x, an imaginary one (im, re)
  unsigned lo[8], hi[8];
  const uint4 *wr = reinterpret_cast<const uint4 *>(f) + ((lane >> 3) * 4 + q) * 2;
  const uint4 dl = wr[im_row ? 1 : 0], dh = wr[im_row ? 0 : 1];
  const int We = (int)dl.w >> 16;
  unpack(dl, 0x3c003c00u, 0xe480e480u, lo);
  unpack(dh, im_row ? 0x3c003c00u : 0xbc00bc00u, im_row ? 0xe480e480u : 0x64806480u, hi);
  lo[7] = hi[7] = 0;
  int E = 0;
#pragma unroll
  for (int g = 0; g < 2; ++g) E = max(E, max(__double2hiint(x[g].x) & 0x7fffffff, __double2hiint(x[g].y) & 0x7fffffff));
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
  E = max(E, __shfl_xor_sync(0xffffffffu, E, 2)) >> 20;
  if (E < 64) E += 4096;  // groups below 2^-959 are taken as zero
  unsigned re[8], im[8];
  digits_of(x[0].x, x[1].x, E, re);
  digits_of(x[0].y, x[1].y, E, im);
  float s[8][4];
#pragma unroll
  for (int c = 0; c < 8; ++c) mma_first(s[c], lo[0], lo[1], hi[0], hi[1], re[c], im[c]);
#pragma unroll
  for (int i = 2; i < 8; i += 2)
#pragma unroll
    for (int c = i; c < 8; ++c) mma_add(s[c], lo[i], lo[i + 1], hi[i], hi[i + 1], re[c - i], im[c - i]);
  double r[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int Es = __shfl_sync(0xffffffffu, E, (q * 2 + c) * 4);  // the exponent of state 2 q + c
    // digit places j come from the upper rows of accumulator j and the lower ones of j - 1
    unsigned at[8];
    at[0] = bits(s[0][c]) + (0x00800000u - kMagicBits);
#pragma unroll
    for (int j = 1; j < 8; ++j) at[j] = bits(s[j][c]) + bits(s[j - 1][c + 2]) + ((j & 1 ? 0u : 0x00800000u) - 2u * kMagicBits);
    r[c] = fixed_to_double(weigh(at[0] * 256u + at[1], at[2] * 256u + at[3], at[4] * 256u + at[5], at[6] * 256u + at[7]),
                           (Es & 4095) == 0x7ff ? kNotFinite : We + (Es & 4095) - 1023 - 56);
  }
  return make_double2(sum.x + r[0], sum.y + r[1]);
}

// One item: {system, tile, first window | windows << 16, slot}; yb: the lane's place in the warp's
// sweep buffer, smem: the warp's stages.
__device__ __forceinline__ void digit_item(const DigitSweep &a, int4 item, int lane, double2 *yb, char *smem) {
  const int q = lane & 3;
  const int4 sy = a.sys[item.x];
  const int len = sy.z, w0 = item.z & 0xffff, w1 = w0 + (item.z >> 16);
  const int64_t row0 = sy.w;
  const int dstep = a.tiles * kStateRec, ustep = a.tiles * kTile, pstep = a.tiles * 32;
  double2 *part0 = reinterpret_cast<double2 *>(a.part + (((int64_t)item.w * a.nrows + row0) * a.tiles + item.y) * 64) + lane;
  const unsigned sm = (unsigned)__cvta_generic_to_shared(smem);
  for (int w = w0; w < w1; ++w) {
    {  // forward: y_i = r_i - l y_{i-1}; the next row's r is formed beside the FMAs of this one
      const char *f = a.fwd + (row0 * a.nwin + (int64_t)w * len) * kFwdRec + lane * 16;
      const char *dig = a.dig + (row0 * a.tiles + item.y) * kStateRec + lane * 16;
      const int *uexp = a.uexp + (row0 * a.tiles + item.y) * kTile;
      int todo = len;
      unsigned to = sm;
      auto issue = [&]() {
        if (todo > 0) {
          copy_async(to + lane * 16, f);
          copy_async(to + kSIn + lane * 16, dig);
          copy_async(to + kSIn + 512 + lane * 16, dig + 512);
          if (lane < 10) copy_async(to + 512 + lane * 16, f + 512);
          else if (lane < 12) copy_async(to + kSU + (lane - 10) * 16, uexp + (lane - 10) * 4);
          f += kFwdRec;
          dig += dstep;
          uexp += ustep;
          --todo;
          to = to == sm + (kFwdStages - 1) * kStage ? sm : to + kStage;
        }
        copy_commit();
      };
      __syncwarp();  // every lane has read the stages of the window before
      issue();
      issue();
      const char *stage = smem;
      double2 *yp = yb;
      double2 y[2] = {make_double2(0, 0), make_double2(0, 0)}, r[2], l[2];
      for (int i = 0; i <= len; ++i) {
        if (i > 0) {
          y[0] = cfms(r[0], l[0], y[0]);
          y[1] = cfms(r[1], l[1], y[1]);
        }
        if (i < len) {
          copy_wait<1>();
          __syncwarp();  // row i has landed for every lane; the stage of row i - 1 has been read
          issue();
          right_hand_sides(stage, lane, r);
          l[0] = reinterpret_cast<const double2 *>(stage + kLOff)[2 * q];
          l[1] = reinterpret_cast<const double2 *>(stage + kLOff)[2 * q + 1];
          stage = stage == smem + (kFwdStages - 1) * kStage ? smem : stage + kStage;
        }
        if (i > 0) {
          yp[0] = y[0];
          yp[32] = y[1];
          yp += 64;
        }
      }
    }
    {  // backward: x_i = y_i - |Chat| x_{i+1}; the sums of row i + 1 beside the FMAs of row i
      const char *f = a.bwd + (row0 * a.nwin + (int64_t)(w + 1) * len - 1) * kBwdRec + lane * 16;
      int todo = len;
      unsigned odd = 0;
      auto issue = [&]() {
        if (todo > 0) {
          const unsigned to = sm + odd * kBwdRec + lane * 16;
          copy_async(to, f);
          if (lane < 4) copy_async(to + 512, f + 512);
          f -= kBwdRec;
          --todo;
          odd ^= 1;
        }
        copy_commit();
      };
      copy_wait<0>();
      __syncwarp();
      issue();
      const double2 *yp = yb + (len - 1) * 64;
      double2 *part = part0 + (int64_t)(len - 1) * pstep;
      double2 x[2] = {yp[0], yp[32]};  // Chat is zero in the last row
      double2 y[2] = {x[0], x[1]};
      if (len > 1) {
        y[0] = yp[-64];
        y[1] = yp[-32];
      }
      for (int i = len - 1; i >= 0; --i) {
        double2 sum = make_double2(0, 0);
        if (w > w0) sum = *part;
        const char *stage = smem + (odd ^ 1) * kBwdRec;
        copy_wait<0>();
        __syncwarp();  // row i has landed for every lane; the stage of row i + 1 has been read
        issue();
        // Chat of row i - 1 is stored with row i (zero with row 0, whose xn is not used)
        const double2 c = reinterpret_cast<const double2 *>(stage + kCOff)[q];
        const double2 xn[2] = {make_double2(fma(-c.x, x[0].x, y[0].x), fma(-c.x, x[0].y, y[0].y)),
                               make_double2(fma(-c.y, x[1].x, y[1].x), fma(-c.y, x[1].y, y[1].y))};
        if (i > 1) {
          y[0] = yp[-128];
          y[1] = yp[-96];
        }
        *part = weighted_sums(stage, x, lane, sum);
        part -= pstep;
        yp -= 64;
        x[0] = xn[0];
        x[1] = xn[1];
      }
    }
  }
}

}  // namespace digit_solve
}  // namespace rexi
