// The sweeps of solve_limbs.cu, shared with the ragged launch.
#pragma once

#include <cuda_runtime.h>

#include "fixed.h"
#include "rexi_internal.h"

namespace rexi {
namespace limb_solve {

using namespace fixed;

constexpr int kBlock = 64;  // poles per record
// per (row, block of 64 poles): [g][e][f] limbs, l, exponents (kNoPole past the last pole)
constexpr int kFL = 3 * 1024, kFE = 4 * 1024, kFwd = 4 * 1024 + 256;
constexpr int kNoPole = 1000;
// per (row, block): Chat of the row before, [bd][bad][zp][zm] limbs, the four exponents
constexpr int kBW = 1024, kBE = 5 * 1024, kBwd = 5 * 1024 + 16;

// v as limbs: v = x 2^30 + y, -2^29 <= y < 2^29
__device__ __forceinline__ int2 limbs(long long v) {
  const int y = (int)((unsigned)v << 2) >> 2;
  return make_int2((int)((v + (1 << 29)) >> 30), y);
}
__device__ __forceinline__ int4 limbs2(long long re, long long im) {
  const int2 a = limbs(re), b = limbs(im);
  return make_int4(a.x, a.y, b.x, b.y);
}

struct LimbSweep {
  const char *fwd, *bwd;
  const int4 *dig;
  const int *uexp;
  const int4 *sys, *items;  // {system, tile, first window | windows << 16, slot}
  double *part;             // [slots][nrows][B][4 streams][re, im]
  double2 *ybuf;            // per resident warp: [lmax][2][32]
  unsigned *counter;
  int64_t nrows;
  int nitems, B, P, nblk, lmax, kc;
};

// Staging: each lane copies the factors of its poles for the rows ahead into shared memory
// (three forward stages, two backward), and the row's inputs are copied once per warp.  Bytes
// of a forward stage: (g, e, f, l) per pole of the lane, exponents, inputs and their exponents.
constexpr int kSE = 2 * 4 * 512, kSIn = kSE + 256, kSU = kSIn + 256, kStage = kSU + 64;
constexpr int kFwdStages = 3;
constexpr int kSmemWarp = kFwdStages * kStage;
static_assert(kSmemWarp >= 2 * 2 * 5 * 512, "two backward stages");

template <int BYTES>
__device__ __forceinline__ void copy_async(unsigned to, const void *from) {
  if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" : : "r"(to), "l"(from) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" : : "r"(to), "l"(from), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" : : : "memory"); }
template <int PENDING>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" : : "n"(PENDING) : "memory"); }

// acc += a b in one instruction (written as a C++ product it compiles to several)
__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// high and middle sums of limb products; a and b stand for (x 2^30 + y)
__device__ __forceinline__ void mad(long long &hh, long long &hl, int ax, int ay, int bx, int by) {
  mad_wide(hh, ax, bx);
  mad_wide(hl, ax, by);
  mad_wide(hl, ay, bx);
}

// |x| < 2^(E + 1) as a signed 59-bit integer, E (biased) its group's largest exponent
__device__ __forceinline__ long long fixed59(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int d = min(E - (int)((hi >> 20) & 0x7ff), 63);
  unsigned h = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 6), l = lo << 6;
  if (d >= 32) {
    l = h;
    h = 0;
  }
  const long long s = (int)hi >> 31;
  return (long long)(((unsigned long long)(h >> (d & 31)) << 32 | __funnelshift_r(l, h, d & 31)) ^ (unsigned long long)s) - s;
}

// r = delta0 - g Phi0 - e zeta0_{n-1} - f zeta0_{n+1} at one row for the lane's KC poles, and l,
// from a forward stage; s: the lane's state
template <int KC>
__device__ __forceinline__ void right_hand_sides(const char *stage, int s, int lane, double2 (&r)[2], double2 (&l)[2]) {
  int4 in[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) in[j] = reinterpret_cast<const int4 *>(stage + kSIn)[s * 4 + j];
  const int U = reinterpret_cast<const int *>(stage + kSU)[s] - 57;
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    const int e = reinterpret_cast<const int *>(stage + kSE)[c * 32 + lane];
    // delta: its weight is a power of two, one limb
    const int one = e > 28 ? 0 : 1 << (28 - e);
    long long rh = 0, rl = 1 << 28, ih = 0, il = 1 << 28;  // the middle sums are rounded at bit 29
    mad_wide(rh, one, in[0].x);
    mad_wide(rl, one, in[0].y);
    mad_wide(ih, one, in[0].z);
    mad_wide(il, one, in[0].w);
#pragma unroll
    for (int j = 1; j < 4; ++j) {
      const int4 v = reinterpret_cast<const int4 *>(stage)[(c * 4 + j - 1) * 32 + lane];
      mad(rh, rl, v.x, v.y, in[j].x, in[j].y);
      mad(rh, rl, -v.z, -v.w, in[j].z, in[j].w);
      mad(ih, il, v.x, v.y, in[j].z, in[j].w);
      mad(ih, il, v.z, v.w, in[j].x, in[j].y);
    }
    l[c] = reinterpret_cast<const double2 *>(stage)[(c * 4 + 3) * 32 + lane];
    r[c] = make_double2(fixed_to_double((rh << 1) + (rl >> 29), U + e), fixed_to_double((ih << 1) + (il >> 29), U + e));
  }
}

// The window's weighted sums of a row's solutions x, over the lanes of each state: returns the
// one of the eight (stream, part) values that this lane ends up with (index: see sum_index).
template <int SB, int KC>
__device__ __forceinline__ double weighted_sums(const char *stage, int wexp, const double2 (&x)[2], int lane) {
  constexpr int LPS = 32 / SB;  // lanes per state
  int E = 0;
#pragma unroll
  for (int c = 0; c < KC; ++c) E = max(E, max(__double2hiint(x[c].x) & 0x7fffffff, __double2hiint(x[c].y) & 0x7fffffff));
#pragma unroll
  for (int o = 1; o < LPS; o <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  E >>= 20;
  const bool finite = E != 0x7ff;
  const int Ew = E - 1023 - 53;
  if (E < 64) E += 4096;  // groups below 2^-959 are taken as zero
  long long hh[8], hl[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) hh[j] = 0, hl[j] = 1 << 29;  // rounded at bit 30
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    const int2 re = limbs(fixed59(x[c].x, E)), im = limbs(fixed59(x[c].y, E));
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int4 v = reinterpret_cast<const int4 *>(stage)[(c * 5 + 1 + s) * 32 + lane];
      mad(hh[2 * s], hl[2 * s], v.x, v.y, re.x, re.y);
      mad(hh[2 * s], hl[2 * s], v.z, v.w, -im.x, -im.y);
      mad(hh[2 * s + 1], hl[2 * s + 1], v.x, v.y, im.x, im.y);
      mad(hh[2 * s + 1], hl[2 * s + 1], v.z, v.w, re.x, re.y);
    }
  }
  long long t[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) t[j] = hh[j] + (hl[j] >> 30);
  int n = 8;
#pragma unroll
  for (int o = LPS / 2; o > 0; o >>= 1) {
    if (n > 1) {  // keep one half of the values, add the partner's
      n >>= 1;
      const bool up = lane & o;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < n) {
          const long long give = up ? t[j] : t[j + n], keep = up ? t[j + n] : t[j];
          t[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    } else {
      t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
    }
  }
  return fixed_to_double(t[0], finite ? Ew + wexp : kNotFinite);
}

// the value a lane holds after weighted_sums (2 stream + part), -1 for lanes that repeat another's
template <int SB>
__device__ __forceinline__ int sum_index(int lane) {
  constexpr int LPS = 32 / SB;
  const int k = lane & (LPS - 1), rest = LPS / 8;
  return (k & (rest - 1)) ? -1 : k / rest;
}

template <int SB, int KC>
__device__ void sweep_window(const LimbSweep &a, int64_t row0, int len, int p0, int b0, int idx, double *part, bool first,
                             double2 *yb, char *smem, int lane) {
  constexpr int LPS = 32 / SB;
  const int k = lane & (LPS - 1), s = lane / LPS, blk = p0 / kBlock, pk = p0 % kBlock + k;
  const int64_t rec = row0 * a.nblk + (int64_t)blk * len;
  const unsigned sm = (unsigned)__cvta_generic_to_shared(smem);
  {  // forward: y_i = r_i - l y_{i-1}; row i + 1's r is formed beside the FMAs of row i
    const char *f = a.fwd + rec * kFwd;
    const int4 *dig = a.dig + (row0 * a.B + b0) * 4;
    const int *uexp = a.uexp + row0 * a.B + b0;
    const int ns = min(SB, a.B - b0);  // states with inputs of their own
    int todo = len;                    // rows not copied yet
    unsigned to = sm;
    auto issue = [&]() {
      if (todo > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) {
#pragma unroll
          for (int j = 0; j < 4; ++j) copy_async<16>(to + (c * 4 + j) * 512 + lane * 16, f + j * 1024 + (pk + c * LPS) * 16);
          copy_async<4>(to + kSE + (c * 32 + lane) * 4, f + kFE + (pk + c * LPS) * 4);
        }
        if (lane < 4 * ns) copy_async<16>(to + kSIn + lane * 16, dig + lane);
        else if (lane >= 16 && lane < 16 + ns) copy_async<4>(to + kSU + (lane - 16) * 4, uexp + lane - 16);
        f += kFwd;
        dig += a.B * 4;
        uexp += a.B;
        --todo;
        to = to == sm + (kFwdStages - 1) * kStage ? sm : to + kStage;
      }
      copy_commit();
    };
    __syncwarp();  // every lane has read the stages of the window before
    issue();
    issue();
    const int mine = min(s, ns - 1);
    double2 *yp = yb;
    const char *stage = smem;
    double2 y[2] = {make_double2(0, 0), make_double2(0, 0)}, r[2], l[2];
    for (int i = 0; i <= len; ++i) {
      if (i > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) y[c] = cfms(r[c], l[c], y[c]);
      }
      if (i < len) {
        copy_wait<1>();
        __syncwarp();  // row i has landed for every lane; the stage of row i - 1 has been read
        issue();
        right_hand_sides<KC>(stage, mine, lane, r, l);
        stage = stage == smem + (kFwdStages - 1) * kStage ? smem : stage + kStage;
      }
      if (i > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) yp[c * 32] = y[c];
        yp += 64;
      }
    }
  }
  {  // backward: x_i = y_i - Chat x_{i+1}; the sums of row i + 1 beside the FMAs of row i
    const char *f = a.bwd + (rec + len - 1) * kBwd;
    int todo = len;
    unsigned odd = 0;
    auto issue = [&]() {  // the lane's own copies only
      if (todo > 0) {
        const unsigned to = sm + odd * (KC * 5 * 512) + lane * 16;
#pragma unroll
        for (int c = 0; c < KC; ++c)
#pragma unroll
          for (int j = 0; j < 5; ++j) copy_async<16>(to + (c * 5 + j) * 512, f + j * 1024 + (pk + c * LPS) * 16);
        f -= kBwd;
        --todo;
        odd ^= 1;
      }
      copy_commit();
    };
    const int *we = reinterpret_cast<const int *>(f + kBE) + (idx >= 0 ? idx >> 1 : 0);
    copy_wait<0>();
    __syncwarp();
    issue();
    const double2 *yp = yb + (len - 1) * 64;
    part += (int64_t)(len - 1) * a.B * 8 + (idx > 0 ? idx : 0);
    double2 x[2], y[2];
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      x[c] = yp[c * 32];  // Chat is zero in the last row
      y[c] = len > 1 ? yp[c * 32 - 64] : x[c];
    }
    for (int i = len - 1; i >= 0; --i) {
      const char *stage = smem + (odd ^ 1) * (KC * 5 * 512);
      const int wexp = __ldg(we);
      double sum = 0;
      if (!first && idx >= 0) sum = *part;
      copy_wait<0>();
      issue();
      double2 xn[2];
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        // Chat of row i - 1 is stored with row i (zero with row 0, whose xn is not used)
        xn[c] = cfms(y[c], reinterpret_cast<const double2 *>(stage)[(c * 5) * 32 + lane], x[c]);
        if (i > 1) y[c] = yp[c * 32 - 128];
      }
      const double v = weighted_sums<SB, KC>(stage, wexp, x, lane);
      if (idx >= 0) *part = sum + v;
      part -= a.B * 8;
      we = reinterpret_cast<const int *>(reinterpret_cast<const char *>(we) - kBwd);
      yp -= 64;
#pragma unroll
      for (int c = 0; c < KC; ++c) x[c] = xn[c];
    }
  }
}

// One item: {system, tile, first window | windows << 16, slot}; yb: the lane's place in the warp's
// sweep buffer, smem: the warp's stages.
template <int SB>
__device__ __forceinline__ void limb_item(const LimbSweep &a, int4 item, int lane, double2 *yb, char *smem) {
  constexpr int LPS = 32 / SB;
  const int per = a.kc * LPS;  // poles per window
  const int4 sy = a.sys[item.x];
  const int w0 = item.z & 0xffff, w1 = w0 + (item.z >> 16);
  // lanes of a state past the batch repeat the last one and write nothing
  const int b0 = item.y * SB, state = b0 + lane / LPS, idx = state < a.B ? sum_index<SB>(lane) : -1;
  double *part = a.part + (((int64_t)item.w * a.nrows + sy.w) * a.B + min(state, a.B - 1)) * 8;
  for (int w = w0; w < w1; ++w) {
    const int p0 = w * per;
    if (a.kc == 2 && p0 + LPS < a.P) sweep_window<SB, 2>(a, sy.w, sy.z, p0, b0, idx, part, w == w0, yb, smem, lane);
    else sweep_window<SB, 1>(a, sy.w, sy.z, p0, b0, idx, part, w == w0, yb, smem, lane);
  }
}

}  // namespace limb_solve
}  // namespace rexi
