// The sweeps of solve_limbs.cu, shared with the ragged launch.
#pragma once

#include <cuda_runtime.h>

#include "fixed.h"
#include "rexi_internal.h"

namespace rexi {
namespace limb_solve {

using namespace fixed;

// Poles per record.  Every factor of a row is a product of one of four complex numbers per pole
// with a real number per row (row_scale) or 1: 1/s_{n-1} and 1/s_{n+1}, s_n = alpha + i tau sigma_n
// (shared by neighbouring rows), 1/alpha (per pole only), and beta/d'; and the recurrences'
// l and Chat.  Records are [pole] arrays of 16 B: `inv` one per (system, block, j = 0..len) of
// 1/s at degree n0 - 1 + 2 j, `fwd` one per (row, block) of l, `bwd` of Chat of the row before
// and beta/d', with the latter's exponents (per pole) behind.
constexpr int kBlock = 64;
constexpr int kRec = kBlock * 16;
constexpr int kBE = 2 * kRec, kBwd = 2 * kRec + kBlock * 4;

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
  const char *fwd, *bwd, *inv;
  const int4 *inv_alpha;    // [P padded]
  const int4 *dig;
  const int *uexp;
  const int4 *sys, *items;  // {system, state, first window | windows << 16, slot}
  double *part;             // [slots][nrows][B][4 streams][re, im]
  double2 *ybuf;            // per resident warp: [lmax][2][32]
  unsigned *counter;
  int64_t nrows;
  int nitems, B, P, nblk, lmax;
  int kc;                   // poles per lane; 3: one, by a CTA per window
  int sms;
  const int *eblk;          // per block of poles: the exponent of its largest 1/s or 1/alpha
  int e0;                   // exponent of the limbs of 1/s and 1/alpha
};

// Staging: each lane copies the factors of its poles for the rows ahead into shared memory
// (rings of four stages), and the row's inputs are copied once per warp.  Bytes of a forward
// stage: (1/s, l) per pole of the lane, inputs and their exponents; of a backward one: (1/s,
// Chat, beta/d').  Behind the ring: 1/alpha per pole of the lane.
constexpr int kSIn = 2 * 2 * 512, kSU = kSIn + 256, kStage = 2 * 3 * 512;
constexpr int kInvAlpha = 4 * kStage, kSmemWarp = kInvAlpha + 2 * 512;
static_assert(kSU + 64 <= kStage, "forward stage");

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

// acc += v w for complex limb pairs (re hi, re lo, im hi, im lo)
__device__ __forceinline__ void cmad(long long &rh, long long &rl, long long &ih, long long &il, int4 v, int4 w) {
  mad(rh, rl, v.x, v.y, w.x, w.y);
  mad(rh, rl, -v.z, -v.w, w.z, w.w);
  mad(ih, il, v.x, v.y, w.z, w.w);
  mad(ih, il, v.z, v.w, w.x, w.y);
}

// r = delta0 + Phi'/alpha + zeta'_{n-1}/s_{n-1} + zeta'_{n+1}/s_{n+1} at one row for the lane's KC
// poles (the inputs carry the row's real factors), and l, from the row's stage and the next
template <int KC>
__device__ __forceinline__ void right_hand_sides(const char *stage, const char *next, const char *inv_alpha, int e0,
                                                 const int (&one)[2], int lane, double2 (&r)[2], double2 (&l)[2]) {
  int4 in[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) in[j] = reinterpret_cast<const int4 *>(stage + kSIn)[j];
  const int e = *reinterpret_cast<const int *>(stage + kSU) + e0 - 57;
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    // delta: its weight 1 is one limb (0 past the last pole)
    long long rh = 0, rl = 1 << 28, ih = 0, il = 1 << 28;  // the middle sums are rounded at bit 29
    mad_wide(rh, one[c], in[0].x);
    mad_wide(rl, one[c], in[0].y);
    mad_wide(ih, one[c], in[0].z);
    mad_wide(il, one[c], in[0].w);
    cmad(rh, rl, ih, il, reinterpret_cast<const int4 *>(inv_alpha)[c * 32 + lane], in[1]);
    cmad(rh, rl, ih, il, reinterpret_cast<const int4 *>(stage)[c * 32 + lane], in[2]);
    cmad(rh, rl, ih, il, reinterpret_cast<const int4 *>(next)[c * 32 + lane], in[3]);
    l[c] = reinterpret_cast<const double2 *>(stage)[(2 + c) * 32 + lane];
    r[c] = make_double2(fixed_to_double((rh << 1) + (rl >> 29), e), fixed_to_double((ih << 1) + (il >> 29), e));
  }
}

// The window's sums over the lanes of u = (beta/d') x, u/alpha, u/s_{n+1} and
// u/s_{n-1}, x a row's solutions: returns the one of the eight (stream, part) values that this lane
// ends up with (index: see sum_index).  prev: the stage of the row before (n + 2); be: the
// exponents of beta/d'; fine: the bits by which the block's reciprocals are below 2^e0; sexp: the
// exponent of the lane's stream.  beta, 1/d' and x vary over the poles by some bits each and not
// together, so each pole's u has an exponent of its own and the window's unit is that of its
// largest u.
template <int KC>
__device__ __forceinline__ double weighted_sums(const char *stage, const char *prev, const char *inv_alpha,
                                                const int (&be)[2], int fine, int sexp, const double2 (&x)[2], int lane) {
  long long ur[2], ui[2];
  int eu[2], E = -(1 << 20);
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    int e = max(__double2hiint(x[c].x) & 0x7fffffff, __double2hiint(x[c].y) & 0x7fffffff) >> 20;
    eu[c] = e == 0x7ff ? kNotFinite : e - 1023 + be[c];
    E = max(E, eu[c]);
    if (e < 64) e += 4096;  // below 2^-959: taken as zero
    long long rh = 0, rl = 1 << 29, ih = 0, il = 1 << 29;
    cmad(rh, rl, ih, il, reinterpret_cast<const int4 *>(stage)[(2 * KC + c) * 32 + lane],
         limbs2(fixed59(x[c].x, e), fixed59(x[c].y, e)));
    ur[c] = rh + (rl >> 30);
    ui[c] = ih + (il >> 30);
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  // sums over up to 64 poles of numbers below 2^59: kept in units of 2^3
  long long hh[8], hl[8], t[8];
  t[0] = t[1] = 4;
#pragma unroll
  for (int j = 2; j < 8; ++j) hh[j] = hl[j] = 0;
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    const int d = min(E - eu[c], 62);
    const long long half = (1ll << d) >> 1;
    ur[c] = (ur[c] + half) >> d;
    ui[c] = (ui[c] + half) >> d;
    t[0] += ur[c];
    t[1] += ui[c];
    const int4 u = limbs2(ur[c], ui[c]);
    cmad(hh[2], hl[2], hh[3], hl[3], reinterpret_cast<const int4 *>(inv_alpha)[c * 32 + lane], u);
    cmad(hh[4], hl[4], hh[5], hl[5], reinterpret_cast<const int4 *>(prev)[c * 32 + lane], u);
    cmad(hh[6], hl[6], hh[7], hl[7], reinterpret_cast<const int4 *>(stage)[c * 32 + lane], u);
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) t[j] = (j < 2 ? t[j] : (hh[j] << fine) + (hl[j] >> (30 - fine)) + 4) >> 3;
  int n = 8;
#pragma unroll
  for (int o = 32 / 2; o > 0; o >>= 1) {
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
  return fixed_to_double(t[0], E >= kNotFinite / 2 ? kNotFinite : E + sexp);
}

// the value a lane holds after weighted_sums (2 stream + part), -1 for lanes that repeat another's
__device__ __forceinline__ int sum_index(int lane) {
  return lane & 3 ? -1 : lane >> 2;
}

template <int KC>
__device__ void sweep_window(const LimbSweep &a, int sysid, int64_t row0, int len, int p0, int b, int idx, double *part,
                             bool first, double2 *yb, char *smem, int lane) {
  const int blk = p0 / kBlock, pk = p0 % kBlock + lane;
  const int64_t rec = row0 * a.nblk + (int64_t)blk * len;
  const char *inv0 = a.inv + ((row0 + sysid) * a.nblk + (int64_t)blk * (len + 1)) * kRec + pk * 16;
  const unsigned sm = (unsigned)__cvta_generic_to_shared(smem);
  const char *ia = smem + kInvAlpha;
  {  // forward: y_i = r_i - l y_{i-1}; row i + 1's r is formed beside the FMAs of row i
    const char *f = a.fwd + rec * kRec + pk * 16, *inv = inv0;
    const int4 *dig = a.dig + (row0 * a.B + b) * 4;
    const int *uexp = a.uexp + row0 * a.B + b;
    int j = 0;                         // next stage to copy, 0..len
    auto issue = [&]() {
      if (j <= len) {
        const unsigned to = sm + (j & 3) * kStage;
#pragma unroll
        for (int c = 0; c < KC; ++c) copy_async<16>(to + (c * 32 + lane) * 16, inv + c * 32 * 16);
        if (j < len) {
#pragma unroll
          for (int c = 0; c < KC; ++c) copy_async<16>(to + ((2 + c) * 32 + lane) * 16, f + c * 32 * 16);
          if (lane < 4) copy_async<16>(to + kSIn + lane * 16, dig + lane);
          else if (lane == 4) copy_async<4>(to + kSU, uexp);
        }
        inv += kRec;
        f += kRec;
        dig += a.B * 4;
        uexp += a.B;
        ++j;
      }
      copy_commit();
    };
    __syncwarp();  // every lane has read the stages of the window before
#pragma unroll
    for (int c = 0; c < KC; ++c) copy_async<16>(sm + kInvAlpha + (c * 32 + lane) * 16, a.inv_alpha + p0 + lane + c * 32);
    issue();
    issue();
    issue();
    const int one[2] = {p0 + lane < a.P ? 1 << (28 - a.e0) : 0, p0 + lane + 32 < a.P ? 1 << (28 - a.e0) : 0};
    double2 *yp = yb;
    double2 y[2] = {make_double2(0, 0), make_double2(0, 0)}, r[2], l[2];
    for (int i = 0; i <= len; ++i) {
      if (i > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) y[c] = cfms(r[c], l[c], y[c]);
      }
      if (i < len) {
        copy_wait<1>();
        __syncwarp();  // stages i and i + 1 have landed for every lane; i - 1 has been read
        issue();
        right_hand_sides<KC>(smem + (i & 3) * kStage, smem + ((i + 1) & 3) * kStage, ia, a.e0, one, lane, r, l);
      }
      if (i > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) yp[c * 32] = y[c];
        yp += 64;
      }
    }
  }
  {  // backward: x_i = y_i - Chat x_{i+1}; the sums of row i + 1 beside the FMAs of row i
    const char *f = a.bwd + (rec + len - 1) * kBwd + pk * 16, *inv = inv0 + (int64_t)len * kRec;
    const int *we = reinterpret_cast<const int *>(a.bwd + (rec + len - 1) * kBwd + kBE) + pk;
    const int fine = min(a.e0 - __ldg(a.eblk + blk), 8), sexp = idx > 1 ? a.e0 - fine - 51 : -53;
    int be[2], bn[2];
#pragma unroll
    for (int c = 0; c < KC; ++c) be[c] = bn[c] = __ldg(we + c * 32);
    int j = len;  // next stage to copy, len..0; the lane's own copies only
    auto issue = [&]() {
      if (j >= 0) {
        const unsigned to = sm + (j & 3) * kStage + lane * 16;
#pragma unroll
        for (int c = 0; c < KC; ++c) copy_async<16>(to + c * 512, inv + c * 32 * 16);
        if (j < len) {
#pragma unroll
          for (int c = 0; c < KC; ++c) {
            copy_async<16>(to + (KC + c) * 512, f + c * 32 * 16);
            copy_async<16>(to + (2 * KC + c) * 512, f + kRec + c * 32 * 16);
          }
          f -= kBwd;
        }
        inv -= kRec;
        --j;
      }
      copy_commit();
    };
    copy_wait<0>();
    __syncwarp();
    issue();
    issue();
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
      const char *stage = smem + (i & 3) * kStage;
      double sum = 0;
      if (!first && idx >= 0) sum = *part;
      we = reinterpret_cast<const int *>(reinterpret_cast<const char *>(we) - kBwd);
      if (i > 0) {
#pragma unroll
        for (int c = 0; c < KC; ++c) bn[c] = __ldg(we + c * 32);
      }
      copy_wait<1>();  // stages i + 1 and i
      issue();         // stage i - 2, in the place of i + 2
      double2 xn[2];
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        // Chat of row i - 1 is stored with row i (zero with row 0, whose xn is not used)
        xn[c] = cfms(y[c], reinterpret_cast<const double2 *>(stage)[(KC + c) * 32 + lane], x[c]);
        if (i > 1) y[c] = yp[c * 32 - 128];
      }
      const double v = weighted_sums<KC>(stage, smem + ((i + 1) & 3) * kStage, ia, be, fine, sexp, x, lane);
      if (idx >= 0) *part = sum + v;
      part -= a.B * 8;
      yp -= 64;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        x[c] = xn[c];
        be[c] = bn[c];
      }
    }
  }
}

// One item: {system, state, first window | windows << 16, slot}; yb: the lane's place in the warp's
// sweep buffer, smem: the warp's stages.
__device__ __forceinline__ void limb_item(const LimbSweep &a, int4 item, int lane, double2 *yb, char *smem) {
  const int per = a.kc * 32;  // poles per window
  const int4 sy = a.sys[item.x];
  const int w0 = item.z & 0xffff, w1 = w0 + (item.z >> 16);
  const int b = item.y, idx = sum_index(lane);
  double *part = a.part + (((int64_t)item.w * a.nrows + sy.w) * a.B + b) * 8;
  for (int w = w0; w < w1; ++w) {
    const int p0 = w * per;
    if (a.kc == 2 && p0 + 32 < a.P) sweep_window<2>(a, item.x, sy.w, sy.z, p0, b, idx, part, w == w0, yb, smem, lane);
    else sweep_window<1>(a, item.x, sy.w, sy.z, p0, b, idx, part, w == w0, yb, smem, lane);
  }
}

// A window of one pole per lane by a CTA of four warps, for launches whose warps are too few to
// hide a row's chain (1800 cycles where one warp does all of it): one warp carries the two
// recurrences, 4 FP64 FMAs per row, the others form the right-hand sides and the sums of three
// rows at a time beside it, both through shared memory.  The arithmetic and the order of the
// sums are those of sweep_window.  role: 0 for the recurrences; ring: the warp's stages; rows: in
// those of the recurrences' warp, [2][3 rows][32].
constexpr int kRowsAhead = 3;
inline __device__ void sweep_window_split(const LimbSweep &a, int sysid, int64_t row0, int len, int p0, int b, int idx, double *part,
                                   bool first, double2 *yb, char *ring, double2 *rows, int role, int lane) {
  const int blk = p0 / kBlock, pk = p0 % kBlock + lane;
  const int64_t rec = row0 * a.nblk + (int64_t)blk * len;
  const char *inv = a.inv + ((row0 + sysid) * a.nblk + (int64_t)blk * (len + 1)) * kRec + pk * 16;
  const int chunks = (len + kRowsAhead - 1) / kRowsAhead;
  auto at = [&](int t, int c) { return rows + ((t & 1) * kRowsAhead + c) * 32 + lane; };
  if (role == 0) {
    const double2 zero = make_double2(0, 0);
    const char *f = a.fwd + rec * kRec + pk * 16;
    double2 v = zero, l[kRowsAhead], ln[kRowsAhead];
#pragma unroll
    for (int c = 0; c < kRowsAhead; ++c) l[c] = c < len ? __ldg(reinterpret_cast<const double2 *>(f + (int64_t)c * kRec)) : zero;
    for (int t = 0; t < chunks; ++t) {
#pragma unroll
      for (int c = 0; c < kRowsAhead; ++c) {
        const int i = kRowsAhead * (t + 1) + c;
        ln[c] = i < len ? __ldg(reinterpret_cast<const double2 *>(f + (int64_t)i * kRec)) : zero;
      }
      __syncthreads();  // the chunk's right-hand sides are there
#pragma unroll
      for (int c = 0; c < kRowsAhead; ++c) {
        const int i = kRowsAhead * t + c;
        if (i < len) {
          v = cfms(*at(t, c), l[c], v);
          yb[i * 64] = v;
        }
        l[c] = ln[c];
      }
    }
    // backward: x_i = y_i - Chat x_{i+1}, Chat of row i stored with row i + 1
    const char *g = a.bwd + rec * kBwd + pk * 16;
    double2 y[kRowsAhead], yn[kRowsAhead], h[kRowsAhead], hn[kRowsAhead];
    auto load = [&](int t, double2 (&yy)[kRowsAhead], double2 (&hh)[kRowsAhead]) {
#pragma unroll
      for (int c = 0; c < kRowsAhead; ++c) {
        const int i = len - 1 - kRowsAhead * t - c;
        yy[c] = i >= 0 ? yb[i * 64] : zero;
        hh[c] = i >= 0 && i + 1 < len ? __ldg(reinterpret_cast<const double2 *>(g + (int64_t)(i + 1) * kBwd)) : zero;
      }
    };
    load(0, y, h);
    v = zero;
    for (int t = 0; t < chunks; ++t) {
      load(t + 1, yn, hn);
#pragma unroll
      for (int c = 0; c < kRowsAhead; ++c) {
        v = t + c > 0 ? cfms(y[c], h[c], v) : y[c];
        *at(t, c) = v;
        y[c] = yn[c];
        h[c] = hn[c];
      }
      __syncthreads();  // the chunk's solutions are there
    }
    return;
  }
  const unsigned sm = (unsigned)__cvta_generic_to_shared(ring);
  const char *ia = ring + kInvAlpha;
  const int c0 = role - 1;
  // two stages per row (its own factors, and 1/s of the row after), the next row's being copied
  auto issue = [&](int i, int set) {
    if (i >= 0 && i < len) {
      const unsigned to = sm + 2 * set * kStage;
      copy_async<16>(to + lane * 16, inv + (int64_t)i * kRec);
      copy_async<16>(to + kStage + lane * 16, inv + (int64_t)(i + 1) * kRec);
    }
  };
  auto issue_inputs = [&](int i, int set) {
    issue(i, set);
    if (i < len) {
      const unsigned to = sm + 2 * set * kStage;
      const int64_t st = (row0 + i) * a.B + b;
      if (lane < 4) copy_async<16>(to + kSIn + lane * 16, a.dig + st * 4 + lane);
      else if (lane == 4) copy_async<4>(to + kSU, a.uexp + st);
    }
    copy_commit();
  };
  const int one[2] = {p0 + lane < a.P ? 1 << (28 - a.e0) : 0, 0};
  __syncwarp();  // every lane has read the stages of the window before
  copy_async<16>(sm + kInvAlpha + lane * 16, a.inv_alpha + p0 + lane);
  issue_inputs(c0, 0);
  for (int t = 0; t < chunks; ++t) {
    const int i = kRowsAhead * t + c0;
    issue_inputs(i + kRowsAhead, (t + 1) & 1);
    copy_wait<1>();
    __syncwarp();
    if (i < len) {
      double2 r[2], l[2];
      const char *stage = ring + 2 * (t & 1) * kStage;
      right_hand_sides<1>(stage, stage + kStage, ia, a.e0, one, lane, r, l);
      *at(t, c0) = r[0];
    }
    __syncthreads();
  }
  copy_wait<0>();
  const char *g = a.bwd + rec * kBwd;
  const int fine = min(a.e0 - __ldg(a.eblk + blk), 8), sexp = idx > 1 ? a.e0 - fine - 51 : -53;
  int be[2] = {0, 0}, bn = 0;
  auto issue_weights = [&](int i, int set) {
    issue(i, set);
    if (i >= 0) {
      copy_async<16>(sm + 2 * set * kStage + (64 + lane) * 16, g + (int64_t)i * kBwd + kRec + pk * 16);
      bn = __ldg(reinterpret_cast<const int *>(g + (int64_t)i * kBwd + kBE) + pk);
    }
    copy_commit();
  };
  issue_weights(len - 1 - c0, 0);
  for (int t = 0; t < chunks; ++t) {
    const int i = len - 1 - kRowsAhead * t - c0;
    be[0] = bn;
    issue_weights(i - kRowsAhead, (t + 1) & 1);
    double *p = part + (int64_t)i * a.B * 8 + (idx > 0 ? idx : 0);
    double sum = 0;
    if (!first && idx >= 0 && i >= 0) sum = *p;
    copy_wait<1>();
    __syncthreads();
    if (i >= 0) {
      const double2 x[2] = {*at(t, c0), make_double2(0, 0)};
      const char *stage = ring + 2 * (t & 1) * kStage;
      const double v = weighted_sums<1>(stage, stage + kStage, ia, be, fine, sexp, x, lane);
      if (idx >= 0) *p = sum + v;
    }
  }
  copy_wait<0>();
}

// One item by a CTA of four warps (kc 3); smem: the CTA's stages
__device__ __forceinline__ void limb_item_split(const LimbSweep &a, int4 item, int lane, int warp, int lead, double2 *yb,
                                                char *smem) {
  const int4 sy = a.sys[item.x];
  const int w0 = item.z & 0xffff, w1 = w0 + (item.z >> 16);
  const int b = item.y, idx = sum_index(lane);
  double *part = a.part + (((int64_t)item.w * a.nrows + sy.w) * a.B + b) * 8;
  for (int w = w0; w < w1; ++w)
    sweep_window_split(a, item.x, sy.w, sy.z, w * 32, b, idx, part, w == w0, yb, smem + warp * kSmemWarp,
                           reinterpret_cast<double2 *>(smem + lead * kSmemWarp), (warp - lead) & 3, lane);
}

}  // namespace limb_solve
}  // namespace rexi
