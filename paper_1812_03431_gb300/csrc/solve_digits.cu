// Banded shifted solves of whole batches with their two contractions on the tensor cores,
// exactly (paper Sec. 4.2, Sec. 5, Algorithm 1; binary64 delta solver).
//
// The systems, factors and recurrences are those of solve.cu: per (pole k, zonal order m,
// parity) forward  y_i = r_i - l y_{i-1},  r_i = delta0_n - g Phi0_n - e zeta0_{n-1} - f zeta0_{n+1},
// backward  w_i = y_i - Chat w_{i+1},  and the sums over k of bd w, bad w, zp w and zm w.
// Of the 36 FP64 FMAs per (state, pole, row), 8 belong to the two recurrences (6 here: see below);
// the other 28
// are contractions with factors that no state changes: r over the row's four inputs, and the
// four weighted sums over the poles.  GB300's FP64 unit issues one warp instruction per 64
// cycles and scheduler, so the contractions are taken off it:
//   - every operand is written as a 64-bit fixed-point number relative to the largest of its
//     group (a power of two per group), cut into 8-bit balanced digits -128..127, which fp16
//     holds exactly (weights: seven digits, 55 bits and sign; inputs, couplings and w: eight);
//   - digit products are summed by mma.sync m16n8k16 with FP32 accumulators that start at
//     1.5 2^23, so that an accumulator's low bits are the integer sum: every partial sum stays
//     below 2^22 and nothing is rounded (digit pairs i + j <= 7 are taken: what is left out is
//     below 2^-60 of the largest product);
//   - the eight sums of equal weight are put together in a 64-bit integer, which is rounded to
//     binary64 once, on the integer pipe.
// The recurrences take 6: with y_i = p_i y~_i, w_i = p_i w~_i and unit complex p_i such that
// Chat_i p_{i+1} / p_i = |Chat_i|, the backward one multiplies by a real number.  1/p_i goes into the
// couplings and p_i into the weights before they are cut into digits (p is kept to 2^-60), and l
// turns into l p_{i-1} / p_i; nothing else changes.
// The sums are therefore exact up to the 2^-55 rounding of a group's smaller operands and one
// rounding each; the recurrences run in binary64 as before.  The pole sums of an item's
// windows are added in binary64 in window order, and the items' sums in a fixed order, so
// results are bit-reproducible.
//
// Why mma.sync and not tcgen05: the operand fragments of m16n8k16 are exactly what the lanes
// hold (a lane's state and pole are a fragment's column and k pair), so digits go from
// registers into the tensor core and sums come back to the lane that needs them, with no
// shared memory, no descriptors and no waiting.  The work is 40 MMAs per warp and row at 8.8
// cycles each, about a third of the FP64 time beside them, so their rate does not bound it.
//
// Measured on GB300 (solve and the sum of the slots, against the pole-slot solve and its
// reduction): T341, 535 poles, 16 states 8.3 / 30.0 ms; T127, 535 poles, 64 states 4.6 / 17.0;
// T85, 215 poles, 5 states 0.17 / 0.62.  The FP64 unit takes 7 instructions per state, pole and
// row at 64 cycles, one of them the running sum's addition, at 16 warps per SM (12 warps: 10.2 ms
// at T341); with the complex Chat it was 9, 86 % busy, and 9.1 ms.  Rows staged ahead in shared
// memory with asynchronous copies took it there from 78 % (9.9 ms with prefetches into the caches).
//
// A warp takes 8 states x 8 poles (lane: state lane / 4, poles 2 (lane % 4) and the next) of one
// (m, parity) system, window by window of 8 poles, over all rows.  Real and imaginary rows of
// a product take their operand as (re, -im) and (im, re): the couplings' products through two
// forms of the inputs' digits, the weighted sums by keeping the real and the imaginary digits
// of a pole pair in words of their own, which the two kinds of row load in opposite order.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "digit_sweep.h"
#include "rexi_internal.h"

namespace rexi {

using namespace fixed;
using namespace digit_solve;

namespace {

// ---- plan time: the factors as digits ---------------------------------------------------------
struct SetupArgs {
  const double2 *fac;  // [F_NCOMP][nrows][P]
  const int4 *sys;
  char *fwd, *bwd;     // records, system by system: [window][row of the system]
  int *vexp;           // [nrows][4]: the scale of each input (0 for delta)
  int *bad;            // set when the factors are not finite or too unlike in scale
  int P, nwin, kmid;
  int64_t nrows;
};

// Unit complex numbers as pairs of integers in units of 2^-62.  v q, rounded:
__device__ __forceinline__ long long times(long long v, long long q) {
  const unsigned long long l = (unsigned long long)v * (unsigned long long)q;
  return (long long)((unsigned long long)__mul64hi(v, q) << 2 | l >> 62) + (long long)(l >> 61 & 1);
}
__device__ __forceinline__ longlong2 times(longlong2 v, longlong2 q) {
  return longlong2{times(v.x, q.x) - times(v.y, q.y), times(v.x, q.y) + times(v.y, q.x)};
}
__device__ __forceinline__ longlong2 conj(longlong2 q) { return longlong2{q.x, -q.y}; }

// c / |c| (1 where c is zero): in binary64, then its phase and length corrected to first order
__device__ longlong2 unit_of(double2 c) {
  const int e = max(bexp(c.x), bexp(c.y));
  if (e == 0 || e > 2040) return longlong2{1ll << 62, 0};
  const double s = __longlong_as_double((long long)(2046 - e) << 52);
  const double x = c.x * s, y = c.y * s, r = rsqrt(x * x + y * y), ux = x * r, uy = y * r;
  const double w = x * uy, phase = (fma(y, ux, -w) + fma(-x, uy, w)) * r;
  const double big = fmax(fabs(ux), fabs(uy)), small = fmin(fabs(ux), fabs(uy)), b2 = big * big, s2 = small * small;
  const double half = 0.5 * (((1.0 - b2) - s2) - (fma(big, big, -b2) + fma(small, small, -s2)));
  auto q62 = [](double hi, double lo) {
    return __double2ll_rn(hi * 4611686018427387904.0) + __double2ll_rn(lo * 4611686018427387904.0);
  };
  return longlong2{q62(ux, ux * half - uy * phase), q62(uy, uy * half + ux * phase)};
}

// p of every row and u = Chat / |Chat| of the row before, one thread per (pole, system): p_0 = 1,
// p_{i+1} = p_i / u_i.  They go where the pole's coupling digits will be, which the thread that
// reads them writes.
__global__ void digit_phase_kernel(SetupArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int4 sy = a.sys[blockIdx.y];
  if (k >= a.P) return;
  char *to = a.fwd + ((int64_t)sy.w * a.nwin + (int64_t)(k / kWin) * sy.z) * kFwdRec + (k % kWin) * 64;
  longlong2 p{1ll << 62, 0}, u = p;
  for (int i = 0; i < sy.z; ++i, to += kFwdRec) {
    reinterpret_cast<longlong2 *>(to)[0] = p;
    reinterpret_cast<longlong2 *>(to)[1] = u;
    if (i + 1 == sy.z) break;
    u = unit_of(a.fac[((int64_t)F_C * a.nrows + sy.w + i) * a.P + k]);
    p = times(p, conj(u));
  }
}

// v's parts as to_fixed gives them, E the exponent (biased) of their group's leading bit
__device__ __forceinline__ longlong2 fixed_of(double2 v, int E) {
  return longlong2{to_fixed(v.x, E - bexp(v.x)), to_fixed(v.y, E - bexp(v.y))};
}
__device__ __forceinline__ bool reaches_62(longlong2 v) {
  return v.x >= 1ll << 62 || v.x <= -(1ll << 62) || v.y >= 1ll << 62 || v.y <= -(1ll << 62);
}
__device__ __forceinline__ longlong2 halve(longlong2 v) { return longlong2{(v.x + 1) >> 1, (v.y + 1) >> 1}; }

__global__ void digit_factor_kernel(SetupArgs a) {
  const int4 sy = a.sys[blockIdx.y];
  const int len = sy.z;
  const int64_t row0 = sy.w;
  const int64_t total = (int64_t)len * a.nwin * kWin;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = t < total;  // whole groups of 8 threads
  const int p8 = (int)(t & 7);
  const int w = (int)((t >> 3) % a.nwin), i = (int)((t >> 3) / a.nwin);
  const int k = w * kWin + p8;
  const int64_t row = row0 + i;
  const double2 zero = make_double2(0, 0);
  auto get = [&](int comp, int kk) { return live && kk < a.P ? a.fac[((int64_t)comp * a.nrows + row) * a.P + kk] : zero; };
  auto neg = [](double2 v) { return make_double2(-v.x, -v.y); };
  auto emax = [](double2 v) { return max(bexp(v.x), bexp(v.y)); };
  const int64_t rec = row0 * a.nwin + (int64_t)w * len + i;
  char *fr = a.fwd + rec * kFwdRec, *br = a.bwd + rec * kBwdRec;
  bool bad = false;

  // couplings of the four inputs delta, Phi, zeta_{n-1}, zeta_{n+1}
  double2 v[4] = {live && k < a.P ? make_double2(1.0, 0.0) : zero, neg(get(F_G, k)), neg(get(F_E, k)), neg(get(F_F, k))};
  int ve[4], E = 0;
  const int comp[4] = {0, F_G, F_E, F_F};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int mid = j == 0 ? 1023 : emax(get(comp[j], a.kmid));
    ve[j] = mid == 0 ? 0 : mid - 1023;
    const int e = emax(v[j]);
    if (e == 0x7ff) bad = true;
    if (e) E = max(E, e - ve[j]);
  }
  // rotated by 1/p, which can take a part of one past the leading bit
  const longlong2 one{1ll << 62, 0}, *pu = reinterpret_cast<const longlong2 *>(fr + p8 * 64);
  const longlong2 p = live && k < a.P ? pu[0] : one, u = live && k < a.P ? pu[1] : one;
  longlong2 fv[4];
  bool past = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int e = emax(v[j]);
    if (e && E - (e - ve[j]) > kMaxSpread) bad = true;
    fv[j] = times(fixed_of(v[j], E + ve[j]), conj(p));
    past |= reaches_62(fv[j]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (past) fv[j] = halve(fv[j]);
    if (live) reinterpret_cast<uint4 *>(fr)[p8 * 4 + j] = packed_digits(fv[j].x, fv[j].y);
  }
  if (live) {
    // l p_{i-1} / p_i and |Chat| of the row before
    const double2 l = get(F_L, k), c = i > 0 && k < a.P ? a.fac[((int64_t)F_C * a.nrows + row - 1) * a.P + k] : zero;
    const longlong2 fl = times(fixed_of(l, emax(l)), u), fc = times(fixed_of(c, emax(c)), conj(u));
    const int le = emax(l) - 1023 - 61;
    reinterpret_cast<double2 *>(fr + kLOff)[p8] = make_double2(fixed_to_double(fl.x, le), fixed_to_double(fl.y, le));
    reinterpret_cast<int *>(fr + kEOff)[p8] = E - 1023 + past;
    reinterpret_cast<double *>(br + kCOff)[p8] = fixed_to_double(fc.x, emax(c) - 1023 - 61);
    if (w == 0 && p8 < 4) a.vexp[row * 4 + p8] = ve[p8];
  }
  // the four weights, scaled by the largest of the window's eight poles
  const int wc[4] = {F_BD, F_BAD, F_ZP, F_ZM};
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const double2 x = get(wc[s], k);
    int m = emax(x);
    if (m == 0x7ff) bad = true;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    longlong2 f = times(fixed_of(x, m), p);
    int over = reaches_62(f);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) over |= __shfl_xor_sync(0xffffffffu, over, o);
    if (over) {
      f = halve(f);
      ++m;
    }
    // seven digits (rounded to the nearest multiple of the eighth's weight), the real parts of
    // poles 2 q and 2 q + 1 by the even thread, their imaginary parts by the odd one
    const long long re = (f.x + 128) & ~255ll, im = (f.y + 128) & ~255ll;
    const long long other = __shfl_xor_sync(0xffffffffu, p8 & 1 ? re : im, 1);
    uint4 d = packed_digits(p8 & 1 ? other : re, p8 & 1 ? im : other);
    d.w = (d.w & 0xffffu) | (unsigned)(m - 1023) << 16;  // the exponent in the eighth digits' place
    if (live) reinterpret_cast<uint4 *>(br)[s * kWin + p8] = d;
  }
  const double2 l = get(F_L, k), c = get(F_C, k);
  if (emax(l) == 0x7ff || emax(c) > 2040) bad = true;  // unit_of goes up to there
  if (bad) atomicOr(a.bad, 1);
}

// ---- per step: the row inputs as digits ---------------------------------------------------------
struct StateArgs {
  const double2 *sin;  // [3][nspec][B]
  const int4 *sys;
  const int *vexp;
  char *dig;           // [nrows][tiles] records
  int *uexp;           // [nrows][tiles][8]
  unsigned *counter;   // the sweep's next item, set to zero here (null: not)
  int64_t nspec;
  int B, tiles, N;
};

__global__ void digit_state_kernel(StateArgs a) {
  if (a.counter && blockIdx.x + blockIdx.y + threadIdx.x == 0) *a.counter = 0;
  const int4 sy = a.sys[blockIdx.y];
  const int m = sy.x, n0 = sy.y, len = sy.z;
  const int lane = threadIdx.x & 31, s = lane >> 2, q = lane & 3;
  const int wid = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (wid >= len * a.tiles) return;  // whole warps
  const int i = wid / a.tiles, tile = wid - i * a.tiles;
  const int64_t row = sy.w + i;
  const int n = n0 + 2 * i, b = tile * kTile + s, nmin = m > 1 ? m : 1;
  const int nn = q < 2 ? n : (q == 2 ? n - 1 : n + 1);
  const int field = q == 0 ? 2 : (q == 1 ? 0 : 1);
  double2 x = make_double2(0, 0);
  if (b < a.B && nn >= nmin && nn <= a.N) {
    const int64_t ix = (int64_t)m * (2 * a.N + 3 - m) / 2 + (nn - m);
    x = __ldg(a.sin + ((int64_t)field * a.nspec + ix) * a.B + b);
  }
  const int v = a.vexp[row * 4 + q];
  const int er = bexp(x.x), ei = bexp(x.y), e = max(er, ei);
  int U = e ? e + v : -(1 << 24), nf = e == 0x7ff;
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    U = max(U, __shfl_xor_sync(0xffffffffu, U, o));
    nf |= __shfl_xor_sync(0xffffffffu, nf, o);
  }
  unsigned d[8];
  digits(nf ? 0 : to_fixed(x.x, U - (er + v)), nf ? 0 : to_fixed(x.y, U - (ei + v)), d);
  uint4 *o = reinterpret_cast<uint4 *>(a.dig + (row * a.tiles + tile) * kStateRec + lane * 32);
  o[0] = make_uint4(d[0], d[1], d[2], d[3]);
  o[1] = make_uint4(d[4], d[5], d[6], d[7]);
  if (q == 0) a.uexp[(row * a.tiles + tile) * kTile + s] = nf ? kNotFinite : (U < -(1 << 23) ? 0 : U - 1023);
}

// ---- per step: the sweeps (digit_sweep.h) ---------------------------------------------------------
template <int CTAS>
__global__ void __launch_bounds__(128, CTAS) solve_digits_kernel(DigitSweep a) {
  const int lane = threadIdx.x & 31;
  const int wslot = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  double2 *yb = a.ybuf + (int64_t)wslot * a.lmax * 64 + lane;
  extern __shared__ __align__(16) char stages[];
  char *smem = stages + (threadIdx.x >> 5) * kSmemWarp;
  for (;;) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(a.counter, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= (unsigned)a.nitems) break;
    digit_item(a, a.items[it], lane, yb, smem);
  }
}

// ---- per step: the items' sums, the pole-independent terms, Re at m = 0 --------------------------
struct FinishArgs {
  const double *part;  // per (slot, row, tile): `unit` values, [4 streams][re, im][states] or [states][4 streams][re, im]
  const double2 *sin, *w;
  double2 *sout;
  const uint8_t *rflags;
  const int32_t *m_of;
  const int4 *sys;
  double2 sphi;
  int64_t nspec, nrows;
  const double *scale;  // limbs: per row the sums' real factors at 3..5 (see solve_limbs.cu), else null
  int B, tile, tiles, unit, sstr, pstr, slots, N;
};

// SPLIT threads per output, each over every SPLIT-th slot: one where the outputs fill the chip (HBM
// bounds it: T341 x 16 with 8 slots 0.123 to 0.131 ms, 0.137 without four slots' loads in flight), four where
// they are few and the slots many (T85 x 5 with 27 20 / 31 us, T42 x 8 with 19 12 / 16 us).
// BY_STATE: sin and sout are [B][3][nspec], else [3][nspec][B] (a kernel of its own: chosen at run time it
// cost every step 0.7 us at T170 x 1).
template <int SPLIT, bool BY_STATE>
__global__ void digit_finish_kernel(FinishArgs a) {
  const int64_t total = 3 * a.nspec * a.B, slot = a.nrows * a.tiles * a.unit, step = slot * SPLIT;
  const int first = threadIdx.x % SPLIT;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / SPLIT; t < total;
       t += (int64_t)gridDim.x * blockDim.x / SPLIT) {
    const int64_t per = BY_STATE ? 3 * a.nspec : a.B;
    const int b = (int)(BY_STATE ? t / per : t % per);
    const int64_t fi = BY_STATE ? t % per : t / per;
    const int f = (int)(fi / a.nspec);
    const int64_t ix = fi - (int64_t)f * a.nspec;
    const uint8_t fl = a.rflags[fi];
    double2 acc = make_double2(0, 0);
    if (!(fl & 2)) {
      const int m = a.m_of[ix];
      if (fl & 1) {
        const int n = m + (int)(ix - (int64_t)m * (2 * a.N + 3 - m) / 2);
        auto add = [&](int nn, int stream) {  // the slots' sums of the row at degree nn, in slot order
          const int4 sy = a.sys[2 * m + ((nn - m) & 1)];
          const int64_t row = sy.w + (nn - sy.y) / 2;
          const double *p = a.part + (row * a.tiles + b / a.tile) * a.unit + b % a.tile + stream * a.sstr + first * slot;
          const double c = a.scale && stream > 0 ? a.scale[row * 6 + 2 + stream] : 1.0;
          int s = first;
          for (; s + 3 * SPLIT < a.slots; s += 4 * SPLIT) {  // loads of four slots in flight
            double2 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k, p += step) v[k] = make_double2(p[0], p[a.pstr]);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc = make_double2(fma(c, v[k].x, acc.x), fma(c, v[k].y, acc.y));
          }
          for (; s < a.slots; s += SPLIT, p += step) acc = make_double2(fma(c, p[0], acc.x), fma(c, p[a.pstr], acc.y));
        };
        const int nmin = m > 1 ? m : 1;
        if (f != 1) add(n, f == 2 ? 0 : 1);
        else {
          if (n - 1 >= nmin) add(n - 1, 2);
          if (n + 1 <= a.N) add(n + 1, 3);
        }
#pragma unroll
        for (int o = 1; o < SPLIT; o <<= 1) {  // an output's threads are neighbours and take the same branches
          const unsigned group = ((1u << SPLIT) - 1) << (threadIdx.x & 31 & -SPLIT);
          const double re = __shfl_xor_sync(group, acc.x, o), im = __shfl_xor_sync(group, acc.y, o);
          acc = make_double2(acc.x + re, acc.y + im);
        }
      }
      const double2 x0 = a.sin[t];
      if (f == 0) acc = cfma(acc, a.sphi, x0);
      else if (f == 1) acc = cfma(acc, a.w[ix], x0);
      if (m == 0) acc.y = 0.0;
    }
    if (first == 0) a.sout[t] = acc;
  }
}

// resident CTAs per SM: 16 warps at 128 registers
constexpr int kCtas = 4;

// states per tile and poles per window of this plan's windowed solve
int tile_of(const Plan &pl) { return pl.limbs ? 1 : kTile; }
int tiles_of(const Plan &pl, int B) { return (B + tile_of(pl) - 1) / tile_of(pl); }
int windows_of(const Plan &pl, int B, int kc) {
  const int w = pl.limbs ? limb_window(kc) : kWin;
  return (pl.P + w - 1) / w;
}

}  // namespace

void free_digit_factors(DigitFactors &D) {
  if (D.fwd) cudaFree(D.fwd);  // the others lie behind it
  D = DigitFactors{};
}

size_t digit_factor_bytes(const Plan &pl) {
  if (pl.limbs) return limb_factor_bytes(pl);
  return (size_t)pl.nrows * ((pl.P + kWin - 1) / kWin) * (kFwdRec + kBwdRec) + (size_t)pl.nrows * 4 * sizeof(int);
}

namespace {
cudaError_t launch_digit_factors(Plan &pl, const double2 *fac, DigitFactors &D, int *bad) {
  const int nwin = (pl.P + kWin - 1) / kWin;
  const size_t nrec = (size_t)pl.nrows * nwin;
  D.bwd = D.fwd + nrec * kFwdRec;
  D.vexp = reinterpret_cast<int *>(D.bwd + nrec * kBwdRec);
  SetupArgs a;
  a.fac = fac;
  a.sys = pl.sys_dev;
  a.fwd = D.fwd;
  a.bwd = D.bwd;
  a.vexp = D.vexp;
  a.bad = bad;
  a.P = pl.P;
  a.nwin = nwin;
  a.kmid = (int)(std::min_element(pl.alpha.begin(), pl.alpha.end(),
                                  [](const cplx &x, const cplx &y) { return std::abs(x) < std::abs(y); }) -
                 pl.alpha.begin());
  a.nrows = pl.nrows;
  const int64_t most = (int64_t)pl.lmax * nwin * kWin;
  digit_phase_kernel<<<dim3((unsigned)((pl.P + 63) / 64), (unsigned)pl.sys.size()), 64>>>(a);
  digit_factor_kernel<<<dim3((unsigned)((most + 255) / 256), (unsigned)pl.sys.size()), 256>>>(a);
  return cudaGetLastError();
}
}  // namespace

// The factor set as digits or limbs (pl.limbs), from the binary64 factors `fac`.  D stays empty
// (and the other solve kernels serve the plan) where the device memory does not suffice, or
// where a factor is not finite or a pole's couplings differ in scale by more than the
// fixed-point forms cover.
cudaError_t build_digit_factors(Plan &pl, bool adjoint, const double2 *fac, DigitFactors &D) {
  D = DigitFactors{};
  if (pl.nrows == 0 || (pl.P + kWin - 1) / kWin > 0x7fff || pl.sys.size() > 0xffff) return cudaSuccess;
  // one allocation, the flag at its end; the read of the flag waits for the factors
  const size_t bytes = digit_factor_bytes(pl);
  int hbad = 0;
  cudaError_t e = cudaMalloc(&D.fwd, bytes + sizeof(int));
  int *bad = reinterpret_cast<int *>(D.fwd + bytes);
  if (e != cudaSuccess) D.fwd = nullptr;
  if (e == cudaSuccess) e = cudaMemsetAsync(bad, 0, sizeof(int), 0);
  if (e == cudaSuccess) e = pl.limbs ? launch_limb_factors(pl, adjoint, fac, D, bad) : launch_digit_factors(pl, fac, D, bad);
  if (e == cudaSuccess) e = cudaMemcpy(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess || hbad) free_digit_factors(D);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return cudaSuccess;
  }
  return e;
}

size_t digit_state_bytes(const Plan &pl, int B) {
  if (pl.limbs) return limb_state_bytes(pl, B);
  return (size_t)pl.nrows * tiles_of(pl, B) * (kStateRec + kTile * sizeof(int));
}

// partial sums of one slot
size_t digit_slot_bytes(const Plan &pl, int B) {
  return (size_t)pl.nrows * (pl.limbs ? B : tiles_of(pl, B) * kTile) * 8 * sizeof(double);
}

// The items of one plan's batch: `slots` per (system, tile), each over its share of the windows
// (0: enough that the longest item's rows x windows are at most `longest`), capped by the
// partial-sum buffer.  False where the buffer holds no slot.
bool digit_items(const Plan &pl, int B, int slots, double longest, DigitLayout &L, std::vector<DigitItem> &items) {
  const int tiles = tiles_of(pl, B), nwin = windows_of(pl, B, L.kc);
  const int cap = (int)std::min<size_t>((size_t)nwin, pl.partial_elems * sizeof(double2) / digit_slot_bytes(pl, B));
  if (cap < 1) return false;
  int G = slots;
  if (G <= 0) {
    G = 1;
    while (G < nwin && (double)pl.lmax * ((nwin + G - 1) / G) > longest) ++G;
  }
  G = std::max(1, std::min(G, cap));
  for (int s = 0; s < (int)pl.sys.size(); ++s) {
    if (pl.sys[s].len == 0) continue;
    for (int g = 0; g < G; ++g) {
      const int w0 = (int)((int64_t)nwin * g / G), w1 = (int)((int64_t)nwin * (g + 1) / G);
      for (int t = 0; t < tiles; ++t)
        items.push_back(DigitItem{make_int4(s, t, w0 | ((w1 - w0) << 16), g), (int64_t)pl.sys[s].len * (w1 - w0)});
    }
  }
  L.slots = G;
  return true;
}

// rows x windows x tiles of a batch
int64_t digit_work(const Plan &pl, int B, int kc) {
  return pl.nrows * windows_of(pl, B, kc) * tiles_of(pl, B);
}

// Work items (system, tile, windows, slot) for batch B, longest first.  slots: items per
// (system, tile), each over its share of the windows; 0: enough that the longest item is at
// most half a resident warp's share of the work, capped by the partial-sum buffer.  For limbs
// slots carries 65536 x the packing (1 or 2 poles per lane; 3: one, by a CTA per window; 0: the
// default).  A CTA's warps share a window's rows where the windows are fewer than 22 per SM, 5.5 per
// resident CTA (its barriers cost more than the shorter chains give beyond that): T63 x 1 with 71
// poles 0.038 against 0.056 ms for one warp, with 279 poles (7.6 windows per SM) 0.047 / 0.068; T127 x
// 1 with 151 poles (8.4) 0.078 / 0.134, T255 x 1 (17) 0.226 / 0.328; T127 x 1 with 535 poles (29) 0.208 /
// 0.183, T63 x 4 with 279 (30) 0.119 / 0.101.  Otherwise one pole per lane halves a warp's chain of
// FP64 FMAs per row at 0.7 of the whole row's instructions, which pays where items of two are
// fewer than 1.6 per resident warp (26 per SM): T170 x 1 with 535 poles 0.266 / 0.360 ms (20 per SM);
// T128 x 1 with 1047 poles 0.293 / 0.288 (29), T341 x 1 1.14 / 1.09 (40).
rexi_status build_digit_layout(Plan &pl, int B, int slots, DigitLayout &L) {
  L = DigitLayout{};
  if (pl.nrows == 0) return REXI_OK;  // not available
  if (pl.limbs) {
    L.kc = slots >> 16;
    auto windows = [&](int kc) { return (int64_t)pl.sys.size() * windows_of(pl, B, kc) * tiles_of(pl, B); };
    if (L.kc == 0) L.kc = windows(3) < 22 * (int64_t)pl.num_sms ? 3 : windows(2) < 26 * (int64_t)pl.num_sms ? 1 : 2;
    if (limb_configure(L.kc) != cudaSuccess) {
      cudaGetLastError();
      return REXI_OK;
    }
  }
  std::vector<DigitItem> keyed;
  const double teams = (double)kCtas * pl.num_sms * (L.kc == 3 ? 1 : 4);
  if (!digit_items(pl, B, slots & 0xffff, 0.5 * digit_work(pl, B, L.kc) / teams, L, keyed))
    return REXI_OK;
  std::stable_sort(keyed.begin(), keyed.end(), [](const DigitItem &x, const DigitItem &y) { return x.work > y.work; });
  std::vector<int4> items;
  for (const DigitItem &k : keyed) items.push_back(k.it);
  cudaError_t e = cudaMalloc(&L.items_dev, std::max<size_t>(1, items.size()) * sizeof(int4));
  if (e == cudaSuccess) e = cudaMemcpy(L.items_dev, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    free_digit_layout(L);
    set_error(std::string("digit work list: ") + cudaGetErrorString(e));
    return REXI_ENOMEM;
  }
  L.nitems = (int)items.size();
  return REXI_OK;
}

void free_digit_layout(DigitLayout &L) {
  if (L.items_dev) cudaFree(L.items_dev);
  L = DigitLayout{};
}

// the batch's inputs in fixed point, and *counter = 0.  by_state (limbs only): sin is [B][3][nspec], as
// rexi_step takes it, else [3][nspec][B].
cudaError_t launch_digit_state(Plan &pl, bool adjoint, const double2 *sin, bool by_state, int B, unsigned *counter,
                               cudaStream_t st) {
  if (pl.limbs) return launch_limb_state(pl, adjoint, sin, by_state, B, counter, st);
  const int tiles = tiles_of(pl, B);
  StateArgs s;
  s.sin = sin;
  s.sys = pl.sys_dev;
  s.vexp = (adjoint ? pl.dig_adj : pl.dig_fwd).vexp;
  s.dig = pl.dig_state;
  s.uexp = reinterpret_cast<int *>(pl.dig_state + (size_t)pl.nrows * tiles * kStateRec);
  s.counter = counter;
  s.nspec = pl.nspec;
  s.B = B;
  s.tiles = tiles;
  s.N = pl.N;
  digit_state_kernel<<<dim3((unsigned)((pl.lmax * tiles + 7) / 8), (unsigned)pl.sys.size()), 256, 0, st>>>(s);
  return cudaGetLastError();
}

DigitSweep digit_sweep(Plan &pl, const DigitLayout &L, bool adjoint, int B) {
  const DigitFactors &D = adjoint ? pl.dig_adj : pl.dig_fwd;
  const int tiles = tiles_of(pl, B);
  DigitSweep a;
  a.fwd = D.fwd;
  a.bwd = D.bwd;
  a.dig = pl.dig_state;
  a.uexp = reinterpret_cast<const int *>(pl.dig_state + (size_t)pl.nrows * tiles * kStateRec);
  a.sys = pl.sys_dev;
  a.items = L.items_dev;
  a.part = reinterpret_cast<double *>(pl.partial);
  a.ybuf = pl.yscratch;
  a.counter = pl.counter;
  a.nrows = pl.nrows;
  a.nitems = L.nitems;
  a.tiles = tiles;
  a.nwin = windows_of(pl, B, 2);
  a.lmax = pl.lmax;
  return a;
}

cudaError_t launch_solve_digits(Plan &pl, const DigitLayout &L, bool adjoint, const double2 *sin, bool by_state, int B,
                                cudaStream_t st) {
  cudaError_t e = launch_digit_state(pl, adjoint, sin, by_state, B, pl.counter, st);
  if (e != cudaSuccess) return e;
  if (pl.limbs) return launch_solve_limbs(pl, L, adjoint, B, st);
  const int ctas = std::min(pl.num_sms * kCtas, (L.nitems + 3) / 4);
  solve_digits_kernel<kCtas><<<(unsigned)std::max(1, ctas), 128, 4 * kSmemWarp, st>>>(digit_sweep(pl, L, adjoint, B));
  return cudaGetLastError();
}

cudaError_t launch_finish_digits(Plan &pl, const DigitLayout &L, bool adjoint, const double2 *sin, double2 *sout,
                                 bool by_state, int B, cudaStream_t st) {
  FinishArgs f;
  f.part = reinterpret_cast<const double *>(pl.partial);
  f.sin = sin;
  f.w = adjoint ? pl.w_adj : pl.w_fwd;
  f.sout = sout;
  f.rflags = pl.rflags_dev;
  f.m_of = pl.m_of_dev;
  f.sys = pl.sys_dev;
  f.sphi = adjoint ? pl.sphi_adj : pl.sphi_fwd;
  f.nspec = pl.nspec;
  f.nrows = pl.nrows;
  f.B = B;
  f.tile = pl.limbs ? 1 : kTile;
  f.tiles = pl.limbs ? B : tiles_of(pl, B);
  f.unit = 8 * f.tile;
  f.sstr = 2 * f.tile;
  f.pstr = f.tile;
  f.slots = L.slots;
  f.scale = (adjoint ? pl.dig_adj : pl.dig_fwd).scale;
  f.N = pl.N;
  const int64_t total = 3 * pl.nspec * B;
  const int split = L.slots >= 8 && total <= 2048 * (int64_t)pl.num_sms ? 4 : 1;
  auto k = by_state ? (split > 1 ? digit_finish_kernel<4, true> : digit_finish_kernel<1, true>)
                    : (split > 1 ? digit_finish_kernel<4, false> : digit_finish_kernel<1, false>);
  k<<<(unsigned)std::min<int64_t>((total * split + 255) / 256, 1 << 20), 256, 0, st>>>(f);
  return cudaGetLastError();
}

}  // namespace rexi
