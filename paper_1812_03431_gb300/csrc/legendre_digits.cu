// Legendre transforms of the FP64 form (paper Sec. 3) as exact fixed-point products on the tensor
// cores.  The sums are those of legendre.cu; per zonal order m they are contractions of the
// tables Pbar and H with the folded Fourier data (analysis) or the spectral coefficients
// (synthesis), which as FP64 FMAs (10 per degree, latitude pair and state) kept the FP64 unit
// busy at 1/64 of the FP32 rate: 4.4 and 4.1 ms at T341 with 16 states.
//
// As in solve_digits.cu, each operand is a 62-bit fixed-point number relative to the largest of
// its group -- here a table row's or a data column's 64 values along the contraction -- in eight
// balanced 8-bit digits held as fp16; mma.sync m16n8k16 sums digit products in FP32
// accumulators, exactly: over a group an accumulator stays below 2^23.  The eight sums of equal
// weight (digit pairs i + j <= 7: what is left out is below 2^-60 of the largest product) make
// one 64-bit integer, rounded once to binary64 and added to the running sum.  So each output
// carries one rounding per 64 terms in place of 64.
//
// A CTA of eight warps takes one zonal order and four states (blockIdx: states, rows, m; the states'
// CTAs of an order side by side, so that its tables come from HBM once); it cuts a group's data
// into digits in shared memory, each warp then forms the five products of a row tile of 16
// degrees or latitudes.  A tile of the product's columns is one field of the four states (re,
// im), so that a lane ends up with all fields of one state and combines them in registers.  With
// one state that tile would be three quarters padding: there the three fields share one, and two
// products (P and H times all fields) do for the five.  Small batches take that form state by
// state (one_state below).  Tables: 8 B per value as in the FP64 form,
// in fragment order.  Everything is copied ahead with cp.async: a warp's next table fragment, also
// across products and barriers, and the next group's inputs while the products run.
//
// Measured on GB300 (analysis, synthesis; against the FP64 kernels): T341 x 16 0.84, 0.71 / 4.37, 4.07
// ms; T255 x 8 0.212, 0.197 / 1.01, 0.86; T639 x 1 0.52, 0.48; T170 x 1 0.031, 0.033 / 0.114, 0.169;
// T63 x 1 0.012, 0.014 / 0.037, 0.065.  Without the copies ahead and the shared tile: 0.92, 0.79;
// 0.234, 0.204; T170 x 1 0.058, 0.076; T63 x 1 0.020, 0.027.  At T255 x 8 the tensor pipe is 35 %, the
// issue slots 45 % busy (ncu): four warps per scheduler, which wait for each other at the groups'
// barriers and within the chains of a product; registers allow no more warps.  Fewer instructions
// (sums read off the accumulators' bits per 32 terms) gave nothing.  tcgen05 would keep the accumulators
// out of the registers; it is not built (both operands are in shared memory already, but tables
// would have to be expanded to fp16 there).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "fixed.h"
#include "mma_digits.h"
#include "rexi_internal.h"

namespace rexi {

using namespace fixed;

namespace {

constexpr int kGroup = 64;       // contraction length of a group
constexpr int kWarps = 8;
constexpr int kFrag = 2048;      // bytes of a 16 x 16 table fragment
constexpr int kTileDig = (kGroup / 16) * 2 * 2 * 512;  // digits of one column tile
// Shared memory: a group's inputs as they come (two halves -- hemispheres, or degrees of either
// class -- of 64 x 12 complex numbers; even and odd places apart and 13 to a row, so that lanes
// reading every second place meet no bank twice), their zeta/delta scale (synthesis), their digits,
// the columns' exponents, and per warp two table fragments.
constexpr int kPitch = 13;
constexpr int kZd = 2 * 2 * (kGroup / 2) * kPitch * 16, kDig = kZd + 2 * kGroup * 8, kExp = kDig + 6 * kTileDig;
constexpr int kRing = kExp + 48 * 4, kSmem = kRing + kWarps * 2 * kFrag;
static_assert(2 * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");

// The synthesis' groups run over degrees, along which H grows like n and spectra fall: tables are
// divided and data multiplied by the power of two below n + 1, or the products of a smooth field's
// few large coefficients would be small against the group's largest product.
// Without it the wind of one large zonal coefficient among small ones was several roundings off the sum
// of its parts; it takes a hundredth of the synthesis' time.
__device__ __forceinline__ double degree_scale(int n) {
  return __longlong_as_double((long long)(1023 + 31 - __clz(n + 1)) << 52);
}

struct TabArgs {
  const double *tab[2];          // Pbar, H: [nspec][J]
  uint4 *dig;                    // [fragment][P, H][4 registers][32 lanes]
  int *exps;                     // [group][tile][P, H][16 rows]
  const int4 *sys;               // per 2 m + class: {rows, first fragment, first exponent group, 0}
  int N, J, synthesis;
};

// One warp per (m, class, row tile, group, table): analysis tiles are degrees against latitudes,
// synthesis tiles latitudes against degrees.
__global__ void __launch_bounds__(32) legendre_digits_setup(TabArgs a) {
  const int mc = blockIdx.y, m = mc >> 1, cls = mc & 1;
  const int4 sy = a.sys[mc];
  const int rows = a.synthesis ? a.J : sy.x, len = a.synthesis ? sy.x : a.J;
  const int tiles = (rows + 15) / 16, groups = (len + kGroup - 1) / kGroup, kfr = (len + 15) / 16;
  if ((int)(blockIdx.x >> 1) >= tiles * groups) return;  // also the empty systems
  const int x = blockIdx.x & 1, t = (int)(blockIdx.x >> 1) % tiles, g = (int)(blockIdx.x >> 1) / tiles;
  const int lane = threadIdx.x, row = lane >> 2, q = lane & 3;
  const int64_t idx0 = (int64_t)m * (2 * a.N + 3 - m) / 2;
  auto val = [&](int r, int k) {
    if (r >= rows || k >= len) return 0.0;
    const int deg = a.synthesis ? k : r, lat = a.synthesis ? r : k;
    const double v = a.tab[x][(idx0 + cls + 2 * deg) * a.J + lat];
    return a.synthesis ? v * (1.0 / degree_scale(m + cls + 2 * deg)) : v;
  };
  double v[4][4][2];  // k16 step, register, pair
  int e[2] = {0, 0};
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[s][r][h] = val(t * 16 + row + (r & 1) * 8, g * kGroup + s * 16 + (r >> 1) * 8 + 2 * q + h);
        e[r & 1] = max(e[r & 1], bexp(v[s][r][h]));
      }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    e[r] = max(e[r], __shfl_xor_sync(0xffffffffu, e[r], 1));
    e[r] = max(e[r], __shfl_xor_sync(0xffffffffu, e[r], 2));
    if (q == 0) a.exps[(((int64_t)sy.z + g) * tiles + t) * 32 + x * 16 + row + 8 * r] = e[r] - 1023;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s)
    if (g * 4 + s < kfr) {
      uint4 *o = a.dig + ((((int64_t)sy.y + (g * 4 + s)) * tiles + t) * 2 + x) * (kFrag / 16);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        o[r * 32 + lane] = packed_digits(to_fixed(v[s][r][0], e[r & 1] - bexp(v[s][r][0])),
                                         to_fixed(v[s][r][1], e[r & 1] - bexp(v[s][r][1])));
    }
}

struct LegArgs {
  const uint4 *dig;
  const int *exps;
  const int4 *sys;
  double2 *four;     // [nlat][N+1][3B]
  double2 *spec;     // [3][nspec][B]
  const double *zd;  // [nspec]
  int N, nlat, J, B;
  int64_t nspec;
};

__device__ __forceinline__ int raw_at(int half, int k, int c) {
  return ((half * 2 + (k & 1)) * (kGroup / 2) + (k >> 1)) * kPitch + c;
}

template <int BYTES>
__device__ __forceinline__ void copy_or_zero(unsigned to, const void *from, bool ok) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" : : "r"(to), "l"(from), "r"(ok ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" : : "r"(to), "l"(from), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void copy_all() { asm volatile("cp.async.wait_all;" : : : "memory"); }

// Two real columns (a complex number's parts, x and y at this lane's places 2 lane and 2 lane + 1)
// as digits in fragment order, columns `col` and `col` + 1 of tile t, with their exponents.
__device__ __forceinline__ void cut_pair(double2 x, double2 y, uint4 *dig, int *cexp, int t, int col, int lane) {
  uint4 *o = dig + t * (kTileDig / 16) + (((lane >> 3) * 2 + ((lane >> 2) & 1)) * 2) * 32 + col * 4 + (lane & 3);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double u = h ? x.y : x.x, v = h ? y.y : y.x;
    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(bexp(u), bexp(v)));
    if (lane == 0) cexp[t * 8 + col + h] = e == 0x7ff ? kNotFinite : e - 1023;
    unsigned w[8];
    digits(to_fixed(u, e - bexp(u)), to_fixed(v, e - bexp(v)), w);
    o[h * 4] = make_uint4(w[0], w[1], w[2], w[3]);
    o[h * 4 + 32] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// A warp's table fragments, one step ahead in two places of shared memory; a lane reads only what
// it copied.
struct Ring {
  char *at;
  int lane, slot;
  __device__ __forceinline__ void copy(int s, const uint4 *from) const {
    const unsigned to = (unsigned)__cvta_generic_to_shared(at + s * kFrag + lane * 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) copy_or_zero<16>(to + i * 512, from + i * 32 + lane, true);
  }
};

// One product of a row tile: `steps` fragments of the table (`stride` uint4 apart, the first
// already on its way) times one column tile's digits; `next`: the fragment after these, if any.
// r: rows g and g + 8, columns 2 q and 2 q + 1.
__device__ __forceinline__ void product(Ring &ring, const uint4 *a, int64_t stride, const uint4 *next, const uint4 *b, int steps,
                                        int ea0, int ea1, int eb0, int eb1, double (&r)[4]) {
  const int lane = ring.lane;
  float s[8][4];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[c][k] = 0.0f;
#pragma unroll 1
  for (int k = 0; k < steps; ++k) {
    a = k + 1 < steps ? a + stride : next;
    if (a) ring.copy(ring.slot ^ 1, a);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" : : : "memory");
    const uint4 *f = reinterpret_cast<const uint4 *>(ring.at + ring.slot * kFrag) + lane;
    ring.slot ^= 1;
    unsigned w[4][8], v[2][8];
#pragma unroll
    for (int i = 0; i < 4; ++i) unpack(f[i * 32], 0x3c003c00u, 0xe480e480u, w[i]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint4 x = b[(2 * i) * 32 + lane], y = b[(2 * i + 1) * 32 + lane];
      v[i][0] = x.x, v[i][1] = x.y, v[i][2] = x.z, v[i][3] = x.w;
      v[i][4] = y.x, v[i][5] = y.y, v[i][6] = y.z, v[i][7] = y.w;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8 - i; ++j) mma_add(s[i + j], w[0][i], w[1][i], w[2][i], w[3][i], v[0][j], v[1][j]);
    b += 4 * 32;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    auto pair = [&](int c) { return __float2int_rn(s[c][k]) * 256 + __float2int_rn(s[c + 1][k]); };
    // sum of s_c 2^(-8 c) in units of 2^-44
    long long t = (long long)pair(0) << 32;
    asm("mad.wide.s32 %0, %1, 65536, %0;" : "+l"(t) : "r"(pair(2)));
    t += pair(4);
    const int ea = k & 2 ? ea1 : ea0, eb = k & 1 ? eb1 : eb0;
    r[k] = fixed_to_double((t << 4) + (pair(6) >> 12), eb >= kNotFinite ? kNotFinite : ea + eb - 54);
  }
}

__device__ __forceinline__ void add(double2 &s, double x, double y) { s = make_double2(s.x + x, s.y + y); }
__device__ __forceinline__ void add_im(double2 &s, double fm, double x, double y) {  // += i fm (x + i y)
  s = make_double2(fma(-fm, y, s.x), fma(fm, x, s.y));
}
__device__ __forceinline__ double2 of_field(double2 v, int lane, int f) {
  const int from = (lane & ~3) + f;
  return make_double2(__shfl_sync(0xffffffffu, v.x, from), __shfl_sync(0xffffffffu, v.y, from));
}

// Analysis: out[n] = sum_j; blockIdx.x: states, .y: row tiles (eight per CTA, classes 0, 1), .z: m.
// ONE: one state per CTA.  Its three fields share a column tile (lane q holds field q), which
// makes two products, P and H times all fields, of the five.
template <bool ONE>
__global__ void __launch_bounds__(256, 2) legendre_digits_analysis(LegArgs a) {
  extern __shared__ __align__(16) char smem[];
  constexpr int NC = ONE ? 3 : 12, CT = ONE ? 1 : 3;  // complex columns, column tiles of a class
  const double2 *raw = reinterpret_cast<const double2 *>(smem);
  uint4 *dig = reinterpret_cast<uint4 *>(smem + kDig);
  int *cexp = reinterpret_cast<int *>(smem + kExp);
  const int m = blockIdx.z, b0 = blockIdx.x * (ONE ? 1 : 4), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int4 s0 = a.sys[2 * m], s1 = a.sys[2 * m + 1];
  const int t0 = (s0.x + 15) / 16, t1 = (s1.x + 15) / 16;
  if ((int)blockIdx.y * kWarps >= t0 + t1) return;
  const int unit = blockIdx.y * kWarps + warp, cls = unit >= t0, tile = cls ? unit - t0 : unit;
  const bool live = unit < t0 + t1;
  const int4 sy = cls ? s1 : s0;
  const int tiles = cls ? t1 : t0, q = lane & 3, row = lane >> 2;
  const int M1 = a.N + 1, ncol = 3 * a.B;
  const double fm = (double)m;
  const int64_t stride = (int64_t)tiles * 2 * (kFrag / 16);
  const uint4 *fr = a.dig + ((int64_t)sy.y * tiles + tile) * 2 * (kFrag / 16);
  const int *ex = a.exps + ((int64_t)sy.z * tiles + tile) * 32 + row;
  Ring ring{smem + kRing + warp * 2 * kFrag, lane, 0};
  auto fetch = [&](int j0) {
    const unsigned to = (unsigned)__cvta_generic_to_shared(smem);
    for (int t = tid; t < 2 * kGroup * NC; t += 256) {
      const int c = t % NC, u = t / NC, half = u >> 6, jj = u & (kGroup - 1), j = j0 + jj;
      const bool ok = j < a.J && 3 * b0 + c < ncol;
      copy_or_zero<16>(to + raw_at(half, jj, c) * 16,
                       ok ? a.four + ((int64_t)(half ? a.nlat - 1 - j : j) * M1 + m) * ncol + 3 * b0 + c : a.four, ok);
    }
  };
  double2 phi[2], zeta[2], delta[2];  // rows row, row + 8; ONE: of this lane's field, P and H times it
#pragma unroll
  for (int i = 0; i < 2; ++i) phi[i] = zeta[i] = delta[i] = make_double2(0, 0);
  fetch(0);
  if (live) ring.copy(0, fr);
  for (int j0 = 0; j0 < a.J; j0 += kGroup) {
    copy_all();
    __syncthreads();  // the group's inputs are there, the digits of the group before have been used
    for (int u = warp; u < (ONE ? 8 : 24); u += kWarps) {
      const int odd = u & 1, f = ONE ? u >> 1 : (u >> 1) % 3, st = ONE ? 0 : (u >> 1) / 3;
      double2 v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[h] = make_double2(0, 0);
        if (ONE && f == 3) continue;
        const double2 n = raw[raw_at(0, 2 * lane + h, 3 * st + f)], s = raw[raw_at(1, 2 * lane + h, 3 * st + f)];
        v[h] = odd ? make_double2(n.x - s.x, n.y - s.y) : make_double2(n.x + s.x, n.y + s.y);
      }
      cut_pair(v[0], v[1], dig, cexp, odd * CT + (ONE ? 0 : f), 2 * (ONE ? f : st), lane);
    }
    __syncthreads();
    const bool more = j0 + kGroup < a.J;
    if (more) fetch(j0 + kGroup);
    if (!live) continue;
    const int steps = (min(kGroup, a.J - j0) + 15) / 16;
    const uint4 *after = more ? fr + 4 * stride : nullptr;
    // Pbar has the rows' own symmetry, H the other; xn: the table of the product after this one
    auto run = [&](int x, int f, int xn, double (&r)[4]) {
      const int t = (x ? 1 - cls : cls) * CT + f;
      product(ring, fr + x * (kFrag / 16), stride, xn < 0 ? after : fr + xn * (kFrag / 16), dig + t * (kTileDig / 16), steps,
              __ldg(ex + x * 16), __ldg(ex + x * 16 + 8), cexp[t * 8 + 2 * q], cexp[t * 8 + 2 * q + 1], r);
    };
    double r[4];
    if constexpr (ONE) {
      run(0, 0, 1, r);
#pragma unroll
      for (int i = 0; i < 2; ++i) add(phi[i], r[2 * i], r[2 * i + 1]);
      run(1, 0, -1, r);
#pragma unroll
      for (int i = 0; i < 2; ++i) add(zeta[i], r[2 * i], r[2 * i + 1]);
    } else {
      run(0, 0, 0, r);
#pragma unroll
      for (int i = 0; i < 2; ++i) add(phi[i], r[2 * i], r[2 * i + 1]);
      run(0, 2, 1, r);  // i m P V
#pragma unroll
      for (int i = 0; i < 2; ++i) add_im(zeta[i], fm, r[2 * i], r[2 * i + 1]);
      run(1, 1, 0, r);  // H U
#pragma unroll
      for (int i = 0; i < 2; ++i) add(zeta[i], r[2 * i], r[2 * i + 1]);
      run(0, 1, 1, r);  // i m P U
#pragma unroll
      for (int i = 0; i < 2; ++i) add_im(delta[i], fm, r[2 * i], r[2 * i + 1]);
      run(1, 2, -1, r);  // -H V
#pragma unroll
      for (int i = 0; i < 2; ++i) add(delta[i], -r[2 * i], -r[2 * i + 1]);
    }
    fr += 4 * stride;
    ex += tiles * 32;
  }
  if (!live) return;
  if constexpr (ONE) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const double2 pu = of_field(phi[i], lane, 1), pv = of_field(phi[i], lane, 2);
      const double2 hu = of_field(zeta[i], lane, 1), hv = of_field(zeta[i], lane, 2);
      zeta[i] = hu;
      add_im(zeta[i], fm, pv.x, pv.y);
      delta[i] = make_double2(-hv.x, -hv.y);
      add_im(delta[i], fm, pu.x, pu.y);
    }
  }
  const int b = ONE ? b0 : b0 + q;
  if (b >= a.B) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = tile * 16 + row + 8 * i;
    if (r >= sy.x) continue;
    const int64_t ix = (int64_t)m * (2 * a.N + 3 - m) / 2 + cls + 2 * r;
    const double s = a.zd[ix];
    if (!ONE || q == 0) a.spec[ix * a.B + b] = phi[i];
    if (!ONE || q == 1) a.spec[(a.nspec + ix) * a.B + b] = make_double2(s * zeta[i].x, s * zeta[i].y);
    if (!ONE || q == 2) a.spec[(2 * a.nspec + ix) * a.B + b] = make_double2(s * delta[i].x, s * delta[i].y);
  }
}

// Synthesis: F[j] = sum_n; blockIdx.x: states, .y: latitude tiles (eight per CTA), .z: m.  ONE: as above.
template <bool ONE>
__global__ void __launch_bounds__(256, 2) legendre_digits_synthesis(LegArgs a) {
  extern __shared__ __align__(16) char smem[];
  constexpr int NC = ONE ? 3 : 12, CT = ONE ? 1 : 3, NS = ONE ? 1 : 4;
  const double2 *raw = reinterpret_cast<const double2 *>(smem);
  const double *zds = reinterpret_cast<const double *>(smem + kZd);
  uint4 *dig = reinterpret_cast<uint4 *>(smem + kDig);
  int *cexp = reinterpret_cast<int *>(smem + kExp);
  const int m = blockIdx.z, b0 = blockIdx.x * (ONE ? 1 : 4), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles = (a.J + 15) / 16, tile = blockIdx.y * kWarps + warp, q = lane & 3, row = lane >> 2;
  const bool live = tile < tiles;
  const int64_t idx0 = (int64_t)m * (2 * a.N + 3 - m) / 2;
  const int deg = a.N - m + 1;
  const double fm = (double)m;
  const int64_t stride = (int64_t)tiles * 2 * (kFrag / 16);
  const int4 s0 = a.sys[2 * m], s1 = a.sys[2 * m + 1];
  const uint4 *fr[2] = {a.dig + ((int64_t)s0.y * tiles + tile) * 2 * (kFrag / 16),
                        a.dig + ((int64_t)s1.y * tiles + tile) * 2 * (kFrag / 16)};
  const int *ex[2] = {a.exps + ((int64_t)s0.z * tiles + tile) * 32 + row, a.exps + ((int64_t)s1.z * tiles + tile) * 32 + row};
  Ring ring{smem + kRing + warp * 2 * kFrag, lane, 0};
  auto fetch = [&](int r0) {  // degrees of both classes, three fields, the states
    const unsigned to = (unsigned)__cvta_generic_to_shared(smem);
    for (int t = tid; t < 2 * kGroup * NC; t += 256) {
      const int st = ONE ? 0 : t & 3, f = (ONE ? t : t >> 2) % 3, d = t / NC, n = 2 * r0 + d;
      const bool ok = n < deg && b0 + st < a.B;
      copy_or_zero<16>(to + raw_at(d & 1, d >> 1, f * NS + st) * 16,
                       ok ? a.spec + ((int64_t)f * a.nspec + idx0 + n) * a.B + b0 + st : a.spec, ok);
    }
    if (tid < 2 * kGroup) {
      const bool ok = 2 * r0 + tid < deg;
      copy_or_zero<8>(to + kZd + tid * 8, ok ? a.zd + idx0 + 2 * r0 + tid : a.zd, ok);
    }
  };
  double2 F[2][3][2];  // symmetry class, field, rows row and row + 8; ONE: P and H times this lane's field
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int f = 0; f < 3; ++f) F[c][f][0] = F[c][f][1] = make_double2(0, 0);
  fetch(0);
  if (live) ring.copy(0, fr[0]);
  for (int r0 = 0; r0 * 2 < deg; r0 += kGroup) {
    copy_all();
    __syncthreads();
    for (int u = warp; u < (ONE ? 8 : 24); u += kWarps) {
      const int odd = u & 1, f = ONE ? u >> 1 : (u >> 1) % 3, st = ONE ? 0 : (u >> 1) / 3;
      double2 v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[h] = make_double2(0, 0);
        if (ONE && f == 3) continue;
        const int d = 2 * (2 * lane + h) + odd;
        v[h] = raw[raw_at(odd, 2 * lane + h, f * NS + st)];
        double s = degree_scale(m + 2 * r0 + d);
        if (f > 0) s *= zds[d];
        v[h] = make_double2(s * v[h].x, s * v[h].y);
      }
      cut_pair(v[0], v[1], dig, cexp, odd * CT + (ONE ? 0 : f), 2 * (ONE ? f : st), lane);
    }
    __syncthreads();
    const bool more = (r0 + kGroup) * 2 < deg;
    if (more) fetch(r0 + kGroup);
    if (!live) continue;
#pragma unroll
    for (int cls = 0; cls < 2; ++cls) {
      const int left = (cls ? s1.x : s0.x) - r0;
      if (left <= 0) continue;  // class 1 of the last group only
      const int steps = (min(left, kGroup) + 15) / 16;
      const uint4 *after = cls == 0 ? (s1.x > r0 ? fr[1] : nullptr) : (more ? fr[0] + 4 * stride : nullptr);
      auto run = [&](int x, int f, int xn, double (&r)[4]) {
        const int t = cls * CT + f;
        product(ring, fr[cls] + x * (kFrag / 16), stride, xn < 0 ? after : fr[cls] + xn * (kFrag / 16),
                dig + t * (kTileDig / 16), steps, __ldg(ex[cls] + x * 16), __ldg(ex[cls] + x * 16 + 8), cexp[t * 8 + 2 * q],
                cexp[t * 8 + 2 * q + 1], r);
      };
      double r[4];
      if constexpr (ONE) {
        run(0, 0, 1, r);
#pragma unroll
        for (int i = 0; i < 2; ++i) add(F[cls][0][i], r[2 * i], r[2 * i + 1]);
        run(1, 0, -1, r);
#pragma unroll
        for (int i = 0; i < 2; ++i) add(F[cls][1][i], r[2 * i], r[2 * i + 1]);
      } else {
        run(0, 0, 0, r);  // P Phi
#pragma unroll
        for (int i = 0; i < 2; ++i) add(F[cls][0][i], r[2 * i], r[2 * i + 1]);
        run(0, 2, 0, r);  // U: i m P chi'
#pragma unroll
        for (int i = 0; i < 2; ++i) add_im(F[cls][1][i], fm, r[2 * i], r[2 * i + 1]);
        run(0, 1, 1, r);  // V: i m P psi'
#pragma unroll
        for (int i = 0; i < 2; ++i) add_im(F[cls][2][i], fm, r[2 * i], r[2 * i + 1]);
        run(1, 1, 1, r);  // U: -H psi', of the other symmetry
#pragma unroll
        for (int i = 0; i < 2; ++i) add(F[1 - cls][1][i], -r[2 * i], -r[2 * i + 1]);
        run(1, 2, -1, r);  // V: H chi'
#pragma unroll
        for (int i = 0; i < 2; ++i) add(F[1 - cls][2][i], r[2 * i], r[2 * i + 1]);
      }
    }
#pragma unroll
    for (int cls = 0; cls < 2; ++cls) {
      fr[cls] += 4 * stride;
      ex[cls] += tiles * 32;
    }
  }
  if (!live) return;
  const int b = ONE ? b0 : b0 + q, M1 = a.N + 1, ncol = 3 * a.B;
  if constexpr (ONE) {  // lane q takes field q: Phi; U = i m P chi' - H psi'; V = i m P psi' + H chi'
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      double2 o[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double2 p = of_field(F[c][0][i], lane, q == 1 ? 2 : (q == 2 ? 1 : 0)), h = of_field(F[1 - c][1][i], lane, q);
        const double sg = q == 1 ? -1.0 : 1.0;
        o[c] = q == 0 ? p : make_double2(sg * h.x, sg * h.y);
        if (q > 0) add_im(o[c], fm, p.x, p.y);
      }
      F[0][0][i] = o[0];
      F[1][0][i] = o[1];
    }
  }
  if (b >= a.B || (ONE && q == 3)) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int j = tile * 16 + row + 8 * i;
    if (j >= a.J) continue;
    double2 *north = a.four + ((int64_t)j * M1 + m) * ncol + 3 * b;
    double2 *south = a.four + ((int64_t)(a.nlat - 1 - j) * M1 + m) * ncol + 3 * b;
#pragma unroll
    for (int f = 0; f < (ONE ? 1 : 3); ++f) {
      const double2 x = F[0][f][i], y = F[1][f][i];
      north[ONE ? q : f] = make_double2(x.x + y.x, x.y + y.y);
      south[ONE ? q : f] = make_double2(x.x - y.x, x.y - y.y);
    }
  }
}

LegArgs leg_args(const Plan &pl, const LegendreDigits &t, const double2 *four, const double2 *spec, int B, const double *zd) {
  LegArgs a;
  a.dig = t.dig;
  a.exps = t.exps;
  a.sys = t.sys;
  a.four = const_cast<double2 *>(four);
  a.spec = const_cast<double2 *>(spec);
  a.zd = zd;
  a.N = pl.N;
  a.nlat = pl.nlat;
  a.J = pl.J;
  a.B = B;
  a.nspec = pl.nspec;
  return a;
}

}  // namespace

void free_legendre_digits(LegendreDigits &t) {
  if (t.dig) cudaFree(t.dig);  // the others lie behind it
  t = LegendreDigits{};
}

namespace {

// where each system's fragments and exponents lie, for one direction
struct TabLayout {
  std::vector<int4> sys;
  int64_t nfrag = 0, nexp = 0;
  int most = 0;
  bool ok = true;
  size_t dig_bytes() const { return (size_t)nfrag * 2 * kFrag; }
  size_t exp_bytes() const { return (size_t)nexp * 32 * sizeof(int); }
  size_t bytes() const { return dig_bytes() + exp_bytes() + sys.size() * sizeof(int4); }
};

TabLayout tab_layout(const Plan &pl, bool synthesis) {
  TabLayout L;
  int64_t frags = 0, groups = 0;
  const int jt = (pl.J + 15) / 16, jg = (pl.J + kGroup - 1) / kGroup;
  for (int m = 0; m <= pl.N; ++m)
    for (int c = 0; c < 2; ++c) {
      const int rows = (pl.N - m + 2 - c) / 2, rt = (rows + 15) / 16, rg = (rows + kGroup - 1) / kGroup;
      // fragment (k, tile) of the system is at (first + k) tiles + tile: `first` counts in the
      // system's own tiles, so the offset is rounded up to them
      const int tiles = std::max(1, synthesis ? jt : rt), kfr = synthesis ? rt : jt, kg = synthesis ? rg : jg;
      frags = (L.nfrag + tiles - 1) / tiles;
      groups = (L.nexp + tiles - 1) / tiles;
      L.sys.push_back(make_int4(rows, (int)frags, (int)groups, 0));
      if (frags > INT32_MAX || groups > INT32_MAX) L.ok = false;
      L.nfrag = (frags + kfr) * tiles;
      L.nexp = (groups + kg) * tiles;
      L.most = std::max(L.most, 2 * tiles * kg);
    }
  return L;
}

}  // namespace

// of both directions
size_t legendre_digit_bytes(const Plan &pl) { return tab_layout(pl, false).bytes() + tab_layout(pl, true).bytes(); }

// The tables in fragment order for one direction, from pl.tabP and pl.tabH; t stays empty (and
// the FP64 kernels of legendre.cu serve the plan) where the device memory does not suffice.
cudaError_t build_legendre_digits(Plan &pl, bool synthesis, LegendreDigits &t) {
  t = LegendreDigits{};
  const TabLayout L = tab_layout(pl, synthesis);
  const std::vector<int4> &sys = L.sys;
  if (!L.ok) return cudaSuccess;
  char *mem = nullptr;
  if (cudaMalloc(&mem, L.bytes()) != cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;
  }
  t.dig = reinterpret_cast<uint4 *>(mem);
  t.exps = reinterpret_cast<int *>(mem + L.dig_bytes());
  t.sys = reinterpret_cast<int4 *>(mem + L.dig_bytes() + L.exp_bytes());
  cudaError_t e = cudaMemcpy(t.sys, sys.data(), sys.size() * sizeof(int4), cudaMemcpyHostToDevice);
  TabArgs a;
  a.tab[0] = pl.tabP;
  a.tab[1] = pl.tabH;
  a.dig = t.dig;
  a.exps = t.exps;
  a.sys = t.sys;
  a.N = pl.N;
  a.J = pl.J;
  a.synthesis = synthesis;
  if (e == cudaSuccess) {
    legendre_digits_setup<<<dim3((unsigned)L.most, (unsigned)sys.size()), 32>>>(a);
    e = cudaGetLastError();
  }
  for (auto k : {legendre_digits_analysis<true>, legendre_digits_analysis<false>, legendre_digits_synthesis<true>,
                 legendre_digits_synthesis<false>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) free_legendre_digits(t);
  t.bytes = L.bytes();
  return e;
}

namespace {
// One state per CTA in place of four: a batch of one, and batches with few CTAs, where a CTA's chain of
// two products in place of five is what counts: up to two CTAs of one state per SM, which find their
// places at once, for the analysis, four for the synthesis.  With the FFT, us, one / four states per CTA:
// analysis T21 x 2 13.8 / 19.9 (FP64 kernels 18.5), T63 x 4 (256 CTAs) 20.8 / 26.0, T24 x 12 (300) 19.2 / 24.0;
// past the line T28 x 12 (348) 27.8 / 26.6, T24 x 16 (400) 27.1 / 25.7, T127 x 8 (1024) 91.6 / 73.5.
// Synthesis T21 x 2 14.6 / 24.5 (22.0), T63 x 4 22.5 / 32.7, T48 x 8 (392) 33.7 / 37.2, T85 x 6 (516) 44.0 / 52.7,
// T48 x 12 (588) 37.2 / 39.0; past the line T42 x 16 (688) 40.5 / 38.9, T63 x 12 (768) 47.6 / 42.9.
bool one_state(const Plan &pl, int B, unsigned rows, int per_sm) {
  return B == 1 || (int64_t)(pl.N + 1) * rows * B <= (int64_t)per_sm * pl.num_sms;
}
}  // namespace

cudaError_t launch_leg_ana_digits(Plan &pl, const double2 *four, double2 *sint, int B, const double *zd, cudaStream_t st) {
  const int tiles = (pl.N / 2 + 1 + 15) / 16 + ((pl.N + 1) / 2 + 15) / 16;
  const unsigned rows = (unsigned)((tiles + kWarps - 1) / kWarps);
  const bool one = one_state(pl, B, rows, 2);
  const dim3 g((unsigned)(one ? B : (B + 3) / 4), rows, (unsigned)(pl.N + 1));
  (one ? legendre_digits_analysis<true> : legendre_digits_analysis<false>)<<<g, 32 * kWarps, kSmem, st>>>(
      leg_args(pl, pl.leg_ana, four, sint, B, zd));
  return cudaGetLastError();
}

cudaError_t launch_leg_syn_digits(Plan &pl, const double2 *sint, double2 *four, int B, const double *zd, cudaStream_t st) {
  const unsigned rows = (unsigned)(((pl.J + 15) / 16 + kWarps - 1) / kWarps);
  const bool one = one_state(pl, B, rows, 4);
  const dim3 g((unsigned)(one ? B : (B + 3) / 4), rows, (unsigned)(pl.N + 1));
  (one ? legendre_digits_synthesis<true> : legendre_digits_synthesis<false>)<<<g, 32 * kWarps, kSmem, st>>>(
      leg_args(pl, pl.leg_syn, four, sint, B, zd));
  return cudaGetLastError();
}

}  // namespace rexi
