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
// A CTA of eight warps takes one zonal order and four states (blockIdx: m, states, rows); it
// folds and cuts a group's data into digits in shared memory, each warp then forms the five
// products of a row tile of 16 degrees or latitudes.  A tile of the product's columns is one
// field of the four states (re, im), so that a lane ends up with all fields of one state and
// combines them in registers.  Tables: 8 B per value as in the FP64 form, in fragment order.
//
// Measured on GB300 (analysis, synthesis; against the FP64 kernels): T341 x 16 0.92, 0.79 / 4.37, 4.07
// ms; T255 x 8 0.234, 0.204 / 1.01, 0.86; T170 x 1 0.058, 0.076 / 0.114, 0.169; T63 x 1 0.020, 0.027 /
// 0.037, 0.065.  The tensor pipe is a third busy (ncu, T255 x 8), the rest is waiting for table
// fragments and at the groups' barriers; two CTAs per SM (one: 1.39, 1.11 ms at T341).
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
constexpr int kColPitch = kGroup + 1;
constexpr int kBuf = 48 * kColPitch * 8;             // two classes of 24 real columns, binary64
constexpr int kTileDig = (kGroup / 16) * 2 * 2 * 512;  // digits of one column tile
constexpr int kSmem = kBuf + 6 * kTileDig + 48 * 4;
constexpr int kFrag = 2048;      // bytes of a 16 x 16 table fragment

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
    return a.tab[x][(idx0 + cls + 2 * deg) * a.J + lat];
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

// The columns in `buf` ([48][kColPitch] binary64, `n` values each, zero up to a multiple of 16)
// as digits in fragment order in `dig`, their exponents in `cexp`.  Column 8 t + c of six
// tiles; each warp takes six columns.
__device__ __forceinline__ void cut_columns(const double *buf, uint4 *dig, int *cexp, int warp, int lane) {
#pragma unroll 2
  for (int u = 0; u < 6; ++u) {
    const int col = warp * 6 + u, t = col >> 3, c = col & 7;
    const double x = buf[col * kColPitch + 2 * lane], y = buf[col * kColPitch + 2 * lane + 1];
    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(bexp(x), bexp(y)));
    if (lane == 0) cexp[col] = e == 0x7ff ? kNotFinite : e - 1023;
    unsigned w[8];
    digits(to_fixed(x, e - bexp(x)), to_fixed(y, e - bexp(y)), w);
    uint4 *o = dig + t * (kTileDig / 16) + (((lane >> 3) * 2 + ((lane >> 2) & 1)) * 2) * 32 + c * 4 + (lane & 3);
    o[0] = make_uint4(w[0], w[1], w[2], w[3]);
    o[32] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// One product of a row tile: `steps` fragments of the table (`stride` uint4 apart) times one
// column tile's digits.  r: rows g and g + 8, columns 2 q and 2 q + 1.
__device__ __forceinline__ void product(const uint4 *a, int64_t stride, const uint4 *b, int steps, int lane, int ea0, int ea1,
                                        int eb0, int eb1, double (&r)[4]) {
  float s[8][4];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[c][k] = 0.0f;
#pragma unroll 1
  for (int k = 0; k < steps; ++k) {
    unsigned w[4][8], v[2][8];
#pragma unroll
    for (int i = 0; i < 4; ++i) unpack(__ldg(a + i * 32 + lane), 0x3c003c00u, 0xe480e480u, w[i]);
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
    a += stride;
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

// Analysis: out[n] = sum_j; blockIdx.x: m, .y: states, .z: row tiles (eight per CTA, classes 0, 1)
__global__ void __launch_bounds__(256, 2) legendre_digits_analysis(LegArgs a) {
  extern __shared__ __align__(16) char smem[];
  double *buf = reinterpret_cast<double *>(smem);
  uint4 *dig = reinterpret_cast<uint4 *>(smem + kBuf);
  int *cexp = reinterpret_cast<int *>(smem + kBuf + 6 * kTileDig);
  const int m = blockIdx.x, b0 = blockIdx.y * 4, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int4 s0 = a.sys[2 * m], s1 = a.sys[2 * m + 1];
  const int t0 = (s0.x + 15) / 16, t1 = (s1.x + 15) / 16;
  if ((int)blockIdx.z * kWarps >= t0 + t1) return;
  const int unit = blockIdx.z * kWarps + warp, cls = unit >= t0, tile = cls ? unit - t0 : unit;
  const bool live = unit < t0 + t1;
  const int4 sy = cls ? s1 : s0;
  const int tiles = cls ? t1 : t0, q = lane & 3, row = lane >> 2;
  const int M1 = a.N + 1, ncol = 3 * a.B;
  const double fm = (double)m;
  double2 phi[2], zeta[2], delta[2];  // rows row, row + 8
#pragma unroll
  for (int i = 0; i < 2; ++i) phi[i] = zeta[i] = delta[i] = make_double2(0, 0);
  for (int j0 = 0, g = 0; j0 < a.J; j0 += kGroup, ++g) {
    const int jn = min(kGroup, a.J - j0);
    __syncthreads();  // the digits of the group before have been used
    for (int t = tid; t < kGroup * 12; t += 256) {
      const int jj = t / 12, c = t - jj * 12, f = c % 3, st = c / 3, cg = 3 * b0 + c;
      double2 n = make_double2(0, 0), s = n;
      if (jj < jn && cg < ncol) {
        n = a.four[((int64_t)(j0 + jj) * M1 + m) * ncol + cg];
        s = a.four[((int64_t)(a.nlat - 1 - j0 - jj) * M1 + m) * ncol + cg];
      }
      double *e = buf + (f * 8 + 2 * st) * kColPitch + jj, *o = e + 24 * kColPitch;
      e[0] = n.x + s.x;
      e[kColPitch] = n.y + s.y;
      o[0] = n.x - s.x;
      o[kColPitch] = n.y - s.y;
    }
    __syncthreads();
    cut_columns(buf, dig, cexp, warp, lane);
    __syncthreads();
    if (!live) continue;
    const int steps = (jn + 15) / 16;
    const int64_t stride = (int64_t)tiles * 2 * (kFrag / 16);
    const uint4 *fr = a.dig + (((int64_t)sy.y + g * 4) * tiles + tile) * 2 * (kFrag / 16);
    const int *ex = a.exps + (((int64_t)sy.z + g) * tiles + tile) * 32 + row;
    // Pbar has the rows' own symmetry, H the other
    auto run = [&](int x, int f, double (&r)[4]) {
      const int t = (x ? 1 - cls : cls) * 3 + f;
      product(fr + x * (kFrag / 16), stride, dig + t * (kTileDig / 16), steps, lane, __ldg(ex + x * 16), __ldg(ex + x * 16 + 8),
              cexp[t * 8 + 2 * q], cexp[t * 8 + 2 * q + 1], r);
    };
    double r[4];
    run(0, 0, r);
#pragma unroll
    for (int i = 0; i < 2; ++i) phi[i] = make_double2(phi[i].x + r[2 * i], phi[i].y + r[2 * i + 1]);
    run(0, 2, r);  // i m P V
#pragma unroll
    for (int i = 0; i < 2; ++i) zeta[i] = make_double2(fma(-fm, r[2 * i + 1], zeta[i].x), fma(fm, r[2 * i], zeta[i].y));
    run(1, 1, r);  // H U
#pragma unroll
    for (int i = 0; i < 2; ++i) zeta[i] = make_double2(zeta[i].x + r[2 * i], zeta[i].y + r[2 * i + 1]);
    run(0, 1, r);  // i m P U
#pragma unroll
    for (int i = 0; i < 2; ++i) delta[i] = make_double2(fma(-fm, r[2 * i + 1], delta[i].x), fma(fm, r[2 * i], delta[i].y));
    run(1, 2, r);  // -H V
#pragma unroll
    for (int i = 0; i < 2; ++i) delta[i] = make_double2(delta[i].x - r[2 * i], delta[i].y - r[2 * i + 1]);
  }
  const int b = b0 + q;
  if (!live || b >= a.B) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = tile * 16 + row + 8 * i;
    if (r >= sy.x) continue;
    const int64_t ix = (int64_t)m * (2 * a.N + 3 - m) / 2 + cls + 2 * r;
    const double s = a.zd[ix];
    a.spec[ix * a.B + b] = phi[i];
    a.spec[(a.nspec + ix) * a.B + b] = make_double2(s * zeta[i].x, s * zeta[i].y);
    a.spec[(2 * a.nspec + ix) * a.B + b] = make_double2(s * delta[i].x, s * delta[i].y);
  }
}

// Synthesis: F[j] = sum_n; blockIdx.x: m, .y: states, .z: latitude tiles (eight per CTA)
__global__ void __launch_bounds__(256, 2) legendre_digits_synthesis(LegArgs a) {
  extern __shared__ __align__(16) char smem[];
  double *buf = reinterpret_cast<double *>(smem);
  uint4 *dig = reinterpret_cast<uint4 *>(smem + kBuf);
  int *cexp = reinterpret_cast<int *>(smem + kBuf + 6 * kTileDig);
  const int m = blockIdx.x, b0 = blockIdx.y * 4, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles = (a.J + 15) / 16, tile = blockIdx.z * kWarps + warp, q = lane & 3, row = lane >> 2;
  const bool live = tile < tiles;
  const int64_t idx0 = (int64_t)m * (2 * a.N + 3 - m) / 2;
  const int deg = a.N - m + 1;
  const double fm = (double)m;
  double2 F[2][3][2];  // symmetry class, field, rows row and row + 8
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int f = 0; f < 3; ++f) F[c][f][0] = F[c][f][1] = make_double2(0, 0);
  for (int r0 = 0, g = 0; r0 * 2 < deg; r0 += kGroup, ++g) {
    __syncthreads();
    for (int t = tid; t < 2 * kGroup * 12; t += 256) {  // degrees of both classes, three fields, four states
      const int d = t / 12, c = t - d * 12, st = c & 3, f = c >> 2, b = b0 + st, n = 2 * r0 + d;
      double2 v = make_double2(0, 0);
      if (n < deg && b < a.B) {
        v = a.spec[((int64_t)f * a.nspec + idx0 + n) * a.B + b];
        if (f > 0) {
          const double s = a.zd[idx0 + n];
          v = make_double2(s * v.x, s * v.y);
        }
      }
      double *o = buf + ((d & 1) * 24 + f * 8 + 2 * st) * kColPitch + (d >> 1);
      o[0] = v.x;
      o[kColPitch] = v.y;
    }
    __syncthreads();
    cut_columns(buf, dig, cexp, warp, lane);
    __syncthreads();
    if (!live) continue;
#pragma unroll
    for (int cls = 0; cls < 2; ++cls) {
      const int4 sy = a.sys[2 * m + cls];
      const int left = sy.x - r0;
      if (left <= 0) continue;
      const int steps = (min(left, kGroup) + 15) / 16;
      const int64_t stride = (int64_t)tiles * 2 * (kFrag / 16);
      const uint4 *fr = a.dig + (((int64_t)sy.y + g * 4) * tiles + tile) * 2 * (kFrag / 16);
      const int *ex = a.exps + (((int64_t)sy.z + g) * tiles + tile) * 32 + row;
      auto run = [&](int x, int f, double (&r)[4]) {
        const int t = cls * 3 + f;
        product(fr + x * (kFrag / 16), stride, dig + t * (kTileDig / 16), steps, lane, __ldg(ex + x * 16),
                __ldg(ex + x * 16 + 8), cexp[t * 8 + 2 * q], cexp[t * 8 + 2 * q + 1], r);
      };
      auto add = [](double2 &s, double x, double y) { s = make_double2(s.x + x, s.y + y); };
      double r[4];
      run(0, 0, r);  // P Phi
#pragma unroll
      for (int i = 0; i < 2; ++i) add(F[cls][0][i], r[2 * i], r[2 * i + 1]);
      run(0, 2, r);  // U: i m P chi'
#pragma unroll
      for (int i = 0; i < 2; ++i)
        F[cls][1][i] = make_double2(fma(-fm, r[2 * i + 1], F[cls][1][i].x), fma(fm, r[2 * i], F[cls][1][i].y));
      run(0, 1, r);  // V: i m P psi'
#pragma unroll
      for (int i = 0; i < 2; ++i)
        F[cls][2][i] = make_double2(fma(-fm, r[2 * i + 1], F[cls][2][i].x), fma(fm, r[2 * i], F[cls][2][i].y));
      run(1, 1, r);  // U: -H psi', of the other symmetry
#pragma unroll
      for (int i = 0; i < 2; ++i) add(F[1 - cls][1][i], -r[2 * i], -r[2 * i + 1]);
      run(1, 2, r);  // V: H chi'
#pragma unroll
      for (int i = 0; i < 2; ++i) add(F[1 - cls][2][i], r[2 * i], r[2 * i + 1]);
    }
  }
  const int b = b0 + q, M1 = a.N + 1, ncol = 3 * a.B;
  if (!live || b >= a.B) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int j = tile * 16 + row + 8 * i;
    if (j >= a.J) continue;
    double2 *north = a.four + ((int64_t)j * M1 + m) * ncol + 3 * b;
    double2 *south = a.four + ((int64_t)(a.nlat - 1 - j) * M1 + m) * ncol + 3 * b;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const double2 x = F[0][f][i], y = F[1][f][i];
      north[f] = make_double2(x.x + y.x, x.y + y.y);
      south[f] = make_double2(x.x - y.x, x.y - y.y);
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
  for (void *p : {(void *)t.dig, (void *)t.exps, (void *)t.sys})
    if (p) cudaFree(p);
  t = LegendreDigits{};
}

// The tables in fragment order for one direction, from pl.tabP and pl.tabH; t stays empty (and
// the FP64 kernels of legendre.cu serve the plan) where the device memory does not suffice.
cudaError_t build_legendre_digits(Plan &pl, bool synthesis, LegendreDigits &t) {
  t = LegendreDigits{};
  std::vector<int4> sys;
  int64_t frags = 0, groups = 0, nfrag = 0, nexp = 0;
  int most = 0;
  const int jt = (pl.J + 15) / 16, jg = (pl.J + kGroup - 1) / kGroup;
  for (int m = 0; m <= pl.N; ++m)
    for (int c = 0; c < 2; ++c) {
      const int rows = (pl.N - m + 2 - c) / 2, rt = (rows + 15) / 16, rg = (rows + kGroup - 1) / kGroup;
      // fragment (k, tile) of the system is at (first + k) tiles + tile: `first` counts in the
      // system's own tiles, so the offset is rounded up to them
      const int tiles = std::max(1, synthesis ? jt : rt), kfr = synthesis ? rt : jt, kg = synthesis ? rg : jg;
      frags = (nfrag + tiles - 1) / tiles;
      groups = (nexp + tiles - 1) / tiles;
      sys.push_back(make_int4(rows, (int)frags, (int)groups, 0));
      if (frags > INT32_MAX || groups > INT32_MAX) return cudaSuccess;
      nfrag = (frags + kfr) * tiles;
      nexp = (groups + kg) * tiles;
      most = std::max(most, 2 * tiles * kg);
    }
  cudaError_t e = cudaSuccess;
  if (cudaMalloc(&t.dig, (size_t)nfrag * 2 * kFrag) != cudaSuccess ||
      cudaMalloc(&t.exps, (size_t)nexp * 32 * sizeof(int)) != cudaSuccess ||
      cudaMalloc(&t.sys, sys.size() * sizeof(int4)) != cudaSuccess) {
    cudaGetLastError();
    free_legendre_digits(t);
    return cudaSuccess;
  }
  e = cudaMemcpy(t.sys, sys.data(), sys.size() * sizeof(int4), cudaMemcpyHostToDevice);
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
    legendre_digits_setup<<<dim3((unsigned)most, (unsigned)sys.size()), 32>>>(a);
    e = cudaGetLastError();
  }
  for (auto k : {legendre_digits_analysis, legendre_digits_synthesis})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) free_legendre_digits(t);
  t.bytes = (size_t)nfrag * 2 * kFrag + (size_t)nexp * 32 * sizeof(int);
  return e;
}

cudaError_t launch_leg_ana_digits(Plan &pl, const double2 *four, double2 *sint, int B, const double *zd, cudaStream_t st) {
  const int tiles = (pl.N / 2 + 1 + 15) / 16 + ((pl.N + 1) / 2 + 15) / 16;
  const dim3 g((unsigned)(pl.N + 1), (unsigned)((B + 3) / 4), (unsigned)((tiles + kWarps - 1) / kWarps));
  legendre_digits_analysis<<<g, 32 * kWarps, kSmem, st>>>(leg_args(pl, pl.leg_ana, four, sint, B, zd));
  return cudaGetLastError();
}

cudaError_t launch_leg_syn_digits(Plan &pl, const double2 *sint, double2 *four, int B, const double *zd, cudaStream_t st) {
  const dim3 g((unsigned)(pl.N + 1), (unsigned)((B + 3) / 4), (unsigned)(((pl.J + 15) / 16 + kWarps - 1) / kWarps));
  legendre_digits_synthesis<<<g, 32 * kWarps, kSmem, st>>>(leg_args(pl, pl.leg_syn, four, sint, B, zd));
  return cudaGetLastError();
}

}  // namespace rexi
