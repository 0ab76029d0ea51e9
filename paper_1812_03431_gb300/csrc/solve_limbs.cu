// Banded shifted solves of small batches (one to four states) with their two contractions in
// exact integer arithmetic (paper Sec. 4.2, Sec. 5, Algorithm 1; binary64 delta solver).
//
// As in solve_digits.cu, only the 8 FP64 FMAs per (state, pole, row) of the two recurrences stay
// on the FP64 unit (one warp instruction per 64 cycles and scheduler); the right-hand sides
// and the beta-weighted sums, 28 of the 36, are fixed-point products.  With one state a factor is
// used once, so the tensor cores would multiply mostly padding: here each operand is a 59-bit
// integer (weights: 56) relative to the largest of its group, held as two signed limbs of radix
// 2^30, and a product is three 32 x 32 -> 64 bit multiply-adds into a high and a middle 64-bit
// sum, 40 for the four inputs of a right-hand side and 48 for the four weighted sums of a pole.
// The product of the low limbs, below 2^-60 of the largest product, is left out; nothing else
// is rounded until a sum is put together (59 bits below the largest product) and rounded to
// binary64 once.  A window's sums over the lanes are 64-bit integer additions.
//
// Measured on GB300 (solve with its sums, against the fused FP64 solve): T341, 535 poles, one state
// 0.91 / 2.10 ms, four states 3.04 / 8.12; T170 x 1 0.27 / 0.56, T128 x 1 with 1047 poles 0.29 / 0.61,
// T639 x 1 3.05 / 7.87 (slot solve), T63 x 1 with 279 poles 0.073 / 0.089.  With one state the factors
// bound it (T639: 16.3 GB per step, 5.3 TB/s), with four the FP64 unit and the instruction issue
// share it; small truncations wait on the row-to-row chain of their few warps.
//
// Lanes of a warp are (state, pole): SB states x 32 / SB poles, two poles per lane where the
// window is full (poles k and k + 32 / SB), one for a short last window.  The factors are as
// large as the binary64 set (148 B per row and pole) and each is read once per tile of states.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "limb_sweep.h"
#include "rexi_internal.h"

namespace rexi {

using namespace fixed;
using namespace limb_solve;

namespace {

// ---- plan time ----------------------------------------------------------------------------------
struct SetupArgs {
  const double2 *fac;  // [F_NCOMP][nrows][P]
  const int4 *sys;
  char *fwd, *bwd;     // records, system by system: [block][row of the system]
  int *vexp;           // [nrows][4]: the scale of each input (0 for delta)
  int *bad;            // set when the factors are not finite or too unlike in scale
  int P, nblk, kmid;
  int64_t nrows;
};

__global__ void __launch_bounds__(kBlock) limb_factor_kernel(SetupArgs a) {
  __shared__ int emx[2][4];
  const int4 sy = a.sys[blockIdx.y];
  const int len = sy.z, i = blockIdx.x / a.nblk, blk = blockIdx.x - i * a.nblk;
  if (i >= len) return;
  const int64_t row0 = sy.w, row = row0 + i;
  const int p = threadIdx.x, k = blk * kBlock + p;
  const bool live = k < a.P;
  auto get = [&](int comp, int kk) {
    return kk < a.P ? a.fac[((int64_t)comp * a.nrows + row) * a.P + kk] : make_double2(0, 0);
  };
  auto emax = [](double2 v) { return max(bexp(v.x), bexp(v.y)); };
  const int64_t rec = row0 * a.nblk + (int64_t)blk * len + i;
  char *fr = a.fwd + rec * kFwd, *br = a.bwd + rec * kBwd;
  bool bad = false;

  // couplings of Phi, zeta_{n-1}, zeta_{n+1} (delta's is 1), negated; 59 bits below the pole's largest
  const int comp[3] = {F_G, F_E, F_F};
  double2 v[3];
  int ve[3], E = live ? 1023 : 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    v[j] = get(comp[j], k);
    v[j] = make_double2(-v[j].x, -v[j].y);
    const int mid = emax(get(comp[j], a.kmid)), e = emax(v[j]);
    ve[j] = mid == 0 ? 0 : mid - 1023;
    if (e == 0x7ff) bad = true;
    if (e) E = max(E, e - ve[j]);
  }
  if (live && E - 1023 > kMaxSpread) bad = true;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int e = emax(v[j]);
    if (e && E - (e - ve[j]) > kMaxSpread) bad = true;
    reinterpret_cast<int4 *>(fr)[j * kBlock + p] = limbs2((to_fixed(v[j].x, E - (bexp(v[j].x) - ve[j])) + 4) >> 3,
                                                          (to_fixed(v[j].y, E - (bexp(v[j].y) - ve[j])) + 4) >> 3);
  }
  const double2 l = get(F_L, k), c = get(F_C, k);
  if (emax(l) == 0x7ff || emax(c) == 0x7ff) bad = true;
  reinterpret_cast<double2 *>(fr + kFL)[p] = l;
  reinterpret_cast<int *>(fr + kFE)[p] = live ? E - 1023 : kNoPole;
  reinterpret_cast<double2 *>(br)[p] =
      i > 0 && k < a.P ? a.fac[((int64_t)F_C * a.nrows + row - 1) * a.P + k] : make_double2(0, 0);
  if (blk == 0 && p < 4) a.vexp[row * 4 + p] = p == 0 ? 0 : ve[p - 1];

  // the four weights, 56 bits below the block's largest
  const int wc[4] = {F_BD, F_BAD, F_ZP, F_ZM};
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    int m = emax(get(wc[s], k));
    if (m == 0x7ff) bad = true;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((p & 31) == 0) emx[p >> 5][s] = m;
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const double2 x = get(wc[s], k);
    const int m = max(emx[0][s], emx[1][s]);
    reinterpret_cast<int4 *>(br + kBW)[s * kBlock + p] =
        limbs2((to_fixed(x.x, m - bexp(x.x)) + 32) >> 6, (to_fixed(x.y, m - bexp(x.y)) + 32) >> 6);
    if (p == s) reinterpret_cast<int *>(br + kBE)[s] = m - 1023;
  }
  if (bad) atomicOr(a.bad, 1);
}

// ---- per step: the row inputs as limbs ----------------------------------------------------------
struct StateArgs {
  const double2 *sin;  // [3][nspec][B]
  const int4 *sys;
  const int *vexp;
  int4 *dig;           // [nrows][B][4 inputs]
  int *uexp;           // [nrows][B]
  int64_t nspec;
  int B, N;
};

__global__ void limb_state_kernel(StateArgs a) {
  const int4 sy = a.sys[blockIdx.y];
  const int m = sy.x, n0 = sy.y, len = sy.z, nmin = m > 1 ? m : 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x, q = t & 3, rb = t >> 2;
  const bool live = rb < len * a.B;  // whole groups of 4 threads
  const int i = rb / a.B, b = rb - i * a.B;
  const int64_t at = ((int64_t)sy.w + i) * a.B + b;
  const int n = n0 + 2 * i, nn = q < 2 ? n : (q == 2 ? n - 1 : n + 1), field = q == 0 ? 2 : (q == 1 ? 0 : 1);
  double2 x = make_double2(0, 0);
  if (live && nn >= nmin && nn <= a.N) {
    const int64_t ix = (int64_t)m * (2 * a.N + 3 - m) / 2 + (nn - m);
    x = __ldg(a.sin + ((int64_t)field * a.nspec + ix) * a.B + b);
  }
  const int v = live ? a.vexp[((int64_t)sy.w + i) * 4 + q] : 0;
  const int er = bexp(x.x), ei = bexp(x.y), e = max(er, ei);
  int U = e ? e + v : -(1 << 24), nf = e == 0x7ff;
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    U = max(U, __shfl_xor_sync(0xffffffffu, U, o));
    nf |= __shfl_xor_sync(0xffffffffu, nf, o);
  }
  if (!live) return;
  a.dig[at * 4 + q] = nf ? make_int4(0, 0, 0, 0)
                         : limbs2((to_fixed(x.x, U - (er + v)) + 4) >> 3, (to_fixed(x.y, U - (ei + v)) + 4) >> 3);
  if (q == 0) a.uexp[at] = nf ? kNotFinite : (U < -(1 << 23) ? 0 : U - 1023);
}

// ---- per step: the sweeps (limb_sweep.h) ----------------------------------------------------------
template <int SB, int CTAS>
__global__ void __launch_bounds__(128, CTAS) solve_limbs_kernel(LimbSweep a) {
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
    limb_item<SB>(a, a.items[it], lane, yb, smem);
  }
}

// resident CTAs of four warps per SM
constexpr int kCtas = 4;

}  // namespace

int limb_tile(int B) { return B >= 3 ? 4 : B; }                    // states per warp

namespace {
void (*kernel_for(int B))(LimbSweep) {
  switch (limb_tile(B)) {
    case 1: return solve_limbs_kernel<1, kCtas>;
    case 2: return solve_limbs_kernel<2, kCtas>;
    default: return solve_limbs_kernel<4, kCtas>;
  }
}
}  // namespace

// raises the kernel's shared-memory limit, when a layout is built
cudaError_t limb_configure(int B) {
  return cudaFuncSetAttribute(kernel_for(B), cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kSmemWarp);
}

int limb_window(int B, int kc) { return kc * 32 / limb_tile(B); }  // poles per window, kc per lane
size_t limb_factor_bytes(const Plan &pl) {
  return (size_t)pl.nrows * ((pl.P + kBlock - 1) / kBlock) * (kFwd + kBwd) + (size_t)pl.nrows * 4 * sizeof(int);
}
size_t limb_state_bytes(const Plan &pl, int B) { return (size_t)pl.nrows * B * (4 * sizeof(int4) + sizeof(int)); }

// The factor set as limbs; D's buffers are allocated, D.vexp with one more int for `bad`.
cudaError_t launch_limb_factors(Plan &pl, const double2 *fac, DigitFactors &D, int kmid, int *bad) {
  SetupArgs a;
  a.fac = fac;
  a.sys = pl.sys_dev;
  a.fwd = D.fwd;
  a.bwd = D.bwd;
  a.vexp = D.vexp;
  a.bad = bad;
  a.P = pl.P;
  a.nblk = (pl.P + kBlock - 1) / kBlock;
  a.kmid = kmid;
  a.nrows = pl.nrows;
  limb_factor_kernel<<<dim3((unsigned)(pl.lmax * a.nblk), (unsigned)pl.sys.size()), kBlock>>>(a);
  return cudaGetLastError();
}

void limb_record_bytes(size_t *fwd, size_t *bwd, int *block) {
  *fwd = kFwd;
  *bwd = kBwd;
  *block = kBlock;
}

cudaError_t launch_limb_state(Plan &pl, bool adjoint, const double2 *sin, int B, cudaStream_t st) {
  StateArgs s;
  s.sin = sin;
  s.sys = pl.sys_dev;
  s.vexp = (adjoint ? pl.dig_adj : pl.dig_fwd).vexp;
  s.dig = reinterpret_cast<int4 *>(pl.dig_state);
  s.uexp = reinterpret_cast<int *>(pl.dig_state + (size_t)pl.nrows * B * 4 * sizeof(int4));
  s.nspec = pl.nspec;
  s.B = B;
  s.N = pl.N;
  limb_state_kernel<<<dim3((unsigned)((pl.lmax * B * 4 + 255) / 256), (unsigned)pl.sys.size()), 256, 0, st>>>(s);
  return cudaGetLastError();
}

LimbSweep limb_sweep(Plan &pl, const DigitLayout &L, bool adjoint, int B) {
  const DigitFactors &D = adjoint ? pl.dig_adj : pl.dig_fwd;
  LimbSweep a;
  a.fwd = D.fwd;
  a.bwd = D.bwd;
  a.dig = reinterpret_cast<const int4 *>(pl.dig_state);
  a.uexp = reinterpret_cast<const int *>(pl.dig_state + (size_t)pl.nrows * B * 4 * sizeof(int4));
  a.sys = pl.sys_dev;
  a.items = L.items_dev;
  a.part = reinterpret_cast<double *>(pl.partial);
  a.ybuf = pl.yscratch;
  a.counter = pl.counter;
  a.nrows = pl.nrows;
  a.nitems = L.nitems;
  a.B = B;
  a.P = pl.P;
  a.nblk = (pl.P + kBlock - 1) / kBlock;
  a.lmax = pl.lmax;
  a.kc = L.kc;
  return a;
}

cudaError_t launch_solve_limbs(Plan &pl, const DigitLayout &L, bool adjoint, int B, cudaStream_t st) {
  const unsigned ctas = (unsigned)std::max(1, std::min(pl.num_sms * kCtas, (L.nitems + 3) / 4));
  kernel_for(B)<<<ctas, 128, 4 * kSmemWarp, st>>>(limb_sweep(pl, L, adjoint, B));
  return cudaGetLastError();
}

}  // namespace rexi
