// Banded shifted solves of small batches (one to five states) with their two contractions in
// exact integer arithmetic (paper Sec. 4.2, Sec. 5, Algorithm 1; binary64 delta solver).
//
// As in solve_digits.cu, only the 8 FP64 FMAs per (state, pole, row) of the two recurrences stay
// on the FP64 unit (one warp instruction per 64 cycles and scheduler); the right-hand sides
// and the beta-weighted sums, 28 of the 36, are fixed-point products.  With one state a factor is
// used once, so the tensor cores would multiply mostly padding: here each operand is a 59-bit
// integer relative to the largest of its group, held as two signed limbs of radix 2^30, and a
// product is three 32 x 32 -> 64 bit multiply-adds into a high and a middle 64-bit sum.  The
// product of the low limbs, below 2^-60 of the largest product, is left out.
//
// A row's couplings and weights are not stored one by one: each is a real number of the row
// times 1/alpha, 1/s_{n-1}, 1/s_{n+1} (s_n = alpha + i tau sigma_n, shared by neighbouring rows), and
// for the weights beta/d'.  The real numbers go into the inputs before the sweep and into the
// sums after it; the sweep forms u = (beta/d') w once and sums u, u/alpha, u/s_{n+1} and u/s_{n-1}:
// 40 multiply-adds for a right-hand side and 48 for the sums as with stored factors, at 68 B per
// row and pole instead of 148.  Roundings: u at 2^-59 of the window's largest u, a lane's sums at
// 2^-56, the total once to binary64; sums over the lanes are 64-bit integer additions.  beta, 1/d'
// and w differ over the poles by several bits and not together: with one exponent of beta/d' per
// block of poles and one of w per window, the outputs lost 1e-15 on white noise; with an exponent
// per pole they agree with the tensor-core solve's to 3e-16, for 4 B per row and pole more.
//
// Measured on GB300 (solve with its sums, against the fused FP64 solve): T341, 535 poles, one state
// 0.82 / 2.10 ms, four states 3.11 / 8.12; T170 x 1 0.26 / 0.56, T128 x 1 with 1047 poles 0.28 / 0.61,
// T639 x 1 2.77 / 7.87 (slot solve), T63 x 1 with 279 poles 0.047 / 0.089.  With every factor of a
// row stored (148 B per row and pole) one state waited on HBM: T639 3.05 ms, T341 0.91.  Now the
// integer pipe is 59 % and the FP64 unit 57 % busy (ncu, T341 x 1) and the rest is latency.  Small
// truncations waited on the row-to-row chain of their few warps (T63 0.066 ms): there a CTA's four
// warps share a window (sweep_window_split).
//
// Lanes of a warp are poles of one state: two per lane where the window is full (poles k and
// k + 32), one for a short last window.  Two or four states by a warp's lanes, which read each
// factor once for them, were no faster (T341 x 4 3.18 / 3.14 ms, T170 x 4 0.86 / 0.83, T42 x 4 0.053 /
// 0.055) and padded three states to four (T341 x 3 3.13 / 2.38, T170 x 3 0.82 / 0.63).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
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
  const double2 *alpha;
  const double *coef;  // [nspec][4]: sigma, ct, dt, G
  const int4 *sys;
  char *fwd, *bwd, *inv;
  int4 *inv_alpha;
  int *eblk;           // [nblk]
  double *scale;       // [nrows][6]: inputs Phi, zeta_{n-1}, zeta_{n+1}; sums Phi, zeta_{n+1}, zeta_{n-1}
  int *bad;            // set when the factors are not finite or too unlike in scale
  int P, nblk, N, e0, adjoint;
  int64_t nrows;
  double tau, q, phibar;  // q = 2 Omega tau
};

// One block of threads per (system, block of poles, j = 0..len): 1/s at degree n0 - 1 + 2 j and,
// for j < len, the row's l, Chat and beta/d' and its real factors.
__global__ void __launch_bounds__(kBlock) limb_factor_kernel(SetupArgs a) {
  const int4 sy = a.sys[blockIdx.y];
  const int m = sy.x, n0 = sy.y, len = sy.z, j = blockIdx.x / a.nblk, blk = blockIdx.x - j * a.nblk;
  if (len == 0 || j > len) return;
  const int64_t row0 = sy.w, row = row0 + j;
  const int p = threadIdx.x, k = blk * kBlock + p, nmin = m > 1 ? m : 1;
  const bool live = k < a.P;
  const double2 zero = make_double2(0, 0);
  auto C4 = [&](int n, int c) {
    return n < nmin || n > a.N ? 0.0 : a.coef[4 * ((int64_t)m * (2 * a.N + 3 - m) / 2 + (n - m)) + c];
  };
  auto emax = [](double2 v) { return max(bexp(v.x), bexp(v.y)); };
  bool bad = false;
  int largest = -1023;
  // the reciprocal of s as 59 bits below 2^(e0 + 1); the poles' may differ by kMaxSpread bits
  auto inverse = [&](double2 s) {
    if (!live) return make_int4(0, 0, 0, 0);
    const double d = s.x * s.x + s.y * s.y;
    const double2 v = make_double2(s.x / d, -s.y / d);
    const int e = emax(v), top = a.e0 + 1023;
    largest = max(largest, e - 1023);
    if (e > top || e + kMaxSpread < top) {  // also what is not finite
      bad = true;
      return make_int4(0, 0, 0, 0);
    }
    return limbs2((to_fixed(v.x, top - bexp(v.x)) + 4) >> 3, (to_fixed(v.y, top - bexp(v.y)) + 4) >> 3);
  };
  double2 al = live ? a.alpha[k] : make_double2(1, 0);
  if (a.adjoint) al.y = -al.y;
  const double sg = a.tau * C4(n0 - 1 + 2 * j, 0);
  reinterpret_cast<int4 *>(a.inv + ((row0 + blockIdx.y) * a.nblk + (int64_t)blk * (len + 1) + j) * kRec)[p] =
      inverse(make_double2(al.x, a.adjoint ? al.y - sg : al.y + sg));
  if (row == 0 && j == 0) a.inv_alpha[k] = inverse(al);
  if (j < len) {
    auto get = [&](int comp, int64_t r) { return live ? a.fac[((int64_t)comp * a.nrows + r) * a.P + k] : zero; };
    const int64_t rec = row0 * a.nblk + (int64_t)blk * len + j;
    const double2 l = get(F_L, row), c = j > 0 ? get(F_C, row - 1) : zero, b = get(F_BD, row);
    if (emax(l) == 0x7ff || emax(c) == 0x7ff || emax(b) == 0x7ff) bad = true;
    char *br = a.bwd + rec * kBwd;
    reinterpret_cast<double2 *>(a.fwd + rec * kRec)[p] = l;
    reinterpret_cast<double2 *>(br)[p] = c;
    // beta/d': 59 bits, each with its exponent
    const int top = emax(b);
    reinterpret_cast<int4 *>(br + kRec)[p] =
        limbs2((to_fixed(b.x, top - bexp(b.x)) + 4) >> 3, (to_fixed(b.y, top - bexp(b.y)) + 4) >> 3);
    reinterpret_cast<int *>(br + kBE)[p] = top - 1023;
    if (blk == 0 && p == 0) {
      const int n = n0 + 2 * j;
      double *s = a.scale + row * 6;
      s[0] = a.adjoint ? a.tau * a.phibar : -a.tau * C4(n, 3);
      s[1] = a.adjoint ? a.q * C4(n - 1, 2) : -a.q * C4(n, 1);
      s[2] = a.adjoint ? a.q * C4(n + 1, 1) : -a.q * C4(n, 2);
      s[3] = a.adjoint ? -a.tau * C4(n, 3) : a.tau * a.phibar;
      s[4] = a.adjoint ? -a.q * C4(n, 2) : a.q * C4(n + 1, 1);
      s[5] = a.adjoint ? -a.q * C4(n, 1) : a.q * C4(n - 1, 2);
    }
  }
  largest = (int)__reduce_max_sync(0xffffffffu, (unsigned)(largest + 2048)) - 2048;
  if ((p & 31) == 0) atomicMax(a.eblk + blk, largest);
  if (bad) atomicOr(a.bad, 1);
}

// ---- per step: the row inputs as limbs ----------------------------------------------------------
struct StateArgs {
  const double2 *sin;  // [3][nspec] places `place` apart, states `state` apart
  const int4 *sys;
  const double *scale;
  int4 *dig;           // [nrows][B][4 inputs]
  int *uexp;           // [nrows][B]
  unsigned *counter;   // the sweep's next item, set to zero here (null: not)
  int64_t nspec, place, state;
  int B, N;
};

__global__ void limb_state_kernel(StateArgs a) {
  if (a.counter && blockIdx.x + blockIdx.y + threadIdx.x == 0) *a.counter = 0;
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
    x = __ldg(a.sin + ((int64_t)field * a.nspec + ix) * a.place + b * a.state);
  }
  if (live && q > 0) {
    const double v = a.scale[((int64_t)sy.w + i) * 6 + q - 1];
    x = make_double2(v * x.x, v * x.y);
  }
  const int er = bexp(x.x), ei = bexp(x.y), e = max(er, ei);
  int U = e, nf = e == 0x7ff;
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    U = max(U, __shfl_xor_sync(0xffffffffu, U, o));
    nf |= __shfl_xor_sync(0xffffffffu, nf, o);
  }
  if (!live) return;
  a.dig[at * 4 + q] = nf ? make_int4(0, 0, 0, 0)
                         : limbs2((to_fixed(x.x, U - er) + 4) >> 3, (to_fixed(x.y, U - ei) + 4) >> 3);
  if (q == 0) a.uexp[at] = nf ? kNotFinite : U - 1023;
}

// ---- per step: the sweeps (limb_sweep.h) ----------------------------------------------------------
// resident CTAs of four warps per SM
constexpr int kCtas = 4;

__global__ void __launch_bounds__(128, kCtas) solve_limbs_kernel(LimbSweep a) {
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
    limb_item(a, a.items[it], lane, yb, smem);
  }
}

// The recurrences' warp differs between an SM's CTAs (blocks fill the SMs in turn), so that
// each scheduler's FP64 unit gets one of the four.
__global__ void __launch_bounds__(128, kCtas) solve_limbs_split_kernel(LimbSweep a) {
  __shared__ unsigned next;
  extern __shared__ __align__(16) char stages[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lead = (blockIdx.x / a.sms) & 3;
  double2 *yb = a.ybuf + (int64_t)(blockIdx.x * 4 + warp) * a.lmax * 64 + lane;
  for (;;) {
    if (threadIdx.x == 0) next = atomicAdd(a.counter, 1u);
    __syncthreads();
    const unsigned it = next;
    if (it >= (unsigned)a.nitems) break;
    limb_item_split(a, a.items[it], lane, warp, lead, yb, stages);
  }
}

}  // namespace

// raises the kernel's shared-memory limit, when a layout is built
cudaError_t limb_configure(int kc) {
  return cudaFuncSetAttribute(kc == 3 ? solve_limbs_split_kernel : solve_limbs_kernel,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kSmemWarp);
}

// poles per window: kc per lane; 3: one per lane, a CTA per window
int limb_window(int kc) { return kc == 2 ? 64 : 32; }
namespace {
int blocks_of(const Plan &pl) { return (pl.P + kBlock - 1) / kBlock; }
size_t inv_bytes(const Plan &pl) { return (size_t)(pl.nrows + (int64_t)pl.sys.size()) * blocks_of(pl) * kRec; }
size_t scale_bytes(const Plan &pl) { return (size_t)pl.nrows * 6 * sizeof(double); }
int *block_exponents(const Plan &pl, const DigitFactors &D) { return reinterpret_cast<int *>(D.scale + (size_t)pl.nrows * 6); }
}  // namespace
size_t limb_factor_bytes(const Plan &pl) {
  return (size_t)pl.nrows * blocks_of(pl) * (kRec + kBwd) + inv_bytes(pl) + scale_bytes(pl) +
         (size_t)blocks_of(pl) * (kBlock * sizeof(int4) + sizeof(int));
}
size_t limb_state_bytes(const Plan &pl, int B) { return (size_t)pl.nrows * B * (4 * sizeof(int4) + sizeof(int)); }

// The exponent of the reciprocals' limbs: |1/s| <= 1/|Re alpha| < 2^(e0 + 1), and 1 (delta's weight)
// below it as well.
int limb_exponent(const Plan &pl) {
  double least = 1.0;
  for (const cplx &a : pl.alpha) least = std::min(least, std::fabs(a.real()));
  return least > 0.0 ? std::max(0, std::ilogb(1.0 / least)) : kMaxSpread + 1;
}

// The factor set as limbs, in the limb_factor_bytes at D.fwd; `bad` set where it does not serve.
cudaError_t launch_limb_factors(Plan &pl, bool adjoint, const double2 *fac, DigitFactors &D, int *bad) {
  const size_t nrec = (size_t)pl.nrows * blocks_of(pl);
  D.bwd = D.fwd + nrec * kRec;
  D.inv = D.bwd + nrec * kBwd;
  D.inv_alpha = reinterpret_cast<int4 *>(D.inv + inv_bytes(pl));
  D.scale = reinterpret_cast<double *>(D.inv_alpha + (size_t)blocks_of(pl) * kBlock);  // every part a multiple of 16 B so far
  SetupArgs a;
  a.fac = fac;
  a.alpha = pl.alpha_dev;
  a.coef = pl.coef_dev;
  a.sys = pl.sys_dev;
  a.fwd = D.fwd;
  a.bwd = D.bwd;
  a.inv = D.inv;
  a.inv_alpha = D.inv_alpha;
  a.eblk = block_exponents(pl, D);
  a.scale = D.scale;
  a.bad = bad;
  a.P = pl.P;
  a.nblk = blocks_of(pl);
  a.N = pl.N;
  a.e0 = D.e0 = limb_exponent(pl);
  a.adjoint = adjoint;
  a.nrows = pl.nrows;
  a.tau = pl.prm.tau;
  a.q = 2.0 * pl.prm.omega * pl.prm.tau;
  a.phibar = pl.prm.gravity * pl.prm.mean_depth;
  if (a.e0 > kMaxSpread) return cudaMemsetAsync(bad, 1, 1, 0);
  const cudaError_t e = cudaMemsetAsync(a.eblk, 0x80, blocks_of(pl) * sizeof(int), 0);  // a very negative number
  if (e != cudaSuccess) return e;
  limb_factor_kernel<<<dim3((unsigned)((pl.lmax + 1) * a.nblk), (unsigned)pl.sys.size()), kBlock>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_limb_state(Plan &pl, bool adjoint, const double2 *sin, bool by_state, int B, unsigned *counter,
                              cudaStream_t st) {
  StateArgs s;
  s.sin = sin;
  s.sys = pl.sys_dev;
  s.scale = (adjoint ? pl.dig_adj : pl.dig_fwd).scale;
  s.dig = reinterpret_cast<int4 *>(pl.dig_state);
  s.uexp = reinterpret_cast<int *>(pl.dig_state + (size_t)pl.nrows * B * 4 * sizeof(int4));
  s.counter = counter;
  s.nspec = pl.nspec;
  s.place = by_state ? 1 : B;
  s.state = by_state ? 3 * pl.nspec : 1;
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
  a.inv = D.inv;
  a.inv_alpha = D.inv_alpha;
  a.e0 = D.e0;
  a.eblk = block_exponents(pl, D);
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
  a.nblk = blocks_of(pl);
  a.lmax = pl.lmax;
  a.kc = L.kc;
  a.sms = pl.num_sms;
  return a;
}

cudaError_t launch_solve_limbs(Plan &pl, const DigitLayout &L, bool adjoint, int B, cudaStream_t st) {
  const bool split = L.kc == 3;
  const unsigned ctas = (unsigned)std::max(1, std::min(pl.num_sms * kCtas, split ? L.nitems : (L.nitems + 3) / 4));
  (split ? solve_limbs_split_kernel : solve_limbs_kernel)<<<ctas, 128, 4 * kSmemWarp, st>>>(limb_sweep(pl, L, adjoint, B));
  return cudaGetLastError();
}

}  // namespace rexi
