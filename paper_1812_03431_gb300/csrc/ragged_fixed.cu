// Ragged batches with the fixed-point solves: a persistent launch over the merged items of every
// plan of a kind (solve_limbs.cu for plans of up to five states, solve_digits.cu above), each
// item swept as its plan's own step would.  Before it each plan's inputs are put into fixed
// point, after it each plan's slots are summed.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "digit_sweep.h"
#include "limb_sweep.h"
#include "rexi_internal.h"

namespace rexi {

using digit_solve::DigitSweep;
using limb_solve::LimbSweep;

DigitSweep digit_sweep(Plan &pl, const DigitLayout &L, bool adjoint, int B);
LimbSweep limb_sweep(Plan &pl, const DigitLayout &L, bool adjoint, int B);

namespace {

struct View {
  int states;  // per warp: 8 digits, 1 limbs
  union {
    DigitSweep d;
    LimbSweep l;
  };
};
constexpr int kCtas = 4;
constexpr int kViewBytes = (sizeof(View) + 15) / 16 * 16;
constexpr int kWarpBytes = limb_solve::kSmemWarp + kViewBytes;

template <bool DIGITS>
__global__ void __launch_bounds__(128, kCtas)
    ragged_fixed_kernel(const View *views, const int4 *items, const int *plan_of, int nitems, unsigned *counter, double2 *ybuf,
                        int lmax) {
  extern __shared__ __align__(16) char smem_all[];
  const int lane = threadIdx.x & 31;
  const int wslot = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  double2 *yb = ybuf + (int64_t)wslot * lmax * 64 + lane;
  char *smem = smem_all + (threadIdx.x >> 5) * kWarpBytes;
  View *view = reinterpret_cast<View *>(smem + limb_solve::kSmemWarp);
  int have = -1;
  for (;;) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(counter, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= (unsigned)nitems) break;
    const int p = plan_of[it];
    if (p != have) {  // the item's plan, into the warp's shared memory
      __syncwarp();
      for (int i = lane; i < (int)(sizeof(View) / 4); i += 32)
        reinterpret_cast<int *>(view)[i] = reinterpret_cast<const int *>(views + p)[i];
      __syncwarp();
      have = p;
    }
    const int4 item = items[it];
    if constexpr (DIGITS) digit_solve::digit_item(view->d, item, lane, yb, smem);
    else limb_solve::limb_item(view->l, item, lane, yb, smem);
  }
}

}  // namespace

void free_fixed_ragged(FixedRagged &R) {
  if (R.views_dev) cudaFree(R.views_dev);
  if (R.items_dev) cudaFree(R.items_dev);
  R = FixedRagged{};
}

// False where a plan has no fixed-point factors, or where the tiles' padding makes the fused
// solve the cheaper one: per row and pole a digit tile costs about 8 x 12 FP64 FMAs' time
// whatever its states, limbs 14 per state, the fused solve 39 per state
// (T170: 8 states 1.25 ms, 4 states 0.80, fused 0.52 per state).  Over 170 random calls (one to eight
// states of one to three plans, T10 to T250, 55 to 535 poles) the choice took 0.10 to 1.06 times the fused
// launch's time, median 0.28.  Limbs hold two poles per lane here whatever the windows: the launch
// has every plan's items.
bool build_fixed_ragged(const std::vector<Plan *> &plans, const std::vector<int> &counts, FixedRagged &R) {
  R = FixedRagged{};
  double fixed_cost = 0, fused_cost = 0, work[9] = {};  // per kind: states per warp
  auto kind = [&](size_t p) { return plans[p]->limbs ? 1 : 8; };
  for (size_t p = 0; p < plans.size(); ++p) {
    const int c = counts[p];
    if (c == 0) continue;
    const Plan &pl = *plans[p];
    if (!pl.dig_fwd.fwd || pl.nrows == 0 || c > pl.prm.max_batch) return false;
    const double rows = (double)pl.nrows * pl.P;
    fixed_cost += rows * (pl.limbs ? 14.0 * c : 96.0 * ((c + 7) / 8));
    fused_cost += rows * 39.0 * c;
    work[kind(p)] += (double)digit_work(pl, c, 2);
  }
  if (fixed_cost >= fused_cost) return false;
  R.layouts.resize(plans.size());
  std::vector<View> views(plans.size());
  struct Tagged { DigitItem it; int plan; };
  std::vector<Tagged> all;
  int num_sms = 1;
  for (size_t p = 0; p < plans.size(); ++p) num_sms = std::max(num_sms, plans[p]->num_sms);
  for (size_t p = 0; p < plans.size(); ++p) {
    const int c = counts[p];
    if (c == 0) continue;
    Plan &pl = *plans[p];
    std::vector<DigitItem> items;
    if (!digit_items(pl, c, 0, 0.5 * work[kind(p)] / (4.0 * kCtas * num_sms), R.layouts[p], items)) return false;
    for (const DigitItem &it : items) all.push_back(Tagged{it, (int)p});
    views[p].states = kind(p);
    if (pl.limbs) views[p].l = limb_sweep(pl, R.layouts[p], false, c);
    else views[p].d = digit_sweep(pl, R.layouts[p], false, c);
    R.lmax = std::max(R.lmax, pl.lmax);
  }
  // one kind of sweep after the other, in a launch each, longest first within it: warps that run
  // different sweeps side by side miss the instruction caches (48 states, T63 to T341: 19.6 ms with
  // all items longest first), and one kernel that calls both spills in either (12.5 ms;
  // two 11.0)
  std::stable_sort(all.begin(), all.end(), [&](const Tagged &x, const Tagged &y) {
    const int kx = views[x.plan].states, ky = views[y.plan].states;
    return kx != ky ? kx > ky : x.it.work > y.it.work;
  });
  std::vector<int4> items;
  std::vector<int> plan_of;
  for (const Tagged &t : all) {
    items.push_back(t.it.it);
    plan_of.push_back(t.plan);
  }
  R.nitems = (int)items.size();
  R.ndigits = (int)std::count_if(all.begin(), all.end(), [&](const Tagged &t) { return views[t.plan].states == 8; });
  const size_t n = items.size();
  cudaError_t e = cudaMalloc(&R.views_dev, views.size() * sizeof(View));
  if (e == cudaSuccess) e = cudaMalloc(&R.items_dev, n * (sizeof(int4) + sizeof(int)));
  if (e == cudaSuccess) e = cudaMemcpy(R.views_dev, views.data(), views.size() * sizeof(View), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(R.items_dev, items.data(), n * sizeof(int4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(R.items_dev + n, plan_of.data(), n * sizeof(int), cudaMemcpyHostToDevice);
  for (auto k : {ragged_fixed_kernel<true>, ragged_fixed_kernel<false>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kWarpBytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    free_fixed_ragged(R);
    return false;
  }
  return true;
}

// every plan's s_in -> s_out; ybuf: [resident warps][lmax of the ragged object][2][32]
cudaError_t launch_fixed_ragged(const std::vector<Plan *> &plans, const std::vector<int> &counts, const FixedRagged &R,
                                double2 *ybuf, unsigned *counter, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  int num_sms = 1;
  for (size_t p = 0; p < plans.size() && e == cudaSuccess; ++p) {
    num_sms = std::max(num_sms, plans[p]->num_sms);
    if (counts[p] > 0) e = launch_digit_state(*plans[p], false, plans[p]->s_in, false, counts[p], nullptr, st);
  }
  if (e != cudaSuccess) return e;
  for (int kind = 0; kind < 2 && e == cudaSuccess; ++kind) {
    const int first = kind == 0 ? 0 : R.ndigits, n = kind == 0 ? R.ndigits : R.nitems - R.ndigits;
    if (n == 0) continue;
    e = cudaMemsetAsync(counter, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    (kind == 0 ? ragged_fixed_kernel<true> : ragged_fixed_kernel<false>)<<<
        (unsigned)std::min(num_sms * kCtas, (n + 3) / 4), 128, 4 * kWarpBytes, st>>>(
        static_cast<const View *>(R.views_dev), R.items_dev + first,
        reinterpret_cast<const int *>(R.items_dev + R.nitems) + first, n, counter, ybuf, R.lmax);
    e = cudaGetLastError();
  }
  for (size_t p = 0; p < plans.size() && e == cudaSuccess; ++p)
    if (counts[p] > 0)
      e = launch_finish_digits(*plans[p], R.layouts[p], false, plans[p]->s_in, plans[p]->s_out, false, counts[p], st);
  return e;
}

}  // namespace rexi
