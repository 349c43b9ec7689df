// The choice of the cluster kernel and its radix schedules (clusterkern.hpp).
//
// The general kernel calls its line transforms (bigfft.cuh: fifteen register DFTs are too
// many to inline four times), and a call with its stages costs about 700 cycles more than
// inlined stages do; in FP32 its 16 warps leave 128 registers, and what is live across
// the call spills.  It pays where it replaces long stages: FP32 lines by single warps,
// factors 7, 11 and 13 (whose staged form is a direct sum), fewer stages where the lines
// are long enough.  The staged kernel takes the rest.  us an iteration, start of either
// form / general / staged, 3 loads: FP32 17^2 10.1 / 13.7 / 8.9, 27^2 10.8 / 13.4 / 10.5,
// 136^2 53.2 / 59.1 / 43.1, 26^2 19.8 / 15.2 / 19.6; FP64 60^2 27.9 / 35.7 / 27.6,
// 12 x 240 28.3 / 48.1 / 28.3, 100^2 64.1 / 55.8 / 63.5, 22^2 105.3 / 35.8 / 105.
#include <algorithm>

#include "bigsplit.hpp"
#include "clusterkern.hpp"

namespace fh {

namespace {

bool divides_any(int n, std::initializer_list<int> ps) {
  for (int p : ps)
    if (n % p == 0) return true;
  return false;
}

// one axis: `lines` lines of N points in a CTA of a cluster of 8.  Counted for clusters of
// 8 in either size, so that a solve's bits do not depend on the cluster that a batch or
// the tuner picks.
struct Axis {
  int N, lines;
  FftPlan plan, big, mid, tiny;   // radices to 8 of the staged form, to 16, to 8, to 4

  bool init(int n, int nlines) {
    N = n;
    lines = nlines;
    return make_plan(n, &plan) && make_big_plan(n, 16, &big) && make_big_plan(n, 8, &mid) && make_big_plan(n, 4, &tiny);
  }
  bool pow2() const { return (N & (N - 1)) == 0; }
  bool splits() const { return line_split(N).R1 > 0; }
  bool large_prime() const { return std::any_of(plan.r, plan.r + plan.np, [](int r) { return r > 13; }); }
  bool shorter() const { return big.np < plan.np; }
  // fewer stages, each with more butterflies than half of the CTA's 256 threads (an FP64
  // stage of fewer lasts one thread's butterfly, and a radix of 9 to 16 is a long one)
  bool long_stages() const {
    return shorter() && std::all_of(big.r, big.r + big.np, [this](int r) { return lines * (N / r) > 128; });
  }
  // An FP64 warp instruction takes its quarter of the SM 64 cycles whatever its lanes do,
  // so a small grid's stage lasts one thread's butterfly: radix 4 where there are at most
  // two points a thread (32^2: 19.6 -> 17.4 us an iteration).
  bool few_points() const { return lines * N <= 512; }
};

}  // namespace

bool cluster_choice(int N0, int L, int nv, bool fp32, ClusterChoice* out) {
  const int rows = (N0 + 7) / 8, cols = (L / 2 + 1 + 7) / 8;
  Axis a, b;
  if (!a.init(N0, nv * cols) || !b.init(L, (rows * nv + 1) / 2)) return false;
  const Axis* ax[2] = {&a, &b};
  FftPlan* plan[2] = {&out->plan0, &out->plan1};
  if (a.pow2() && b.pow2()) {
    out->kind = kClusterPow2;
    for (int q = 0; q < 2; ++q) *plan[q] = !fp32 && ax[q]->few_points() ? ax[q]->tiny : ax[q]->plan;
    return true;
  }
  bool general;
  if (fp32) {
    // lines by single warps, or 11 and 13 as register DFTs; else fewer (or cheaper: 7)
    // stages on grids large enough to pay for the calls (27 000 values a load), or as
    // many (200 = 8 5 5) on larger ones: 200^2 32.0 / 30.3 / 31.9, 125^2 18.5 / 19.6 / 18.3
    bool split = true, heavy = false, fewer = true;
    for (const Axis* x : ax) {
      if (x->splits()) continue;
      split = false;
      heavy = heavy || divides_any(x->N, {11, 13});
      fewer = fewer && (x->shorter() || x->N % 7 == 0);
    }
    general = split || (!a.large_prime() && !b.large_prime() && (heavy || (long long)nv * N0 * L >= (fewer ? 27000 : 100000)));
  } else {
    general = divides_any(N0, {7, 11, 13}) || divides_any(L, {7, 11, 13}) || (a.long_stages() && b.long_stages());
  }
  out->kind = general ? kClusterGeneral : kClusterStaged;
  for (int q = 0; q < 2; ++q) {
    const Axis& x = *ax[q];
    if (!fp32 && x.few_points()) *plan[q] = x.tiny;
    else if (!general) *plan[q] = x.plan;
    else *plan[q] = fp32 || x.long_stages() ? x.big : x.mid;
  }
  return true;
}

}  // namespace fh
