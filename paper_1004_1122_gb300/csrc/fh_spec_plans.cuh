// fh_spec_plans.cuh -- compile-time plans of the frequency-domain CG kernels
// and the dispatch on a run-time plan; included by the fh_spec_*.cu files.
//
// Which lengths: the odd lengths whose only prime factors are 3 and 5, from 75
// nodes (shorter axes belong to grids that launch latency bounds); each entry
// is the plan make_fft_plan picks for that length, in mirror_order.  Other
// lengths, and the small-radix plans of small grids, run the run-time-plan
// kernels.  Lengths with a factor 7 are left out to keep the compile time: some
// twenty-five more plans would instantiate three column, two middle and up to
// six row kernels each; what they would gain has not been measured.
#pragma once

#include "fh_launch_impl.cuh"

namespace fh {

template <typename... Ps> struct PlanList {};

using SpecPlans3D = PlanList<CPlan<25, 3>, CPlan<27, 3>, CPlan<25, 5>, CPlan<27, 5>, CPlan<25, 9>, CPlan<27, 9>>;
using SpecPlans = PlanList<CPlan<25, 3>, CPlan<27, 3>, CPlan<25, 5>, CPlan<27, 5>, CPlan<25, 9>, CPlan<27, 9>,
                           CPlan<25, 15>, CPlan<27, 15>, CPlan<25, 25>, CPlan<27, 25>, CPlan<27, 27>,
                           CPlan<25, 5, 9>, CPlan<27, 5, 9>, CPlan<25, 3, 25>, CPlan<27, 3, 25>, CPlan<27, 3, 27>>;

// Calls f(P{}) for the compile-time plan of the list that equals pl, or
// f(DynPlan{}) when there is none.
template <typename F>
static cudaError_t with_plan(const FFTPlan&, PlanList<>, F&& f) {
  return f(DynPlan{});
}
template <typename P, typename... Ps, typename F>
static cudaError_t with_plan(const FFTPlan& pl, PlanList<P, Ps...>, F&& f) {
  if (cplan_is<P>(pl)) return f(P{});
  return with_plan(pl, PlanList<Ps...>{}, f);
}

// f(tag) for the kernels that run plan pl.  Plans = PlanList<>: run-time plans
// only (the set-up passes).  X: extended plans are compiled (one load per launch).
template <typename Plans, bool X, typename F>
static cudaError_t on_plan(const FFTPlan& pl, F&& f) {
  if (pl.ext == kRadixExt) {
    if constexpr (X) return f(DynPlanX{});
    return cudaErrorInvalidValue;
  }
  if (pl.ext == kRadixSmall) return f(DynPlan9{});
  return with_plan(pl, Plans{}, f);
}

template <typename Plans> static bool plan_is_ct(const FFTPlan& pl) {
  bool ct = false;
  if (pl.ext == kRadixStd)
    with_plan(pl, Plans{}, [&](auto t) {
      ct = PlanLen<decltype(t)>::value > 0;
      return cudaSuccess;
    });
  return ct;
}

}  // namespace fh
