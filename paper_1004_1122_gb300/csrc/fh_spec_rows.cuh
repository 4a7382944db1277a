// fh_spec_rows.cuh -- launchers of the row pass of the frequency-domain CG
// iteration for one dimension; included by fh_spec_rows_d2.cu and _d3.cu.
#pragma once

#include "fh_spec_plans.cuh"

namespace fh {

template <int D, int NL, typename Plans> struct SpecRows {
  static constexpr bool kX = NL == 1;
  // a launch too large for the compile-time plan's thread limit runs the run-time plan
  template <typename F> static cudaError_t hot(const FFTPlan& pl, const Launch& L, F&& f) {
    return L.block <= kSpecRowCtThreads ? on_plan<Plans, kX>(pl, f) : on_plan<PlanList<>, kX>(pl, f);
  }
  // the load and add passes: compile-time plans for one load (the operator's
  // product), else run-time plans (twice per solve)
  template <typename F> static cudaError_t ends(const FFTPlan& pl, const Launch& L, F&& f) {
    if constexpr (NL == 1) return hot(pl, L, f);
    return on_plan<PlanList<>, kX>(pl, f);
  }
  static cudaError_t run(int mode, const Launch& L, const SpecRowArgs& a, cudaStream_t st) {
    if (mode == kSpecRowTau)
      return hot(a.plan, L, [&](auto t) {
        seq_launch(k_spec_row<D, NL, kSpecRowTau, decltype(t)>, L, L.smem, st, a);
        return cudaGetLastError();
      });
    return ends(a.plan, L, [&](auto t) {
      if (mode == kSpecRowLoad)
        seq_launch(k_spec_row<D, NL, kSpecRowLoad, decltype(t)>, L, L.smem, st, a);
      else
        seq_launch(k_spec_row<D, NL, kSpecRowAdd, decltype(t)>, L, L.smem, st, a);
      return cudaGetLastError();
    });
  }
  static cudaError_t set_smem(const SpecRowArgs& a, const Launch& L) {
    cudaError_t e = hot(a.plan, L, [&](auto t) { return opt_in_smem(k_spec_row<D, NL, kSpecRowTau, decltype(t)>, L.smem); });
    if (e != cudaSuccess) return e;
    return ends(a.plan, L, [&](auto t) {
      cudaError_t e2 = opt_in_smem(k_spec_row<D, NL, kSpecRowLoad, decltype(t)>, L.smem);
      return e2 == cudaSuccess ? opt_in_smem(k_spec_row<D, NL, kSpecRowAdd, decltype(t)>, L.smem) : e2;
    });
  }
  static bool ct(const FFTPlan& pl, const Launch& L) { return L.block <= kSpecRowCtThreads && plan_is_ct<Plans>(pl); }
};

}  // namespace fh
