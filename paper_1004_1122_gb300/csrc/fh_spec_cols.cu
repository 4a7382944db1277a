// Column passes of the frequency-domain CG iteration.
#include "fh_spec_plans.cuh"

namespace fh {

cudaError_t spec_inv(int mode, const Launch& L, const SpecArgs& a, cudaStream_t st) {
  if (mode == kSpecFinish)
    return on_plan<PlanList<>, true>(a.plan, [&](auto t) {
      seq_launch(k_spec_inv<kSpecFinish, decltype(t)>, L, L.smem, st, a);
      return cudaGetLastError();
    });
  return on_plan<SpecPlans, true>(a.plan, [&](auto t) {
    seq_launch(k_spec_inv<kSpecUpdate, decltype(t)>, L, L.smem, st, a);
    return cudaGetLastError();
  });
}

cudaError_t spec_fwd(int mode, const Launch& L, const SpecArgs& a, cudaStream_t st) {
  if (mode == kSpecProject)
    return on_plan<PlanList<>, true>(a.plan, [&](auto t) {
      seq_launch(k_spec_fwd<kSpecProject, decltype(t)>, L, L.smem, st, a);
      return cudaGetLastError();
    });
  return on_plan<SpecPlans, true>(a.plan, [&](auto t) {
    seq_launch(k_spec_fwd<kSpecApply, decltype(t)>, L, L.smem, st, a);
    return cudaGetLastError();
  });
}

cudaError_t spec_green(const Launch& L, const SpecArgs& a, cudaStream_t st) {
  return on_plan<SpecPlans, true>(a.plan, [&](auto t) {
    seq_launch(k_spec_green<decltype(t)>, L, L.smem, st, a);
    return cudaGetLastError();
  });
}

cudaError_t spec_col_set_smem(const SpecArgs& a, size_t bytes) {
  cudaError_t e = on_plan<SpecPlans, true>(a.plan, [&](auto t) {
    cudaError_t e2 = opt_in_smem(k_spec_green<decltype(t)>, bytes);
    if (e2 == cudaSuccess) e2 = opt_in_smem(k_spec_inv<kSpecUpdate, decltype(t)>, bytes);
    return e2 == cudaSuccess ? opt_in_smem(k_spec_fwd<kSpecApply, decltype(t)>, bytes) : e2;
  });
  if (e != cudaSuccess) return e;
  return on_plan<PlanList<>, true>(a.plan, [&](auto t) {
    cudaError_t e2 = opt_in_smem(k_spec_inv<kSpecFinish, decltype(t)>, bytes);
    return e2 == cudaSuccess ? opt_in_smem(k_spec_fwd<kSpecProject, decltype(t)>, bytes) : e2;
  });
}

bool spec_col_ct(const FFTPlan& pl) { return plan_is_ct<SpecPlans>(pl); }

}  // namespace fh
