// Middle-axis passes (3-D) of the frequency-domain CG iteration.
#include "fh_spec_plans.cuh"

namespace fh {

cudaError_t spec_mid(bool inv, const Launch& L, const SpecMidArgs& a, cudaStream_t st) {
  return on_plan<SpecPlans3D, true>(a.plan, [&](auto t) {
    if (inv)
      seq_launch(k_spec_mid<true, decltype(t)>, L, L.smem, st, a);
    else
      seq_launch(k_spec_mid<false, decltype(t)>, L, L.smem, st, a);
    return cudaGetLastError();
  });
}

cudaError_t spec_mid_set_smem(const SpecMidArgs& a, size_t bytes) {
  return on_plan<SpecPlans3D, true>(a.plan, [&](auto t) {
    cudaError_t e = opt_in_smem(k_spec_mid<true, decltype(t)>, bytes);
    return e == cudaSuccess ? opt_in_smem(k_spec_mid<false, decltype(t)>, bytes) : e;
  });
}

bool spec_mid_ct(const FFTPlan& pl) { return plan_is_ct<SpecPlans3D>(pl); }

}  // namespace fh
