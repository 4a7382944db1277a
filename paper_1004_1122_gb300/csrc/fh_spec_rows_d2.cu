// Row pass of the frequency-domain CG iteration, 2-D.
#include "fh_spec_rows.cuh"

namespace fh {
using R1 = SpecRows<2, 1, SpecPlans>;
using RN = SpecRows<2, 2, SpecPlans>;
cudaError_t spec_row_d2(int mode, const Launch& L, const SpecRowArgs& a, cudaStream_t st) {
  return a.g.nloads == 1 ? R1::run(mode, L, a, st) : RN::run(mode, L, a, st);
}
cudaError_t spec_row_d2_set_smem(const SpecRowArgs& a, const Launch& L) {
  return a.g.nloads == 1 ? R1::set_smem(a, L) : RN::set_smem(a, L);
}
bool spec_row_d2_ct(const FFTPlan& pl, const Launch& L) { return R1::ct(pl, L); }
}  // namespace fh
