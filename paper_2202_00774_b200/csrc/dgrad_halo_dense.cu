// Whole-filter-reuse data gradient of dense dL/dO.
#include "dgrad_halo.cuh"

namespace sdgp {

sdgp_status launch_halo_dense(int bn, int nt, const void* A, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream) {
  return launch_halo<false, false>(bn, nt, A, nullptr, Wt, view, p, stream);
}

bool plan_halo_dense(int bn, int nt, HaloParams* p) { return plan_halo_shape<false>(bn, nt, p); }
cudaError_t take_error_halo_dense(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
