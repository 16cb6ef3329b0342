// Whole-filter-reuse data gradient of compressed dL/dO.
#include "dgrad_halo.cuh"

namespace sdgp {

sdgp_status launch_halo_sparse(int bn, int nt, const void* A, const void* meta, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream) {
  return launch_halo<true, false>(bn, nt, A, meta, Wt, view, p, stream);
}

bool plan_halo_sparse(int bn, int nt, HaloParams* p) { return plan_halo_shape<true>(bn, nt, p); }
cudaError_t take_error_halo_sparse(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
