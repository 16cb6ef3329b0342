// Whole-filter-reuse data gradient of dense dL/dO, pruned inside the kernel.
#include "dgrad_halo.cuh"

namespace sdgp {

sdgp_status launch_halo_fused(int bn, int nt, const void* dO, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream) {
  return launch_halo<true, true>(bn, nt, dO, nullptr, Wt, view, p, stream);
}

cudaError_t take_error_halo_fused(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
