// Instantiations of the speculative MH kernel for GAC_MODEL_AXCAL_SMT (MIXED, trees
// of depth 2 to 5, thinned moments and moments over every post-burn-in state).
#include "launch.h"
#include "mh_spec.cuh"

namespace gac {

const void *mh_spec_ptr_axcal(int depth, bool all) { return spec_kernel_ptr<GAC_MODEL_AXCAL_SMT>(depth, all); }

}  // namespace gac
