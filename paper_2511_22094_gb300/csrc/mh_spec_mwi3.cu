// Instantiations of the speculative MH kernel for GAC_MODEL_MWI3 (MIXED, trees
// of depth 2 to 5, thinned moments and moments over every post-burn-in state).
#include "launch.h"
#include "mh_spec.cuh"

namespace gac {

const void *mh_spec_ptr_mwi3(int depth, bool all) { return spec_kernel_ptr<GAC_MODEL_MWI3>(depth, all); }

}  // namespace gac
