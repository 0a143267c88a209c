// Instantiations of the MH kernel for GAC_MODEL_MONOEXP (all precisions, with and
// without step tracing, both block sizes) and of its lane-split form
// (MIXED, 2 or 4 lanes).
#include "launch.h"
#include "mh_split.cuh"

namespace gac {

const void *mh_ptr_monoexp(int prec, bool trace, int block) { return mh_kernel_ptr_of<GAC_MODEL_MONOEXP>(prec, trace, block); }
const void *mh_split_ptr_monoexp(int G, bool all) { return mh_split_kernel_ptr<GAC_MODEL_MONOEXP>(G, all); }

}  // namespace gac
