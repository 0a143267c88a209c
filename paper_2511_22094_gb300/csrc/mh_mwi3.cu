// Instantiations of the MH kernel for GAC_MODEL_MWI3 (all precisions, with and
// without step tracing, both block sizes, and in slices) and of its lane-split form
// (MIXED, 2 or 4 lanes).
#include "launch.h"
#include "mh_split.cuh"

namespace gac {

const void *mh_ptr_mwi3(int prec, bool trace, int block) { return mh_kernel_ptr_of<GAC_MODEL_MWI3>(prec, trace, block); }
const void *mh_slice_ptr_mwi3() { return reinterpret_cast<const void *>(&mh_slice_kernel<GAC_MODEL_MWI3>); }
const void *mh_split_ptr_mwi3(int G, bool all) { return mh_split_kernel_ptr<GAC_MODEL_MWI3>(G, all); }

}  // namespace gac
