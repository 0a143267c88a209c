// Instantiations of the MH kernel for GAC_MODEL_AXCAL_SMT (all precisions, with and
// without step tracing, both block sizes, and in slices).
#include "launch.h"

namespace gac {

const void *mh_ptr_axcal(int prec, bool trace, int block) { return mh_kernel_ptr_of<GAC_MODEL_AXCAL_SMT>(prec, trace, block); }
const void *mh_slice_ptr_axcal() { return reinterpret_cast<const void *>(&mh_slice_kernel<GAC_MODEL_AXCAL_SMT>); }

}  // namespace gac
