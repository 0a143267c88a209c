// Instantiations of the MH kernel for GAC_MODEL_SMT (all precisions, with and
// without step tracing, both block sizes, and for short protocols).
#include "launch.h"

namespace gac {

const void *mh_ptr_smt(int prec, bool trace, int block, bool few_b) {
    return few_b ? mh_kernel_ptr_of<GAC_MODEL_SMT, kFormMhShort>(prec, trace, block) : mh_kernel_ptr_of<GAC_MODEL_SMT>(prec, trace, block);
}

}  // namespace gac
