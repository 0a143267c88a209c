// Host-side launch interface between the C ABI (gac.cu) and the kernel
// translation units (one per model kind, compiled in parallel).  Every kernel
// takes (const ModelConst, const RunArgs) and is launched with
// cudaLaunchKernel(ptr, ..., {&mc, &ra}, ...).
#pragma once
#include <cuda_runtime.h>

#include "mh_kernel.cuh"

namespace gac {

struct LaunchCfg {
    const void *fn;
    int grid;
    int block;     // threads per block
    int sampling;  // of them, those before the moment warps (speculative kernel)
    size_t smem;
};

// Per-kind kernels defined in mh_<kind>.cu: (precision, trace, kBlock or kHalfBlock)
const void *mh_ptr_monoexp(int prec, bool trace, int block);
const void *mh_ptr_mwi3(int prec, bool trace, int block);
const void *mh_ptr_smt(int prec, bool trace, int block, bool few_b);  // fewer than kAnchor b-values
const void *mh_ptr_axcal(int prec, bool trace, int block);
const void *mh_ptr_linear(int prec, bool trace, int block);
// In slices (mh_slice_kernel: further arguments ss, pos0, q), MIXED.
const void *mh_slice_ptr_mwi3();
const void *mh_slice_ptr_axcal();
// Lane-split kernels (mh_split.cuh): G = 2 or 4 lanes per chain, MIXED; all:
// moments over every post-burn-in state.
const void *mh_split_ptr_monoexp(int G, bool all);
const void *mh_split_ptr_mwi3(int G, bool all);
// Speculative kernels (mh_spec.cuh): trees of depth 2..5, MIXED.
const void *mh_spec_ptr_monoexp(int depth, bool all);
const void *mh_spec_ptr_mwi3(int depth, bool all);
const void *mh_spec_ptr_smt(int depth, bool all);
const void *mh_spec_ptr_axcal(int depth, bool all);

}  // namespace gac
