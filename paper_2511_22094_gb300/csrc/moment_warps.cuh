// Moment warps: the FP64 Welford updates of the speculative sampler
// (mh_spec.cuh) on warps of their own.
//
// GB300 issues 1.68 FP64 results per SM clock: a warp's FP64 instruction holds
// its scheduler's FP64 pipe for ~76 cycles, and an update is a chain of three of
// them (plus a conversion) from one thinned sample to the next.  Taken by the
// sampling warps, which have nothing else to hide it, an update cost ~650
// cycles, more than half of a round of the mono-exponential model.  Here the
// sampling warps drop the thinned states into a ring in shared memory, and
// moment warps at the end of the block, on schedulers that are idle otherwise,
// run the same updates in the same order, one series (parameter of a chain) a
// lane.  Measured, ms: mono-exponential, 100 chains x 1,000 iterations, thinning
// 1: 0.43 -> 0.30, 5: 0.20 -> 0.17; 3-pool, 600 voxels x 4 x 500, thinning 1:
// 0.45 -> 0.33, 5: 0.27 -> 0.24, 100: 0.227 -> 0.220.  (In the lane-split kernel
// the same change slowed the loop between the events by a third, for reasons in
// the code the compiler makes of it; it keeps its own updates.)
//
// The ring has two halves of kMomRing events.  Named barriers 1 and 2 (half
// full) and 3 and 4 (half free again) order them: sampling warps arrive at
// "full" and wait for "free" before they write a half again, moment warps the
// other way round.  Every event is known beforehand (S of them, at the same
// iterations for all chains), so each arrival has its wait.
#pragma once
#include "mh_kernel.cuh"

namespace gac {

constexpr int kMomRing = 8;      // events per half
constexpr int kMomMaxWarps = 4;  // moment warps of a block, at most

// (the forms that do not ask for a converged warp)
__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    asm volatile("barrier.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Moment warps for `series` series, and the ring's bytes.
__host__ __device__ inline int moment_warps(int series, int most) {
    const int w = (series + 31) / 32;
    return w < most ? w : most;
}
__host__ __device__ inline size_t moment_ring_bytes(int series) {
    return 2 * static_cast<size_t>(kMomRing) * series * sizeof(float);
}

// The sampling side.  Every lane of every sampling warp that has a chain calls
// open() and close() around its writes of event e = 0 .. S - 1, to at(e).
struct MomentRing {
    float *ring;   // [2][kMomRing][series]
    int series;
    int n_events;  // S
    int threads;   // of the sampling warps with a chain and the moment warps
    __device__ __forceinline__ float *at(int e) const { return ring + e % (2 * kMomRing) * series; }
    __device__ __forceinline__ void open(int e) const {
        if (e % kMomRing == 0 && e >= 2 * kMomRing) named_sync(3 + ((e / kMomRing) & 1), threads);
    }
    __device__ __forceinline__ void close(int e) const {
        if (e % kMomRing == kMomRing - 1 || e == n_events - 1) named_arrive(1 + ((e / kMomRing) & 1), threads);
    }
};

// A moment warp's run over all events: lane `lane` of `lanes` takes series lane,
// lane + lanes, ... (at most SPL of them) and leaves their means and sums of
// squared deviations in wf_mean, wf_m2 [series].
template <int SPL>
__device__ __forceinline__ void moment_warp_run(const MomentRing &mr, int lane, int lanes, double *wf_mean, double *wf_m2) {
    double m[SPL], m2[SPL];
#pragma unroll
    for (int k = 0; k < SPL; ++k) m[k] = m2[k] = 0.0;
    for (int e0 = 0, half = 0; e0 < mr.n_events; e0 += kMomRing, half ^= 1) {
        const int cnt = min(kMomRing, mr.n_events - e0);
        named_sync(1 + half, mr.threads);
        const float *x = mr.ring + half * kMomRing * mr.series;
#pragma unroll 2
        for (int i = 0; i < cnt; ++i) {
            const double inv_n = inv_count<double, true>(e0 + i + 1);
#pragma unroll
            for (int k = 0; k < SPL; ++k) {
                const int s = lane + k * lanes;
                if (s < mr.series) {
                    const double xd = static_cast<double>(x[i * mr.series + s]);
                    const double d = xd - m[k];
                    m[k] = welford_fma(d, inv_n, m[k]);
                    m2[k] = welford_fma(d, xd - m[k], m2[k]);
                }
            }
        }
        if (e0 + 2 * kMomRing < mr.n_events) named_arrive(3 + half, mr.threads);
    }
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
        const int s = lane + k * lanes;
        if (s < mr.series) {
            wf_mean[s] = m[k];
            wf_m2[s] = m2[k];
        }
    }
}

}  // namespace gac
