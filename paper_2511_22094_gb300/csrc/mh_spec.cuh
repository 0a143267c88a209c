// Speculative one-launch Metropolis-Hastings kernel (mcmc.m hot path, Sec.
// 2.2.2) for problems with too few chains to fill the GPU.
//
// A chain's iterations are serial only through its accept/reject decisions:
// the random numbers are keyed by (seed, t, voxel, chain), so the proposal of
// iteration t+1 is known up to which of two states it starts from.  Here a
// chain owns G = 2^D consecutive lanes of a warp and a round advances it by D
// iterations: lane n >= 1 is node n of the binary tree of decisions (root 1;
// node n's children are 2n, n's proposal rejected, and 2n + 1, accepted).
// Every node builds its own proposal from the round's start state along its
// path, evaluates its likelihood, and takes its decision against the
// likelihood of its nearest accepted ancestor -- all nodes at once.  The
// decisions then select one path through the tree; its D nodes are exactly the
// D iterations the one-thread kernel would have run, computed by the same
// functions from the same values, so every output equals mh_kernel's (MIXED)
// bit for bit.  Lane 0 stands for the round's start state.
//  - Philox calls are dealt over the lanes: item i = k n_calls + call of the
//    next round's iteration k belongs to lane i mod G, which also takes its
//    Box-Muller pairs; the nodes fetch the normals by shuffle.
//  - Rounds end at the burn-in adaptation's windows (and at the last
//    iteration), so all chains stay at the same t.
//  - Lane g stores the samples of parameters g, g + G, ... and keeps their
//    MIXED block partials.  The FP64 Welford updates run on moment warps
//    (moment_warps.cuh); at depth 2, whose warps fill the schedulers, lane g
//    keeps those too.
//
// What bounds it: a lone warp per scheduler issues its instructions in turn
// and waits out every latency (ncu, AxCaliberSMT at depth 5: 1,260 instructions
// a round, one issued every 2.6 cycles), so a round costs little more than one
// iteration of mh_kernel does there, but advances D iterations instead of one.
// The work per iteration grows by 2^D / D, so the host (choose_depth in
// gac.cu) takes the deepest tree whose warps still fit the idle issue slots.
// Measured on GB300, before -> with it: AxCaliberSMT, 100 voxels x 4 chains x
// 25,000 iterations (depth 5): 41.4 -> 7.94 ms; 3-pool, 301 voxels x 4 x 5,000,
// host arrays (depth 4): 5.59 -> 1.58 ms; SMT, 600 chains x 1,000 (depth 5): 0.59 ->
// 0.15 ms.
//
// Scope (the host checks it and otherwise launches mh_kernel): MIXED
// precision, one launch per job, no trace.
#pragma once
#include "mh_split.cuh"
#include "moment_warps.cuh"

namespace gac {

// Threads per block: 8 warps; the deeper trees run with at most 8 warps an SM.
constexpr int kSpecBlock = 256;

// Shared-memory bytes of a block of `threads` threads: the Welford
// accumulators, the measurement tile, and for moments over every post-burn-in
// state the block partials and the rows the states are exchanged through
// (`threads`: the sampling threads), or the moment warps' ring.
__host__ __device__ constexpr int spec_row(int P) { return P | 1; }  // odd: a warp's rows start in distinct banks
__host__ __device__ constexpr bool spec_moment_warps(int depth, bool all) { return depth >= 3 && !all; }
__host__ __device__ inline size_t spec_smem_bytes(int P, int G, int threads, int VB, int row_stride, bool all, bool ring) {
    return tile_smem_bytes(P, sizeof(double), VB, row_stride, true, all, threads / G) +
           (all ? static_cast<size_t>(threads) * spec_row(P) * sizeof(float) : 0) +
           (ring ? moment_ring_bytes(P * (threads / G)) : 0);
}

// The draws of one round: lane g holds items g, g + G, ... (Philox call i %
// n_calls of the round's iteration i / n_calls), each as up to two Box-Muller
// pairs in parts (bm_prefix) and the word that is the acceptance word where
// the item holds it.
template <int P, int D>
struct SpecDraw {
    static constexpr int G = 1 << D;
    static constexpr int NC = n_calls(P);
    static constexpr int CPL = (D * NC + G - 1) / G;       // items per lane
    static constexpr int PAIRS = (P + 1) / 2 < 2 ? 1 : 2;  // Box-Muller pairs per item
    static constexpr int ACALL = (n_words(P) - 1) / 4;     // the call and word of the acceptance uniform
    static constexpr int AWORD = (n_words(P) - 1) % 4;
    float lg[CPL][PAIRS], sn[CPL][PAIRS], cs[CPL][PAIRS];
    float lu[CPL];
    uint32_t w_acc[CPL];

    // iterations t0 + 1 .. t0 + D
    __device__ __forceinline__ void draw(uint32_t t0, int g, uint32_t vg, uint32_t c, uint32_t k0, uint32_t k1) {
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
            const int item = g + j * G;
            const uint32_t k = static_cast<uint32_t>(item / NC), call = static_cast<uint32_t>(item - NC * static_cast<int>(k));
            const Words4 w = philox4x32_10(t0 + 1u + k, vg, (c << 8) | call, 0u, k0, k1);
#pragma unroll
            for (int i = 0; i < PAIRS; ++i) bm_prefix(w.w[2 * i], w.w[2 * i + 1], lg[j][i], sn[j][i], cs[j][i]);
            w_acc[j] = w.w[AWORD];
            lu[j] = __logf(u01_f(w_acc[j]));
        }
    }
};

// One tile of voxels, all I iterations.
template <int KIND, int D, bool ALL>
__device__ __forceinline__ void run_tile_spec(const ModelConst &mc, const RunArgs &ra, int64_t tile,
                                              unsigned char *smem) {
    constexpr int P = model_n_par(KIND);
    constexpr int G = 1 << D;
    constexpr uint32_t kGroup = G == 32 ? 0xffffffffu : (1u << G) - 1u;
    using Draw = SpecDraw<P, D>;
    constexpr bool kHelp = spec_moment_warps(D, ALL);
    const int nthr = blockDim.x;
    const int nsamp = kHelp ? ra.sampling_threads : nthr;
    const int CB = nsamp / G;  // chain slots of the block
    const int tid = threadIdx.x;
    const int C = ra.C;
    const int VB = ra.vox_per_block;
    const int M = mc.n_meas;
    const int slot = tid / G, g = tid & (G - 1);
    const int lane0 = (tid & 31) & ~(G - 1);  // first lane of this chain's group
    const int lv = slot / C, c = slot - lv * C;
    const int64_t v0 = tile * VB;
    const int64_t left = ra.n_vox - v0;
    const int nv = left < VB ? static_cast<int>(left) : VB;
    const bool active = tid < nsamp && slot < VB * C && lv < nv;
    double *wf_mean = reinterpret_cast<double *>(smem);
    double *wf_m2 = wf_mean + P * CB;
    float *ytile = reinterpret_cast<float *>(wf_m2 + P * CB);
    float *bs = ytile + VB * ra.row_stride;  // ALL: FP32 block partials s1 [P][CB], s2, reference
    float *exch = bs + 3 * P * CB;           // ALL: the nodes' proposals [thread][spec_row(P)]
    // the moment warps' ring: the sampling warps with a chain are the first ones
    const MomentRing mom{bs, P * CB, ra.S, (nv * C * G + 31) / 32 * 32 + nthr - nsamp};

    // a1: stage measurements of voxels [v0, v0 + nv) (and the model's table)
    __syncthreads();
    model_smem_load<KIND>(mc);
    {
        const float *src = ra.data + v0 * M;
        const int total = nv * M;
        for (int i = tid; i < total; i += nthr) {
            const int row = i / M, col = i - row * M;
            ytile[row * ra.row_stride + col] = __ldg(src + i);
        }
    }
    __syncthreads();

    // lanes without a chain of their own follow voxel v0's chain 0 (writing
    // nothing), so that every shuffle sees a converged warp; warps without
    // any chain skip the iterations
    const int lvr = active ? lv : 0, cr = active ? c : 0;
    const int64_t v = v0 + lvr;
    const float *y = ytile + lvr * ra.row_stride;
    const float sig = ra.sigma ? __ldg(ra.sigma + v) : ra.sigma_scalar;
    const float inv_s2 = 1.0f / (sig * sig);
    const uint32_t vg = static_cast<uint32_t>(ra.voxel_base + static_cast<uint64_t>(v));
    const uint32_t cu = static_cast<uint32_t>(cr);
    const int64_t ch = v * C + cr;

    // this lane's node: its level, the accept bits of its path, the lane of
    // its nearest accepted ancestor (0: the start state), and the decisions
    // its ancestors must have taken for the path to reach it
    const int node = g;
    const int lvl = 31 - __clz(node);  // -1 for lane 0
    const int tz = node > 0 ? __ffs(node) - 1 : 0;
    const int anc = node > 0 && (node >> tz) != 1 ? node >> (tz + 1) : 0;
    uint32_t anc_mask = 0, anc_want = 0;
    for (int a = node; a > 1; a >>= 1) {
        anc_mask |= 1u << (a >> 1);
        anc_want |= static_cast<uint32_t>(a & 1) << (a >> 1);
    }
    // level k's accept bit of the path (bits below the leading one, the
    // deepest level last)
    auto path_bit = [&](int k) { return k < lvl && ((node >> (lvl - 1 - k)) & 1); };

    int n_acc = 0, n_bad = 0, ad_e = 0;
    if (kHelp && tid >= nsamp) {
        constexpr int kSeries = P * (kSpecBlock / G);  // at most
        moment_warp_run<(kSeries + 32 * kMomMaxWarps - 1) / (32 * kMomMaxWarps)>(mom, tid - nsamp, nthr - nsamp, wf_mean, wf_m2);
    } else if (__any_sync(kFullMask, active)) {
        // a2: initial state
        float th[P];
        if (ra.x0) {
            const float *x0 = ra.x0 + ch * P;
#pragma unroll
            for (int p = 0; p < P; ++p) th[p] = fminf(fmaxf(x0[p], mc.lb_f[p]), mc.ub_f[p]);
        } else {
            uint32_t w0[4 * ((P + 3) / 4)];
            draw_words(w0, kInitIteration, vg, cu, ra.k0, ra.k1);
#pragma unroll
            for (int p = 0; p < P; ++p) th[p] = fmaf(mc.ub_f[p] - mc.lb_f[p], u01_f(w0[p]), mc.lb_f[p]);
        }
        float L = loglik_f<KIND, KahanSum>(th, y, inv_s2, mc);
        if (!kHelp && active) {
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (p % G == g) {
                    wf_mean[p * CB + slot] = 0.0;
                    wf_m2[p * CB + slot] = 0.0;
                }
        }
        int ad_acc0 = 0, n_mom = 0, blk_n = 0;
        // thinned moments without moment warps: lane g's parameters p = g + kG in registers, each
        // update's second half deferred to the next event (as in the
        // lane-split kernel: two short FP64 chains instead of one long one)
        constexpr int PL = (P + G - 1) / G;
        double wm[PL], wm2[PL], wxd[PL], wd[PL];
#pragma unroll
        for (int k = 0; k < PL; ++k) wm[k] = wm2[k] = wxd[k] = wd[k] = 0.0;
        bool wpend = false;
        int to_thin = ra.S > 0 ? ra.B + ra.T : INT_MAX, n_thin = 0;  // B + S T <= I: no overflow
        const int W_ad = ra.adapt_window;
        int to_adapt = (W_ad > 0 && W_ad <= ra.B) ? W_ad : INT_MAX;
        float bm_k = adapt_bm_scale<float>(ad_e);

        Draw dr;
        dr.draw(0u, g, vg, cu, ra.k0, ra.k1);
        float zz[Draw::CPL][2 * Draw::PAIRS];
        auto normals = [&]() {
#pragma unroll
            for (int j = 0; j < Draw::CPL; ++j)
#pragma unroll
                for (int i = 0; i < Draw::PAIRS; ++i)
                    bm_finish(dr.lg[j][i], dr.sn[j][i], dr.cs[j][i], bm_k, zz[j][2 * i], zz[j][2 * i + 1]);
        };
        normals();

        // this round's proposals and acceptance words, and the next round's
        // draws: both are made behind the previous round's decisions, where
        // the draws (independent of them) fill the latency of the shuffles and
        // of the proposals' serial path
        float prop[P], lu;
        uint32_t w_acc;
        auto round_len = [&](int t) { return min(D, min(ra.I, to_adapt) - t); };  // the same for every lane
        auto next_round = [&](int t) {
            // a4: this node's proposal: the start state moved along its path
            float thn[P];
#pragma unroll
            for (int p = 0; p < P; ++p) prop[p] = thn[p] = th[p];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const bool mine = k <= lvl, bit = path_bit(k);
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const int item = k * Draw::NC + p / 4;  // constant after unrolling
                    const float z = __shfl_sync(kFullMask, zz[item / G][p & 3], lane0 + item % G);
                    const float cand = fminf(fmaxf(fmaf(mc.step_f[p], z, thn[p]), mc.lb_f[p]), mc.ub_f[p]);
                    prop[p] = mine ? cand : prop[p];
                    if (k + 1 < D) thn[p] = bit ? cand : thn[p];
                }
            }
            // the acceptance word of this node's iteration
            const int aitem = max(lvl, 0) * Draw::NC + Draw::ACALL;
            lu = __shfl_sync(kFullMask, dr.lu[0], lane0 + (aitem & (G - 1)));
            w_acc = __shfl_sync(kFullMask, dr.w_acc[0], lane0 + (aitem & (G - 1)));
#pragma unroll
            for (int j = 1; j < Draw::CPL; ++j) {
                const float l2 = __shfl_sync(kFullMask, dr.lu[j], lane0 + (aitem & (G - 1)));
                const uint32_t w2 = __shfl_sync(kFullMask, dr.w_acc[j], lane0 + (aitem & (G - 1)));
                lu = aitem / G == j ? l2 : lu;
                w_acc = aitem / G == j ? w2 : w_acc;
            }
            dr.draw(static_cast<uint32_t>(t + round_len(t)), g, vg, cu, ra.k0, ra.k1);
            normals();
        };
        next_round(0);

        for (int t0 = 0; t0 < ra.I;) {
            const int valid = round_len(t0);
            // a5 + a6: forward model and likelihood, every node its own
            const float Le = loglik_f<KIND, KahanSum>(prop, y, inv_s2, mc);
            const float Lp = node == 0 ? L : Le;
            // a7: accept_mixed against the likelihood of the state before this
            // node; a near decision (rare) is taken in FP64
            const float Lb = __shfl_sync(kFullMask, Lp, lane0 + anc);
            const float d32 = Lp - Lb;
            const float margin = fmaf(0x1p-22f, fabsf(d32), 1e-5f);
            const float gap = d32 - lu;
            bool acc = gap > 0.0f;
            if (__builtin_expect(!(fabsf(gap) > margin), 0))
                acc = log(u01_d(w_acc)) < static_cast<double>(Lp) - static_cast<double>(Lb);
            // the path: nodes whose ancestors decided as their path says
            const uint32_t bits = (__ballot_sync(kFullMask, acc) >> lane0) & kGroup;
            const bool onpath = node > 0 && lvl < valid && (bits & anc_mask) == anc_want;
            n_bad += onpath && !isfinite(Lp);
            const uint32_t am = bits & (__ballot_sync(kFullMask, onpath) >> lane0) & kGroup;  // accepted, on the path
            // the lane that holds the state after level l (0: the start state)
            auto state_lane = [&](int l) {
                const uint32_t upto = am & ((2u << ((2 << l) - 1)) - 1u);
                return lane0 + (upto ? 31 - __clz(upto) : 0);
            };
            n_acc += __popc(am);
            const int t1 = t0 + valid;
            // a8: thinning grid and moments
            if (to_thin <= t1) {  // the same for every lane
                do {
                    const int src = state_lane(to_thin - t0 - 1);
                    float x[PL] = {};
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        const float xp = __shfl_sync(kFullMask, prop[p], src);
                        if (p % G == g) x[p / G] = xp;
                    }
                    if (ra.samples && active) {
                        const int sidx = (to_thin - ra.B) / ra.T - 1;
                        float *dst = ra.samples + ((static_cast<int64_t>(sidx) * C + c) * P) * ra.n_vox + v;
#pragma unroll
                        for (int k = 0; k < PL; ++k)
                            if (g + k * G < P) dst[(g + k * G) * ra.n_vox] = x[k];
                    }
                    if constexpr (kHelp) {
                        __syncwarp();
                        mom.open(n_thin);
                        float *ev = mom.at(n_thin);
#pragma unroll
                        for (int k = 0; k < PL; ++k)
                            if (g + k * G < P) ev[(g + k * G) * CB + slot] = x[k];
                        mom.close(n_thin);
                    } else if constexpr (!ALL) {
                        ++n_mom;
                        const double inv_n = inv_count<double, true>(n_mom);
                        if (g < P) {
#pragma unroll
                            for (int k = 0; k < PL; ++k) {
                                if (wpend) wm2[k] = welford_fma(wd[k], wxd[k] - wm[k], wm2[k]);
                                wxd[k] = static_cast<double>(x[k]);
                                wd[k] = wxd[k] - wm[k];
                                wm[k] = welford_fma(wd[k], inv_n, wm[k]);
                            }
                        }
                        wpend = true;
                    }
                    to_thin = ++n_thin < ra.S ? to_thin + ra.T : INT_MAX;
                } while (to_thin <= t1);
            }
            if constexpr (ALL) {
                if (t1 > ra.B) {
                    float *row = exch + tid * spec_row(P);
                    __syncwarp();
#pragma unroll
                    for (int p = 0; p < P; ++p) row[p] = prop[p];
                    __syncwarp();
                    float *s1 = bs + slot, *s2 = bs + P * CB + slot, *ref = bs + 2 * P * CB + slot;
#pragma unroll
                    for (int l = 0; l < D; ++l) {
                        const int t = t0 + 1 + l;
                        if (l >= valid || t <= ra.B) continue;  // the same for every lane
                        const float *xr = exch + ((tid & ~31) + state_lane(l)) * spec_row(P);
#pragma unroll
                        for (int k = 0; k < PL; ++k) {
                            const int p = g + k * G;
                            if (p < P) {
                                if (blk_n == 0) {
                                    ref[p * CB] = xr[p];
                                    s1[p * CB] = 0.0f;
                                    s2[p * CB] = 0.0f;
                                } else {
                                    const float dd = xr[p] - ref[p * CB];
                                    s1[p * CB] += dd;
                                    s2[p * CB] = fmaf(dd, dd, s2[p * CB]);
                                }
                            }
                        }
                        if (++blk_n == kMomBlock || t == ra.I) {
                            const double nb = blk_n, nn = static_cast<double>(n_mom) + nb;
                            const double inv_nb = 1.0 / nb, w_b = nb / nn, cross = static_cast<double>(n_mom) * w_b;
#pragma unroll
                            for (int k = 0; k < PL; ++k) {
                                const int p = g + k * G;
                                if (p < P && active) {
                                    const double a = s1[p * CB];
                                    const double mb = static_cast<double>(ref[p * CB]) + a * inv_nb;
                                    const double m2b = fma(-a, a * inv_nb, static_cast<double>(s2[p * CB]));
                                    const double m = wf_mean[p * CB + slot];
                                    const double delta = mb - m;
                                    wf_mean[p * CB + slot] = fma(delta, w_b, m);
                                    wf_m2[p * CB + slot] += fma(delta * delta, cross, m2b);
                                }
                            }
                            n_mom += blk_n;
                            blk_n = 0;
                        }
                    }
                }
            }
            // the state after the round
            const int end = lane0 + (am ? 31 - __clz(am) : 0);
#pragma unroll
            for (int p = 0; p < P; ++p) th[p] = __shfl_sync(kFullMask, prop[p], end);
            L = __shfl_sync(kFullMask, Lp, end);
            t0 = t1;
            if (__builtin_expect(t0 == to_adapt, 0)) {  // a window of the burn-in adaptation ends (the same t for every lane)
                const int a = n_acc - ad_acc0;
                ad_e += (a > ra.adapt_hi && ad_e < GAC_ADAPT_EMAX) - (a < ra.adapt_lo && ad_e > GAC_ADAPT_EMIN);
                ad_acc0 = n_acc;
                bm_k = adapt_bm_scale<float>(ad_e);
                to_adapt = (W_ad <= ra.B - t0) ? t0 + W_ad : INT_MAX;
                normals();  // the next round takes the new steps
            }
            next_round(t0);
        }
        if constexpr (!ALL && !kHelp) {
            if (active && g < P) {
#pragma unroll
                for (int k = 0; k < PL; ++k)
                    if (g + k * G < P) {
                        if (wpend) wm2[k] = welford_fma(wd[k], wxd[k] - wm[k], wm2[k]);
                        wf_mean[(g + k * G) * CB + slot] = wm[k];
                        wf_m2[(g + k * G) * CB + slot] = wm2[k];
                    }
            }
        }
        // each lane counted its own node's non-finite likelihoods
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) n_bad += __shfl_xor_sync(kFullMask, n_bad, o);
    }
    if (active && g == 0) {
        if (ra.accept) ra.accept[c * ra.n_vox + v] = ra.I > 0 ? float(n_acc) / float(ra.I) : 0.0f;
        if (ra.nonfinite) ra.nonfinite[c * ra.n_vox + v] = n_bad;
        if (ra.step_scale) ra.step_scale[c * ra.n_vox + v] = exp2f(0.25f * static_cast<float>(ad_e));
    }

    // a9: pool the C chains of each voxel; the voxel's C * G threads take its
    // parameters in turn
    __syncthreads();
    if (active && (ra.mean || ra.std || ra.rhat)) {
        const int n_each = ALL ? max(ra.I - ra.B, 0) : ra.S;
        for (int p = c * G + g; p < P; p += C * G)
            pool_chains(wf_mean + p * CB + (slot - c), wf_m2 + p * CB + (slot - c), C, n_each,
                        ra.mean ? ra.mean + p * ra.n_vox + v : nullptr, ra.std ? ra.std + p * ra.n_vox + v : nullptr,
                        ra.rhat ? ra.rhat + p * ra.n_vox + v : nullptr);
    }
}

template <int KIND, int D, bool ALL>
__global__ void __launch_bounds__(kSpecBlock + (spec_moment_warps(D, ALL) ? 32 * kMomMaxWarps : 0), D == 2 ? 2 : 1) mh_spec_kernel(const ModelConst mc, const RunArgs ra) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    for (int64_t tile = blockIdx.x; tile < ra.n_tiles; tile += gridDim.x)
        run_tile_spec<KIND, D, ALL>(mc, ra, tile, smem_raw);
}

// The kernel for a tree of depth 2..5 (nullptr otherwise).
template <int KIND>
const void *spec_kernel_ptr(int depth, bool all) {
    switch (depth) {
    case 2: return all ? reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 2, true>) : reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 2, false>);
    case 3: return all ? reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 3, true>) : reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 3, false>);
    case 4: return all ? reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 4, true>) : reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 4, false>);
    case 5: return all ? reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 5, true>) : reinterpret_cast<const void *>(&mh_spec_kernel<KIND, 5, false>);
    default: return nullptr;
    }
}

}  // namespace gac
