// C ABI of libgac.so (include/gac.h): model registry, argument validation,
// host/device pointer handling and the launch of the persistent MH kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "gac.h"
#include "gac_internal.h"
#include "launch.h"
#include "mh_spec.cuh"

namespace gac {

// ------------------------------------------------------------ errors -------
static thread_local std::string g_last_error;

gac_status fail(gac_status st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return st;
}

gac_status cuda_fail(cudaError_t e, const char *what) {
    cudaGetLastError();  // clear a sticky launch error state where possible
    if (e == cudaErrorMemoryAllocation)
        return fail(GAC_ERR_OOM, "%s: %s", what, cudaGetErrorString(e));
    return fail(GAC_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

void clear_error() { g_last_error.clear(); }

// ----------------------------------------------------------- registry ------
static std::mutex g_reg_mu;
static std::vector<ModelConst> g_models;  // id = index + 1

gac_status model_get(int id, ModelConst *out) {
    std::lock_guard<std::mutex> lk(g_reg_mu);
    if (id < 1 || id > static_cast<int>(g_models.size()))
        return fail(GAC_ERR_UNKNOWN_MODEL, "unknown model id %d", id);
    *out = g_models[id - 1];
    return GAC_OK;
}

static bool all_finite(const double *a, int n) {
    for (int i = 0; i < n; ++i)
        if (!std::isfinite(a[i])) return false;
    return true;
}

// ------------------------------------------------------ pointer kinds ------
bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

DevBuf::~DevBuf() {
    if (owned && ptr) cudaFreeAsync(ptr, stream);
}

// Makes a device view of a caller buffer: device pointers are used in place;
// page-locked host memory is mapped into the device's address space, so the
// kernels read and write it in place (over NVLink-C2C on a Grace-Blackwell
// node: the data crosses once, while the kernel runs, with no staging copy);
// pageable host memory gets a stream-ordered device allocation (copied in
// if `in`, out by copy_out).
gac_status DevBuf::make(void *user, size_t nbytes, bool in, cudaStream_t s, const char *name, bool reread) {
    stream = s;
    bytes = nbytes;
    host = user;
    owned = false;
    if (!user || nbytes == 0) {
        ptr = nullptr;
        return GAC_OK;
    }
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, user) == cudaSuccess) {
        if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) {
            ptr = user;
            return GAC_OK;
        }
        if (a.type == cudaMemoryTypeHost && a.devicePointer && !reread) {
            ptr = a.devicePointer;
            return GAC_OK;
        }
    } else {
        cudaGetLastError();
    }
    cudaError_t e = cudaMallocAsync(&ptr, nbytes, s);
    if (e != cudaSuccess) {
        ptr = nullptr;
        return cuda_fail(e, name);
    }
    owned = true;
    if (in) {
        e = cudaMemcpyAsync(ptr, user, nbytes, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return cuda_fail(e, name);
    }
    return GAC_OK;
}

gac_status DevBuf::copy_out() {
    if (!owned || !ptr || !host) return GAC_OK;
    cudaError_t e = cudaMemcpyAsync(host, ptr, bytes, cudaMemcpyDeviceToHost, stream);
    return e == cudaSuccess ? GAC_OK : cuda_fail(e, "copy result to host");
}

int n_samples(int I, int B, int T) { return (T > 0 && I > B) ? (I - B) / T : 0; }

// Host buffers are staged through the device's default stream-ordered
// memory pool.  Let the pool keep what a call frees (instead of returning it
// to the driver at every synchronisation), so that repeated calls with host
// buffers do not map gigabytes of staging memory anew each time.  Done once
// per device; a caller that needs the memory back can call cudaMemPoolTrimTo
// on the device's default pool.
void keep_staging_pool() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (done[dev]) return;
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t keep = UINT64_MAX;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    cudaGetLastError();
    done[dev] = true;
}

// Lets a kernel be launched with `bytes` of dynamic shared memory.  The limit is
// the process's, not the call's: a call that set its own size would fail another
// thread's launch of the same kernel with a larger one.  So every call sets the
// same value, all that the device gives a block beside the kernel's static
// shared memory, whatever it needs itself.
cudaError_t allow_smem(const void *fn, size_t bytes) {
    cudaFuncAttributes a;
    int dev = 0, block_max = 0;
    cudaError_t e = cudaFuncGetAttributes(&a, fn);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&block_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const int most = block_max - static_cast<int>(a.sharedSizeBytes);
    if (most < 0 || bytes > static_cast<size_t>(most)) return cudaErrorInvalidValue;
    return a.maxDynamicSharedSizeBytes == most ? cudaSuccess
                                               : cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// ------------------------------------------------------ SMT g(x) table ----
// g(x) = int_0^1 exp(-x u^2) du by 40-point Gauss-Legendre quadrature: the
// integrand is entire in u, and for -13 <= x <= 17 the rule agrees with
// 40-digit adaptive quadrature to 2e-15 relative.
namespace {
struct GaussLegendre01 {
    static constexpr int n = 40;
    double node[n], weight[n];  // on [0, 1]
    GaussLegendre01() {
        for (int i = 0; i < n; ++i) {
            // Newton's method on the Legendre polynomial P_n from the
            // asymptotic estimate of its i-th root; P_n by the three-term
            // recurrence, P_n'(z) = n (z P_n - P_{n-1}) / (z^2 - 1)
            double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
            for (int it = 0; it < 100; ++it) {
                double pm = 1.0, p = z;
                for (int j = 2; j <= n; ++j) {
                    const double pn = ((2.0 * j - 1.0) * z * p - (j - 1.0) * pm) / j;
                    pm = p;
                    p = pn;
                }
                dp = n * (z * p - pm) / (z * z - 1.0);
                const double dz = p / dp;
                z -= dz;
                if (std::fabs(dz) < 1e-15) break;
            }
            node[i] = 0.5 * (1.0 + z);
            weight[i] = 1.0 / ((1.0 - z * z) * dp * dp);  // (2 / ((1 - z^2) P_n'^2)) / 2
        }
    }
    double g(double x) const {
        double s = 0.0;
        for (int i = 0; i < n; ++i) s += weight[i] * std::exp(-x * node[i] * node[i]);
        return s;
    }
};
}  // namespace

// Monomial coefficients af[0..K-1] (float) in d of the degree-(K-1)
// polynomial that interpolates f(d) at the K Chebyshev points of [-h, h], and
// the largest relative error of that float polynomial, evaluated in double,
// on 65 points of the interval.
template <int K, class F>
static double cheb_fit(F &&f, float af[K], double h) {
    double T[K][K] = {};  // T[n][m]: coefficient of s^m in the Chebyshev polynomial T_n(s)
    T[0][0] = 1.0;
    T[1][1] = 1.0;
    for (int n = 2; n < K; ++n)
        for (int m = 0; m < K; ++m) T[n][m] = (m > 0 ? 2.0 * T[n - 1][m - 1] : 0.0) - T[n - 2][m];
    double fv[K];
    for (int j = 0; j < K; ++j) fv[j] = f(h * std::cos(M_PI * (j + 0.5) / K));
    double a[K] = {};  // monomial coefficients in s = d / h
    for (int n = 0; n < K; ++n) {
        double b = 0.0;  // Chebyshev coefficient b_n
        for (int j = 0; j < K; ++j) b += fv[j] * std::cos(M_PI * n * (j + 0.5) / K);
        b *= (n == 0 ? 1.0 : 2.0) / K;
        for (int m = 0; m < K; ++m) a[m] += b * T[n][m];
    }
    for (int m = 0; m < K; ++m) af[m] = static_cast<float>(a[m] / std::pow(h, m));  // coefficient of d^m
    double worst = 0.0;
    for (int q = 0; q <= 64; ++q) {
        const double dd = -h + 2.0 * h * q / 64.0;
        double p = af[K - 1];
        for (int m = K - 2; m >= 0; --m) p = p * dd + af[m];
        const double ref = f(dd);
        const double rel = std::fabs(p - ref) / std::fabs(ref);
        worst = (rel > worst || rel != rel) ? rel : worst;
    }
    return worst;
}
template <class F>
static double cheb8_fit(F &&f, float af[8]) {
    return cheb_fit<8>(f, af, 0.5);
}

// Fills mc->gtab with, for each centre c = k/2, k = k_lo .. k_hi, the
// monomial coefficients in d of the degree-5 polynomial that interpolates
// g(c + d) at the six Chebyshev points of [-1/4, 1/4], and checks every
// interval on 65 points against the quadrature (relative error of the float
// coefficients evaluated in double at most 2e-7; the interpolation error
// itself is about 1e-8 on quarter-width half-intervals).  k_hi = the centre
// nearest xmax (the largest argument the model's bounds allow) when that fits
// in kGTabMax intervals: then the kernels need no asymptote.  Otherwise the
// table ends at a centre >= 16 and x >= c_hi + 1/4 takes sqrt(pi)/2 x^-1/2.
static gac_status build_g_table(double xmin, double xmax, ModelConst *mc) {
    static const GaussLegendre01 gl;
    const int k_lo = static_cast<int>(std::floor(2.0 * xmin - 0.5));
    if (k_lo < 2 * static_cast<int>(kSmtArgMin) - 2)
        return fail(GAC_ERR_INVALID_ARG, "SMT argument range starts at %g, below %d", xmin,
                    static_cast<int>(kSmtArgMin));
    const double k_need = std::max(std::ceil(2.0 * xmax - 0.5), 2.0 * kGTail);
    const int n_int = static_cast<int>(std::min<double>(kGTabMax, k_need - k_lo + 1));
    const int k_hi = k_lo + n_int - 1;
    if (k_hi < 2 * static_cast<int>(kGTail)) return fail(GAC_ERR_INVALID_ARG, "g(x) table too short");
    for (int i = 0; i < n_int; ++i) {
        const double c = 0.5 * (k_lo + i);
        float af[6];
        const double err = cheb_fit<6>([&](double d) { return gl.g(c + d); }, af, 0.25);
        for (int m = 0; m < 4; ++m) mc->gtab[i * 4 + m] = af[m];
        mc->gtab[(kGTabMax + i) * 4 + 0] = af[4];
        mc->gtab[(kGTabMax + i) * 4 + 1] = af[5];
        mc->gtab[(kGTabMax + i) * 4 + 2] = 0.0f;
        mc->gtab[(kGTabMax + i) * 4 + 3] = 0.0f;
        if (!(err <= 2e-7)) return fail(GAC_ERR_INVALID_ARG, "g(x) table check failed near x = %g", c);
    }
    const int c_lo = k_lo;
    const double c_hi = 0.5 * k_hi;
    mc->gtab_lo = c_lo;
    mc->gtab_n = n_int;
    mc->gtab_tail = c_hi + 0.25 >= xmax ? 0 : 1;
    mc->gtab_tail_x = static_cast<float>(c_hi + 0.25);
    return GAC_OK;
}

// ------------------------------------------------- AxCaliberSMT constants --
// m-th positive zero of J1' (m >= 1): Newton's method on J1'(x) = J0(x) -
// J1(x)/x, with J1''(x) = -J1'(x)/x - (1 - 1/x^2) J1(x) from Bessel's
// equation, from McMahon's estimate (m - 1/4) pi - 7 / (8 (m - 1/4) pi).
static double j1p_zero(int m) {
    const double beta = (m - 0.25) * M_PI;
    double x = beta - 7.0 / (8.0 * beta);
    for (int it = 0; it < 50; ++it) {
        const double j0 = std::cyl_bessel_j(0.0, x), j1 = std::cyl_bessel_j(1.0, x);
        const double d1 = j0 - j1 / x;
        const double d2 = -d1 / x - (1.0 - 1.0 / (x * x)) * j1;
        const double step = d1 / d2;
        x -= step;
        if (std::fabs(step) < 1e-15 * x) break;
    }
    return x;
}

// N_m of the cylinder series in double (see ax_n_series_f for the forms).
static double ax_n_host(double q, double dl, double DL) {
    const double a = q * dl;
    if (a < 1.0) return 2.0 * (std::expm1(-a) + a) - std::exp(-q * DL) * (std::expm1(a) + std::expm1(-a));
    return 2.0 * a - 2.0 + 2.0 * (std::exp(-a) + std::exp(-q * DL)) - std::exp(-q * (DL - dl)) - std::exp(-q * (DL + dl));
}

// Per-measurement constants, distinct timings, series coefficients and the
// number of terms: the FP32 evaluation keeps the terms whose tail stays below
// 2e-8 of the sum for every timing at 64 radii spanning the prior box; the
// FP64 evaluation keeps all kAxMaxTerms.
static gac_status build_axcal(const gac_model_desc *d, ModelConst *mc) {
    AxConst &ax = mc->ax;
    const int K = d->n_acq / 3;
    if (K > kAxMaxMeas) return fail(GAC_ERR_INVALID_ARG, "at most %d AxCaliberSMT measurements", kAxMaxMeas);
    ax.n_timing = 0;
    for (int k = 0; k < K; ++k) {
        const double b = d->acq[3 * k], Delta = d->acq[3 * k + 1], delta = d->acq[3 * k + 2];
        int t = 0;
        while (t < ax.n_timing && !(ax.Delta_d[t] == Delta && ax.delta_d[t] == delta)) ++t;
        if (t == ax.n_timing) {
            if (t == kAxMaxTiming) return fail(GAC_ERR_INVALID_ARG, "at most %d distinct (Delta, delta)", kAxMaxTiming);
            ax.Delta_d[t] = Delta;
            ax.delta_d[t] = delta;
            ax.Delta_f[t] = static_cast<float>(Delta);
            ax.delta_f[t] = static_cast<float>(delta);
            ++ax.n_timing;
        }
        ax.t[k] = t;
        const double g2 = b / (delta * delta * (Delta - delta / 3.0));
        ax.b_d[k] = b;
        ax.g2_d[k] = g2;
        ax.csf_d[k] = std::exp(-b * kAxDcsfD);
        ax.b_f[k] = static_cast<float>(b);
        ax.g2_f[k] = static_cast<float>(g2);
        ax.csf_f[k] = static_cast<float>(ax.csf_d[k]);
    }
    // the FP32 path's measurements in timing order (stable), with their constants
    constexpr double kLog2e = 1.44269504088896340736;
    int pos = 0;
    for (int t = 0; t < ax.n_timing; ++t) {
        ax.first[t] = pos;
        for (int k = 0; k < K; ++k) {
            if (ax.t[k] != t) continue;
            float *m = ax.meas + 8 * pos++;
            m[0] = static_cast<float>(ax.b_d[k] * kAxDaD);
            m[1] = static_cast<float>(ax.g2_d[k]);
            m[2] = static_cast<float>(ax.g2_d[k] * kLog2e);
            m[3] = static_cast<float>(ax.b_d[k] * kLog2e);
            m[4] = static_cast<float>(ax.b_d[k]);
            m[5] = ax.csf_f[k];
            std::memcpy(&m[6], &k, sizeof k);
            m[7] = 0.0f;
        }
    }
    for (int t = ax.n_timing; t <= kAxMaxTiming; ++t) ax.first[t] = pos;
    double x2d[kAxMaxTerms], c[kAxMaxTerms];
    for (int m = 0; m < kAxMaxTerms; ++m) {
        const double x = j1p_zero(m + 1), x2 = x * x;
        x2d[m] = x2 * kAxDaD;
        c[m] = 2.0 / (kAxDaD * kAxDaD * x2 * x2 * x2 * (x2 - 1.0));
        ax.x2d_d[m] = x2d[m];
        ax.c_d[m] = c[m];
        ax.x2d_f[m] = static_cast<float>(x2d[m]);
        ax.c_f[m] = static_cast<float>(c[m]);
    }
    ax.terms_d = kAxMaxTerms;
    const double r_lo = 0.5 * d->lb[0], r_hi = 0.5 * d->ub[0];
    int terms = 1;
    for (int t = 0; t < ax.n_timing; ++t)
        for (int i = 0; i < 64; ++i) {
            const double R = r_lo * std::pow(r_hi / r_lo, i / 63.0), r2 = R * R;
            double term[kAxMaxTerms], total = 0.0;
            for (int m = 0; m < kAxMaxTerms; ++m) total += term[m] = c[m] * ax_n_host(x2d[m] / r2, ax.delta_d[t], ax.Delta_d[t]);
            double tail = total;
            int need = 0;
            while (need < kAxMaxTerms && tail > 2e-8 * total) tail -= term[need++];
            terms = std::max(terms, need);
        }
    ax.terms_f = terms;
    double dmin = ax.delta_d[0];
    for (int t = 1; t < ax.n_timing; ++t) dmin = std::min(dmin, ax.delta_d[t]);
    ax.careful_f = 0;
    while (ax.careful_f < ax.terms_f && x2d[ax.careful_f] / (r_hi * r_hi) * dmin < 1.0) ++ax.careful_f;
    // the FP32 table of phi_j(R) = R^6 sum_m c_m N_m in u = log2 R: intervals
    // of width <= 1/2 over the prior box (at most kAxTabMax, widened if the
    // box is wider), each checked on 65 points; if any check exceeds 3e-7 the
    // kernels sum the series instead
    const double u_lo = std::log2(r_lo), u_hi = std::log2(r_hi);
    const int n_int = std::min(kAxTabMax, std::max(1, static_cast<int>(std::ceil((u_hi - u_lo) / 0.5))));
    const double w = std::max(u_hi - u_lo, 1e-3) / n_int;
    bool ok = true;
    for (int t = 0; t < ax.n_timing && ok; ++t)
        for (int i = 0; i < n_int && ok; ++i) {
            const double uc = u_lo + (i + 0.5) * w;
            auto phi = [&](double dd) {
                const double R = std::exp2(uc + dd * w), r2 = R * R;
                double sum = 0.0;
                for (int m = 0; m < kAxMaxTerms; ++m) sum += c[m] * ax_n_host(x2d[m] / r2, ax.delta_d[t], ax.Delta_d[t]);
                return r2 * r2 * r2 * sum;
            };
            float af[8];
            ok = cheb8_fit(phi, af) <= 3e-7;
            for (int m = 0; m < 8; ++m) ax.tab[((2 * t + (m < 4 ? 0 : 1)) * kAxTabMax + i) * 4 + (m & 3)] = af[m];
        }
    ax.tab_n = ok ? n_int : 0;
    ax.tab_inv_w = static_cast<float>(1.0 / w);
    ax.tab_off = static_cast<float>(-u_lo / w - 0.5);
    return GAC_OK;
}

// ----------------------------------------------------- launch sizing -------
static int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

int row_stride_for(int kind, int M) {
    // odd stride in the unit the kernel reads (float, or float2 for complex)
    // so that the voxels of a warp fall into distinct shared-memory banks
    if (model_complex(kind)) return 2 * ((M / 2) | 1);
    return M | 1;
}

static size_t smem_bytes_for(int kind, int prec, int C, int M, int moments_mode, int block) {
    const size_t w = (prec == GAC_PREC_FP32) ? sizeof(float) : sizeof(double);
    const bool blocked = prec == GAC_PREC_MIXED && moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    return tile_smem_bytes(model_n_par(kind), w, block / C, row_stride_for(kind, M), true, blocked, block);
}

static const void *mh_kernel_ptr(const ModelConst &mc, int prec, bool trace, int block) {
    switch (mc.kind) {
    case GAC_MODEL_MONOEXP: return mh_ptr_monoexp(prec, trace, block);
    case GAC_MODEL_MWI3: return mh_ptr_mwi3(prec, trace, block);
    case GAC_MODEL_SMT: return mh_ptr_smt(prec, trace, block, mc.n_acq < kAnchor);
    case GAC_MODEL_AXCAL_SMT: return mh_ptr_axcal(prec, trace, block);
    case GAC_MODEL_LINEAR_TEST: return mh_ptr_linear(prec, trace, block);
    default: return nullptr;
    }
}

// Resident blocks of `block` threads per SM of the one-launch kernel, with its
// attributes set.
static gac_status mh_resident(const ModelConst &mc, int prec, bool trace, int C, int moments_mode, int block,
                              LaunchCfg *cfg, int *per_sm) {
    cfg->fn = mh_kernel_ptr(mc, prec, trace, block);
    if (!cfg->fn) return fail(GAC_ERR_INVALID_ARG, "no kernel for kind %d precision %d", mc.kind, prec);
    cfg->block = block;
    cfg->smem = smem_bytes_for(mc.kind, prec, C, mc.n_meas, moments_mode, block);
    cudaError_t e = allow_smem(cfg->fn, cfg->smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    // prefer the largest shared-memory carveout: the tile and Welford
    // accumulators, not L1, decide how many blocks fit
    e = cudaFuncSetAttribute(cfg->fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(carveout)");
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, cfg->fn, block, cfg->smem);
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    if (*per_sm < 1) return fail(GAC_ERR_INVALID_ARG, "kernel does not fit on an SM (smem %zu)", cfg->smem);
    return GAC_OK;
}

// Time of a launch of `tiles` full blocks in units of a full wave: whole waves,
// and a last one in which the fullest SM holds r of its `per_sm` blocks.  An SM
// with few warps waits out their latency, so the last wave costs 1/4 + 3/4 r /
// per_sm of a full one (3-pool, blocks of 128: 0.42, 0.58, 0.80 and 1 measured
// for r = 1..4).
static double waves(int64_t tiles, int per_sm) {
    const int64_t slots = static_cast<int64_t>(per_sm) * sm_count();
    const int64_t rest = tiles % slots;
    if (rest == 0) return static_cast<double>(tiles / slots);
    const int64_t r = (rest + sm_count() - 1) / sm_count();
    return static_cast<double>(tiles / slots) + 0.25 + 0.75 * static_cast<double>(r) / per_sm;
}

// Grid: one block per tile of voxels, capped at the number of blocks that
// are resident at once (the kernel strides over the remaining tiles).  The
// random numbers are keyed by voxel, chain and iteration, so results do not
// depend on the tiling.
static gac_status plan_launch(const ModelConst &mc, int prec, bool trace, int C, int64_t n_vox, int moments_mode,
                              LaunchCfg *cfg, int64_t *n_tiles, int *vb) {
    const int64_t chains = n_vox * C;
    int per_sm = 0;
    gac_status st = mh_resident(mc, prec, trace, C, moments_mode, kBlock, cfg, &per_sm);
    if (st != GAC_OK) return st;
    int threads = kBlock;
    const int64_t resident = static_cast<int64_t>(per_sm) * sm_count();
    if (!trace && prec != GAC_PREC_FP64) {
        // Blocks of kHalfBlock where they spread the chains more evenly: a
        // block's warps go to the SM's four schedulers in turn, so full blocks
        // of four warps load them evenly, while two blocks of eight with
        // some idle warps, or a last wave of few large blocks, leave
        // schedulers with twice the warps of others.  Full waves of half
        // blocks measured up to 3% slower (1.03); the mono-exponential ones have
        // to promise 5.5% (kBlock -> kHalfBlock, us per iteration: 240,000
        // chains, where they promise 2.2%, 2.39 -> 2.46; 200,000, 5.8%, 2.14 ->
        // 2.02; SMT, 393,216 chains, 0.4%: 6.44 -> 6.14).  3-pool, us per iteration,
        // kBlock -> kHalfBlock: 14,400 chains 1.79 -> 1.31, 49,380 3.12 ->
        // 2.51, 120,000 6.09 -> 5.24, 200,000 9.01 -> 8.05.  Below one block
        // an SM, tiles shrink in whole warps of chains: each scheduler gets at
        // most one warp.
        LaunchCfg half;
        int half_per_sm = 0;
        if ((st = mh_resident(mc, prec, trace, C, moments_mode, kHalfBlock, &half, &half_per_sm)) != GAC_OK) return st;
        half_per_sm = std::min(half_per_sm, 2 * per_sm);  // as many warps: 20 instead of 16 ran 2% slower (3-pool)
        const int vb1 = std::max(1, kBlock / C), vb2 = std::max(1, kHalfBlock / C);
        const double t1 = waves((n_vox + vb1 - 1) / vb1, per_sm);
        const double t2 = (mc.kind == GAC_MODEL_MONOEXP ? 1.055 : 1.03) * waves((n_vox + vb2 - 1) / vb2, half_per_sm);
        const int64_t want = (chains + sm_count() - 1) / sm_count();  // chains an SM
        if (t2 < t1 || want <= kHalfBlock) {
            *cfg = half;
            per_sm = half_per_sm;
            threads = static_cast<int>(std::min<int64_t>(kHalfBlock, (want + 31) / 32 * 32));
        }
    }
    // Too few chains for a full tile per resident block: tiles shrink in whole
    // warps of chains, so that the chains spread over all SMs.  Not where they lost
    // to full tiles on fewer SMs, MIXED and FP32 without a trace: SMT (58,400 chains,
    // 1.31 -> 1.35 us an iteration), the 3-pool model and AxCaliberSMT with thinned
    // moments (3-pool, 20,000: 1.58 -> 1.63; over every state, 1.75 -> 1.65, and FP32,
    // 1.66 -> 1.58, they gain) and the mono-exponential model once every SM has a tile
    // (100,000: 1.13 -> 1.18; 20,000: 0.54 -> 0.53).
    const bool two_blocks = mc.kind == GAC_MODEL_MWI3 || mc.kind == GAC_MODEL_AXCAL_SMT;
    const bool spread = trace || prec == GAC_PREC_FP64 ||
                        (two_blocks && (prec == GAC_PREC_FP32 || moments_mode == GAC_MOMENTS_ALL_POSTBURNIN)) ||
                        (mc.kind == GAC_MODEL_MONOEXP && chains < static_cast<int64_t>(sm_count()) * kBlock);
    if (spread && cfg->block == kBlock && chains < resident * kBlock) {
        const int64_t want = (chains + resident - 1) / resident;  // chains per block
        threads = static_cast<int>(std::min<int64_t>(kBlock, std::max<int64_t>(32, (want + 31) / 32 * 32)));
    }
    *vb = std::max(1, threads / C);
    *n_tiles = (n_vox + *vb - 1) / *vb;
    cfg->grid = static_cast<int>(std::min<int64_t>(*n_tiles, static_cast<int64_t>(per_sm) * sm_count()));
    return GAC_OK;
}

// A run in slices (mh_slice_kernel).
struct SlicePlan {
    const void *fn = nullptr;  // nullptr: one launch
    size_t smem = 0;
    int slots = 0;  // resident blocks
    int q = 0;      // iterations of a slice
    int count = 0;  // slices of a tile
    int vb = 0;
    int64_t n_tiles = 0;
};

// Slices for a problem whose last wave of tiles would leave the GPU partly idle:
// the tiles take turns, so that all launches but the last are full.  n_tiles
// tiles in `count` slices take ceil(count n_tiles / slots) launches.  Chosen where
// that is estimated 3% shorter than one launch: whole waves and, for a last one
// that fills the fullest SM to a share f, 0.2 + f / 2 (an AxCaliberSMT wave and
// 0.29 measured 1.45 waves), with 2% for the launches' ends.  Only for the two
// models whose kernels hold 2 blocks an SM, where a wave is longest; thinning of
// at least 16, as the moments live in HBM between slices, and for the 3-pool
// model not over every state (its partial sums cost more to keep than the last
// wave).  us per iteration, one launch -> slices: AxCaliberSMT, 80,000 chains
// 4.21 -> 3.40, 100,004 4.73 -> 4.16, 140,000 6.19 -> 5.66; 3-pool, 80,000 3.56 ->
// 3.21, 93,000 4.18 -> 3.58, 140,000 5.65 -> 5.34; past three waves nothing.
static gac_status plan_slices(const ModelConst &mc, const gac_mcmc_opts *o, int64_t n_vox, const LaunchCfg &one,
                              int64_t one_tiles, SlicePlan *sp) {
    const int C = o->n_chains;
    const bool all = o->moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    const void *fn = mc.kind == GAC_MODEL_AXCAL_SMT     ? mh_slice_ptr_axcal()
                     : mc.kind == GAC_MODEL_MWI3 && !all ? mh_slice_ptr_mwi3()
                                                         : nullptr;
    if (!fn || o->precision != GAC_PREC_MIXED || o->trace_n_vox != 0 || o->lanes_per_chain != 0 || o->iterations < 256 ||
        (!all && o->thin < 16))
        return GAC_OK;
    SlicePlan p;
    p.vb = std::max(1, kBlock / C);
    p.n_tiles = (n_vox + p.vb - 1) / p.vb;
    if (one_tiles <= one.grid) return GAC_OK;  // a single wave
    p.smem = tile_smem_bytes(mc.n_par, sizeof(double), p.vb, row_stride_for(mc.kind, mc.n_meas), false, all);
    cudaError_t e = allow_smem(fn, p.smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBlock, p.smem);
    if (e != cudaSuccess) return cuda_fail(e, "slice kernel occupancy");
    p.slots = per_sm * sm_count();
    if (p.slots < 1 || p.n_tiles <= p.slots) return GAC_OK;
    const int64_t rest = one_tiles % one.grid;
    const double f = static_cast<double>((rest + sm_count() - 1) / sm_count() * sm_count()) / one.grid;
    // in waves of `slots` full blocks
    const double plain = (static_cast<double>(one_tiles / one.grid) + (rest == 0 ? 0.0 : f >= 1.0 ? 1.0 : 0.2 + 0.5 * f)) *
                         one.grid * one.block / (static_cast<double>(p.slots) * kBlock);
    double best = 0.97 * plain;
    for (int m = 2; m <= 24 && o->iterations / m >= 64; ++m) {
        const double t = 1.02 * static_cast<double>((m * p.n_tiles + p.slots - 1) / p.slots) / m;
        if (t < best) {
            best = t;
            p.q = static_cast<int>((static_cast<int64_t>(o->iterations) + m - 1) / m);
        }
    }
    if (p.q == 0) return GAC_OK;
    p.count = static_cast<int>((static_cast<int64_t>(o->iterations) + p.q - 1) / p.q);  // I + q passes 2^31
    p.fn = fn;
    *sp = p;
    return GAC_OK;
}

// Device memory of the chains' state between slices (struct SliceState), carved
// from one allocation: its bytes, and the pointers when `base` is given.
static size_t slice_state(const ModelConst &mc, int64_t chains, bool all, char *base, SliceState *ss) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) & ~static_cast<size_t>(255);
        return base ? base + at : nullptr;
    };
    const size_t P = mc.n_par, n = static_cast<size_t>(chains);
    SliceState s{};
    s.theta = take(P * n * 4);
    s.L = take(n * 4);
    s.n_acc = reinterpret_cast<int32_t *>(take(n * 4));
    s.n_bad = reinterpret_cast<int32_t *>(take(n * 4));
    s.wf_mean = take(P * n * 8);
    s.wf_m2 = take(P * n * 8);
    s.adapt = reinterpret_cast<int32_t *>(take(2 * n * 4));
    s.blk = all ? reinterpret_cast<float *>(take(3 * P * n * 4)) : nullptr;
    if (ss) *ss = s;
    return off;
}

gac_status validate_opts(const gac_mcmc_opts *o, int64_t n_vox) {
    if (!o) return fail(GAC_ERR_INVALID_ARG, "opts is NULL");
    if (o->iterations < 0 || o->iterations == INT32_MAX)
        return fail(GAC_ERR_INVALID_ARG, "iterations must be in [0, 2^31-2]");
    if (o->burnin < 0) return fail(GAC_ERR_INVALID_ARG, "burnin must be >= 0");
    if (o->thin < 1) return fail(GAC_ERR_INVALID_ARG, "thin must be >= 1");
    if (o->n_chains < 1 || o->n_chains > 64) return fail(GAC_ERR_INVALID_ARG, "n_chains must be in [1, 64]");
    if (o->precision < GAC_PREC_MIXED || o->precision > GAC_PREC_FP64)
        return fail(GAC_ERR_INVALID_ARG, "unknown precision %d", o->precision);
    if (o->moments_mode != GAC_MOMENTS_THINNED && o->moments_mode != GAC_MOMENTS_ALL_POSTBURNIN)
        return fail(GAC_ERR_INVALID_ARG, "unknown moments_mode %d", o->moments_mode);
    if (o->trace_n_vox < 0 || o->trace_n_vox > n_vox)
        return fail(GAC_ERR_INVALID_ARG, "trace_n_vox must be in [0, n_vox]");
    if (o->adapt_window < 0) return fail(GAC_ERR_INVALID_ARG, "adapt_window must be >= 0");
    if (o->adapt_window > 0 && !(o->adapt_target > 0.0 && o->adapt_target < 1.0))
        return fail(GAC_ERR_INVALID_ARG, "adapt_target must be in (0, 1)");
    if (o->voxel_base > (1ull << 32) || static_cast<uint64_t>(n_vox) > (1ull << 32) - o->voxel_base)
        return fail(GAC_ERR_INVALID_ARG, "voxel_base + n_vox must be <= 2^32 (32-bit counter word)");
    if (o->lanes_per_chain != 0 && o->lanes_per_chain != 1 && o->lanes_per_chain != 2 && o->lanes_per_chain != 4)
        return fail(GAC_ERR_INVALID_ARG, "lanes_per_chain must be 0, 1, 2 or 4");
    return GAC_OK;
}

// Lanes per chain of a gac_mcmc_run (1: the one-thread kernel).  The
// lane-split kernel handles MIXED runs without trace of the mono-exponential
// and 3-pool models with evenly spaced echoes in 2..4 blocks of kAnchor.  The
// library uses it for the mono-exponential model when the chains would give
// fewer than one warp per SM sub-partition (there it shortens the latency of an
// iteration; on larger problems one thread per chain keeps more chains in
// flight).  The 3-pool model takes it with 7 to 12 echoes, two lanes a chain, where
// trees of depth 2 would put a second warp on a scheduler and thinning is so far
// apart that the lanes' own FP64 moment updates weigh little (12 echoes, us an iteration, split against depth 2 at
// 9,600 chains and against one thread at 14,400: thinning 100 0.68 and 0.77, 0.96
// and 1.02; thinning 5 1.06 and 0.91, 1.36 and 1.37; moments over every state 1.42
// and 1.08, 1.50 and 1.20); with more echoes, four lanes a chain, it lost to both
// (24 echoes, 14,400 chains: 2.35 against 1.30 one thread per chain).
static gac_status choose_lanes(const ModelConst &mc, const gac_mcmc_opts *o, int64_t n_vox, int *lanes) {
    const int nb = (mc.n_acq + kAnchor - 1) / kAnchor;
    const bool eligible = o->precision == GAC_PREC_MIXED && o->trace_n_vox == 0 && mc.even &&
                          (mc.kind == GAC_MODEL_MONOEXP || mc.kind == GAC_MODEL_MWI3) && nb >= 2 && nb <= 4;
    *lanes = 1;
    if (o->lanes_per_chain == 1) return GAC_OK;
    if (o->lanes_per_chain > 1) {
        if (!eligible || nb > o->lanes_per_chain)
            return fail(GAC_ERR_INVALID_ARG,
                        "lanes_per_chain %d needs MIXED precision, no trace and a mono-exponential or 3-pool "
                        "model with evenly spaced echoes in at most %d blocks of %d",
                        o->lanes_per_chain, o->lanes_per_chain, kAnchor);
        *lanes = o->lanes_per_chain;
        return GAC_OK;
    }
    const int64_t one_warp_each = static_cast<int64_t>(sm_count()) * 4 * 32, chains = n_vox * o->n_chains;
    if (!eligible || chains >= one_warp_each) return GAC_OK;
    if (mc.kind == GAC_MODEL_MONOEXP) {
        *lanes = nb <= 2 ? 2 : 4;
    } else if (nb == 2 && 4 * chains > one_warp_each && o->moments_mode == GAC_MOMENTS_THINNED) {
        // the thinning from which it wins, by the kernel it replaces: depth 2; one
        // thread, with at most one and a half split warps a scheduler; with two
        const int least = 2 * chains <= one_warp_each ? 12 : 4 * chains <= 3 * one_warp_each ? 3 : 8;
        if (o->thin >= least) *lanes = 2;
    }
    return GAC_OK;
}

// Lane-split launch: blocks just large enough to give every SM the same
// number of warps (whole voxels per block), as many as fit at once.
static gac_status plan_split(const ModelConst &mc, int G, int C, int64_t n_vox, int moments_mode, LaunchCfg *cfg,
                             int64_t *n_tiles, int *vb) {
    const bool all = moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    const void *fn = mc.kind == GAC_MODEL_MONOEXP ? mh_split_ptr_monoexp(G, all) : mh_split_ptr_mwi3(G, all);
    if (!fn) return fail(GAC_ERR_INVALID_ARG, "no lane-split kernel for kind %d with %d lanes", mc.kind, G);
    const int sms = sm_count();
    const int64_t warps = (n_vox * C * G + 31) / 32;
    int threads = static_cast<int>(std::min<int64_t>(kBlock, 32 * ((warps + sms - 1) / sms)));
    threads = std::max(threads, 32 * ((C * G + 31) / 32));  // at least one voxel
    *vb = std::max(1, threads / (C * G));
    const size_t smem = split_smem_bytes(mc.n_par, G, threads, *vb, row_stride_for(mc.kind, mc.n_meas), all);
    cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem)) != cudaSuccess)
        return cuda_fail(e, "occupancy query");
    if (per_sm < 1) return fail(GAC_ERR_INVALID_ARG, "lane-split kernel does not fit on an SM (smem %zu)", smem);
    *n_tiles = (n_vox + *vb - 1) / *vb;
    cfg->grid = static_cast<int>(std::min<int64_t>(*n_tiles, static_cast<int64_t>(per_sm) * sms));
    cfg->fn = fn;
    cfg->smem = smem;
    cfg->block = threads;
    return GAC_OK;
}

static const void *mh_spec_ptr(int kind, int depth, bool all) {
    switch (kind) {
    case GAC_MODEL_MONOEXP: return mh_spec_ptr_monoexp(depth, all);
    case GAC_MODEL_MWI3: return mh_spec_ptr_mwi3(depth, all);
    case GAC_MODEL_SMT: return mh_spec_ptr_smt(depth, all);
    case GAC_MODEL_AXCAL_SMT: return mh_spec_ptr_axcal(depth, all);
    default: return nullptr;
    }
}

// Blocks of a speculative launch: the warps spread evenly over the SMs in
// blocks of whole voxels.
struct SpecShape {
    int threads, vb;
    int64_t n_tiles;
    int64_t warps() const { return n_tiles * (threads / 32); }
};
static SpecShape spec_shape(int depth, int C, int64_t n_vox) {
    const int G = 1 << depth, sms = sm_count();
    const int64_t warps_per_sm = ((n_vox * C * G + 31) / 32 + sms - 1) / sms;
    const int64_t blocks_per_sm = (warps_per_sm * 32 + kSpecBlock - 1) / kSpecBlock;
    SpecShape sh;
    sh.threads = static_cast<int>(32 * ((warps_per_sm + blocks_per_sm - 1) / blocks_per_sm));
    sh.threads = std::max(sh.threads, 32 * ((C * G + 31) / 32));  // at least one voxel
    sh.vb = std::max(1, sh.threads / (C * G));
    sh.n_tiles = (n_vox + sh.vb - 1) / sh.vb;
    return sh;
}

// Depth of the speculation tree (mh_spec.cuh) for a gac_mcmc_run, 0 for none:
// the deepest tree whose warps find idle schedulers.  Measured on GB300 (ms
// per 1,000 iterations, 1 chain a voxel):
//   chains           200    1,200  2,400  4,800  9,600  14,400  19,200
//   3-pool    one    1.14   1.21   1.21   1.22   1.22   1.30    1.30
//             spec   0.31   0.37   0.47   0.67   0.96   1.31    1.61
//             depth  5      4      3      2      2      -       -
//   SMT       one    0.58   0.59   0.59   0.60   0.60   0.60    0.61
//             spec   0.15   0.18   0.22   0.28   0.41   0.52    0.63
//             depth  5      4      3      3      2      2       -
//   AxCaliber one    1.58   1.60   1.60   1.61   1.61   1.72    1.77
//             spec   0.40   0.49   0.62   0.77   1.10   1.41    1.68
//             depth  5      4      3      3      2      2       2
//   mono-exp  split  0.19   0.20   0.20   0.20   0.19   0.26    0.26
//             spec   0.14   0.17   0.19   -      -      -       -
//             depth  5      4      4
// A round of the trees of depth 3 and more takes as long with a second warp on
// its scheduler only where it waits on table lookups (SMT, AxCaliberSMT); the
// 3-pool round issues paired multiply-adds for most of its cycles.  Depth 2
// doubles the work per iteration and halves the serial path: it pays up to
// four warps a scheduler for AxCaliberSMT, three for SMT and two for the 3-pool
// model, the least latency-bound of the three.  The mono-exponential round is
// short enough that the lane-split kernel's shorter path wins where it applies
// (`split`) past two warps a scheduler at depth 4; with thinning of 4 or less,
// where that kernel's own moment updates weigh, past two at depth 3 (2,000
// iterations of 4,096 chains, thinning 2: 0.76 ms split, 0.62; thinning 5: 0.51
// both).  Where it does not apply (one block of echoes, uneven echoes, more than
// four blocks), depth 2 pays up to three warps a scheduler, and up to four where one
// thread's likelihood takes long for its echoes (us an iteration, one thread ->
// depth 2, at 19,000 chains: 2 echoes 0.37 -> 0.40, 6 echoes 0.46 -> 0.42, 12 uneven
// ones 0.72 -> 0.64, 26 echoes 0.53 -> 0.55, 32 0.59 -> 0.59, 64 0.85 -> 0.76) or
// moments are taken often (thinning 1, 2 echoes: 1.04 -> 0.85).
static int choose_depth(const ModelConst &mc, const gac_mcmc_opts *o, int64_t n_vox, bool split) {
    if (o->precision != GAC_PREC_MIXED || o->trace_n_vox != 0 || o->lanes_per_chain != 0 ||
        !mh_spec_ptr(mc.kind, 2, false))
        return 0;
    const int C = o->n_chains;
    const int64_t schedulers = static_cast<int64_t>(sm_count()) * 4;
    const bool mwi3 = mc.kind == GAC_MODEL_MWI3, mono = mc.kind == GAC_MODEL_MONOEXP;
    const bool all = o->moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    const bool mono4 = !mc.even || mc.n_acq == kAnchor || mc.n_acq >= 48 || (!all && o->thin <= 7);
    for (int depth = 5; depth >= 2; --depth) {
        if (C << depth > kSpecBlock || n_vox * C > (schedulers * 32 * 4 >> depth)) continue;
        // warps a scheduler
        const int per = depth == 5   ? 1
                        : depth == 4 ? (mono && !all ? 2 : 1)
                        : depth == 3 ? (mwi3 ? 1 : 2)
                        : mwi3       ? 2
                        : mc.kind == GAC_MODEL_SMT || (mono && !mono4) ? 3 : 4;
        if (split && (depth == 2 || (mono && depth == 3 && (all || o->thin > 4)))) return 0;
        if (spec_shape(depth, C, n_vox).warps() <= per * schedulers) return depth;
    }
    return 0;
}

static gac_status plan_spec(const ModelConst &mc, int depth, int C, int64_t n_vox, int moments_mode, LaunchCfg *cfg,
                            int64_t *n_tiles, int *vb) {
    const bool all = moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    const void *fn = mh_spec_ptr(mc.kind, depth, all);
    if (!fn) return fail(GAC_ERR_INVALID_ARG, "no speculative kernel for kind %d of depth %d", mc.kind, depth);
    const SpecShape sh = spec_shape(depth, C, n_vox);
    const bool help = spec_moment_warps(depth, all);
    const size_t smem = spec_smem_bytes(mc.n_par, 1 << depth, sh.threads, sh.vb, row_stride_for(mc.kind, mc.n_meas), all, help);
    const int block = sh.threads + (help ? 32 * moment_warps(mc.n_par * (sh.threads >> depth), kMomMaxWarps) : 0);
    cudaError_t e = allow_smem(fn, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem);
    if (e != cudaSuccess) return cuda_fail(e, "speculative kernel occupancy");
    if (per_sm < 1) return fail(GAC_ERR_INVALID_ARG, "speculative kernel does not fit on an SM (smem %zu)", smem);
    *vb = sh.vb;
    *n_tiles = sh.n_tiles;
    cfg->grid = static_cast<int>(std::min<int64_t>(sh.n_tiles, static_cast<int64_t>(per_sm) * sm_count()));
    cfg->fn = fn;
    cfg->smem = smem;
    cfg->block = block;
    cfg->sampling = sh.threads;
    return GAC_OK;
}

}  // namespace gac

using namespace gac;

// ===================================================================== ABI ==
extern "C" {

const char *gac_last_error(void) { return g_last_error.c_str(); }

const char *gac_version(void) { return "gac 0.1 (sm_103a)"; }

gac_status gac_model_register(const gac_model_desc *d, int *model_id) {
    clear_error();
    if (!d || !model_id) return fail(GAC_ERR_INVALID_ARG, "desc and model_id must not be NULL");
    const int P = model_n_par(d->kind);
    if (P < 0) return fail(GAC_ERR_UNKNOWN_MODEL, "unknown model kind %d", d->kind);
    if (d->n_par != P) return fail(GAC_ERR_INVALID_ARG, "kind %d has %d parameters, n_par = %d", d->kind, P, d->n_par);
    if (d->n_acq < 1 || d->n_acq > GAC_MAX_ACQ)
        return fail(GAC_ERR_INVALID_ARG, "n_acq must be in [1, %d]", GAC_MAX_ACQ);
    if (!d->acq || !d->lb || !d->ub || !d->step)
        return fail(GAC_ERR_INVALID_ARG, "acq, lb, ub and step must not be NULL");
    if (!all_finite(d->acq, d->n_acq) || !all_finite(d->lb, P) || !all_finite(d->ub, P) ||
        !all_finite(d->step, P))
        return fail(GAC_ERR_INVALID_ARG, "non-finite acquisition, bound or step");
    for (int p = 0; p < P; ++p) {
        if (d->lb[p] > d->ub[p]) return fail(GAC_ERR_INVALID_ARG, "lb[%d] > ub[%d]", p, p);
        if (d->step[p] < 0) return fail(GAC_ERR_INVALID_ARG, "step[%d] < 0", p);
    }
    if (d->kind == GAC_MODEL_MWI3) {
        for (int j = 3; j < 6; ++j)
            if (d->lb[j] <= 0) return fail(GAC_ERR_INVALID_ARG, "T2* lower bounds must be > 0");
        // phase arguments phi0 - 2 pi df t must stay in the range of sincos_cw
        double tmax = 0, dfmax = 0;
        for (int k = 0; k < d->n_acq; ++k) tmax = std::max(tmax, std::fabs(d->acq[k]));
        for (int j = 6; j < 8; ++j) dfmax = std::max({dfmax, std::fabs(d->lb[j]), std::fabs(d->ub[j])});
        const double amax = std::max(std::fabs(d->lb[8]), std::fabs(d->ub[8])) + kTwoPiMilliD * dfmax * tmax * (kAnchor + 1);
        if (amax > kSinCosMaxArg)
            return fail(GAC_ERR_INVALID_ARG, "phase range %.0f rad exceeds %.0f", amax, static_cast<double>(kSinCosMaxArg));
    }
    if (d->kind == GAC_MODEL_SMT) {
        for (int k = 0; k < d->n_acq; ++k) {
            const double b = d->acq[k];
            if (b < 0) return fail(GAC_ERR_INVALID_ARG, "b-values must be >= 0");
            if (b * (d->lb[2] - d->ub[3]) < kSmtArgMin || b * d->lb[1] < kSmtArgMin)
                return fail(GAC_ERR_INVALID_ARG,
                            "SMT bounds outside the validated range: need b*(ub[De_perp]-lb[De_par]) <= 12");
        }
    }

    if (d->kind == GAC_MODEL_AXCAL_SMT) {
        if (d->n_acq % 3 != 0) return fail(GAC_ERR_INVALID_ARG, "AxCaliberSMT takes (b, Delta, delta) triplets");
        for (int k = 0; k < d->n_acq / 3; ++k) {
            const double b = d->acq[3 * k], Delta = d->acq[3 * k + 1], delta = d->acq[3 * k + 2];
            if (b < 0 || !(delta > 0) || !(Delta >= delta))
                return fail(GAC_ERR_INVALID_ARG, "measurement %d: need b >= 0, delta > 0, Delta >= delta", k);
            if (b * (d->ub[3] - kAxDeParD) > -kSmtArgMin)
                return fail(GAC_ERR_INVALID_ARG, "AxCaliberSMT bounds outside the validated range: b*(ub[De_R]-1.7) <= 12");
        }
        if (!(d->lb[0] > 0)) return fail(GAC_ERR_INVALID_ARG, "the axon diameter's lower bound must be > 0");
    }

    ModelConst mc;
    std::memset(&mc, 0, sizeof mc);
    mc.kind = d->kind;
    mc.n_par = P;
    mc.n_acq = d->n_acq;
    mc.n_meas = model_complex(d->kind) ? 2 * d->n_acq : (d->kind == GAC_MODEL_AXCAL_SMT ? d->n_acq / 3 : d->n_acq);
    for (int k = 0; k < d->n_acq; ++k) {
        mc.acq_d[k] = d->acq[k];
        mc.acq_f[k] = static_cast<float>(d->acq[k]);
        mc.acq_l2e_f[k] = static_cast<float>(d->acq[k] * 1.44269504088896340736);
    }
    for (int p = 0; p < P; ++p) {
        mc.lb_d[p] = d->lb[p];
        mc.ub_d[p] = d->ub[p];
        mc.step_d[p] = d->step[p];
        mc.lb_f[p] = static_cast<float>(d->lb[p]);
        mc.ub_f[p] = static_cast<float>(d->ub[p]);
        mc.step_f[p] = static_cast<float>(d->step[p]);
    }
    // evenly spaced acquisitions (to 1e-9 relative) allow the recurrence
    mc.even = 0;
    if (d->n_acq >= 2) {
        const double t0 = d->acq[0];
        const double dt = (d->acq[d->n_acq - 1] - t0) / (d->n_acq - 1);
        bool even = dt > 0;
        for (int k = 0; k < d->n_acq && even; ++k) {
            const double want = t0 + k * dt;
            if (std::fabs(d->acq[k] - want) > 1e-9 * std::max(1.0, std::fabs(want))) even = false;
        }
        if (even) {
            mc.even = 1;
            mc.t0_f = static_cast<float>(t0);
            mc.dt_f = static_cast<float>(dt);
            mc.dtk_f = static_cast<float>(kAnchor * dt);
            auto dd = [](double x) {
                const float hi = static_cast<float>(x);
                return make_float2(hi, static_cast<float>(x - static_cast<double>(hi)));
            };
            mc.dd_t0 = dd(t0);
            mc.dd_dt = dd(dt);
            mc.dd_w0 = dd(kTwoPiMilliD * t0);
            mc.dd_w1 = dd(kTwoPiMilliD * dt);
            mc.dd_wk = dd(kTwoPiMilliD * kAnchor * dt);
            if (d->kind == GAC_MODEL_MWI3) {
                // the 3-pool set-up evaluates e^{-t/T2*} - 1 for t = t0, dt >= 0 only
                if (t0 < 0) mc.even = 0;
                double dfmax = 0;
                for (int j = 6; j < 8; ++j) dfmax = std::max({dfmax, std::fabs(d->lb[j]), std::fabs(d->ub[j])});
                const double bmax = kTwoPiMilliD * dfmax * std::max(std::fabs(t0), dt);
                const double bkh = kTwoPiMilliD * dfmax * 0.5 * kAnchor * dt;
                mc.dd_wkh = dd(kTwoPiMilliD * 0.5 * kAnchor * dt);
                mc.mwi3_flags = (bmax <= 0.78 ? kMwi3SmallB : 0) | (bkh <= 0.78 ? kMwi3SmallBK : 0) |
                                (std::max(t0, dt) / d->lb[5] <= 0.34 ? kMwi3SmallEW : 0);  // pi/4, ln2/2
            }
        }
    }
    if (d->kind == GAC_MODEL_SMT) {
        // the smallest and largest arguments b Da, b (De_par - De_perp) the bounds allow
        double xmin = 0.0, xmax = 0.0;
        for (int k = 0; k < d->n_acq; ++k) {
            xmin = std::min({xmin, d->acq[k] * d->lb[1], d->acq[k] * (d->lb[2] - d->ub[3])});
            xmax = std::max({xmax, d->acq[k] * d->ub[1], d->acq[k] * (d->ub[2] - d->lb[3])});
        }
        const gac_status st = build_g_table(xmin, xmax, &mc);
        if (st != GAC_OK) return st;
        mc.smt_b0 = mc.acq_f[0] == 0.0f;
        for (int k = 1; k < mc.n_acq; ++k)
            if (mc.acq_f[k] == 0.0f) mc.smt_b0 = 0;
    }
    if (d->kind == GAC_MODEL_AXCAL_SMT) {
        gac_status st = build_axcal(d, &mc);
        if (st != GAC_OK) return st;
        // g arguments: 0 <= b Da - kappa <= b Da (up to rounding) and b (1.7 - De_R)
        double xmin = -1.0, xmax = 0.0;
        for (int k = 0; k < mc.n_meas; ++k) {
            const double b = d->acq[3 * k];
            xmin = std::min(xmin, b * (kAxDeParD - d->ub[3]));
            xmax = std::max({xmax, b * kAxDaD, b * (kAxDeParD - d->lb[3])});
        }
        if ((st = build_g_table(xmin, xmax, &mc)) != GAC_OK) return st;
    }
    std::lock_guard<std::mutex> lk(g_reg_mu);
    for (size_t i = 0; i < g_models.size(); ++i)  // ModelConst is zero-filled before it is set
        if (std::memcmp(&g_models[i], &mc, sizeof mc) == 0) {
            *model_id = static_cast<int>(i + 1);
            return GAC_OK;
        }
    if (g_models.size() >= GAC_MAX_MODELS)
        return fail(GAC_ERR_INVALID_ARG, "at most %d models can be registered", GAC_MAX_MODELS);
    g_models.push_back(mc);
    *model_id = static_cast<int>(g_models.size());
    return GAC_OK;
}

gac_status gac_model_info(int model_id, int *n_par, int *n_meas) {
    clear_error();
    ModelConst mc;
    gac_status st = model_get(model_id, &mc);
    if (st != GAC_OK) return st;
    if (n_par) *n_par = mc.n_par;
    if (n_meas) *n_meas = mc.n_meas;
    return GAC_OK;
}

gac_status gac_result_sizes(int model_id, int64_t n_vox, const gac_mcmc_opts *o, size_t bytes[8]) {
    clear_error();
    ModelConst mc;
    gac_status st = model_get(model_id, &mc);
    if (st != GAC_OK) return st;
    if (!bytes) return fail(GAC_ERR_INVALID_ARG, "bytes must not be NULL");
    if (n_vox < 0) return fail(GAC_ERR_INVALID_ARG, "n_vox must be >= 0");
    if ((st = validate_opts(o, n_vox)) != GAC_OK) return st;
    const size_t N = static_cast<size_t>(n_vox), P = mc.n_par, C = o->n_chains;
    const size_t S = n_samples(o->iterations, o->burnin, o->thin);
    bytes[0] = P * N * sizeof(double);
    bytes[1] = P * N * sizeof(double);
    bytes[2] = S * C * P * N * sizeof(float);
    bytes[3] = C * N * sizeof(float);
    bytes[4] = C * N * sizeof(int32_t);
    bytes[5] = static_cast<size_t>(o->trace_n_vox) * C * o->iterations * sizeof(gac_trace_rec);
    bytes[6] = P * N * sizeof(double);
    bytes[7] = C * N * sizeof(float);
    return GAC_OK;
}

gac_status gac_mcmc_run(int model_id, const void *data, int64_t n_vox, const float *sigma,
                        float sigma_scalar, const float *x0, const gac_mcmc_opts *o,
                        gac_result *out, void *stream) {
    clear_error();
    ModelConst mc;
    gac_status st = model_get(model_id, &mc);
    if (st != GAC_OK) return st;
    if (n_vox < 0) return fail(GAC_ERR_INVALID_ARG, "n_vox must be >= 0");
    if ((st = validate_opts(o, n_vox)) != GAC_OK) return st;
    if (!out) return fail(GAC_ERR_INVALID_ARG, "out must not be NULL");
    if (n_vox > 0 && !data) return fail(GAC_ERR_INVALID_ARG, "data must not be NULL");
    if (!sigma && !(sigma_scalar > 0.0f && std::isfinite(sigma_scalar)))
        return fail(GAC_ERR_INVALID_ARG, "sigma is NULL and sigma_scalar is not a positive number");
    if (o->trace_n_vox > 0 && !out->trace)
        return fail(GAC_ERR_INVALID_ARG, "trace_n_vox > 0 needs out->trace");
    int lanes = 1;  // lanes per chain: a requested count is checked before anything runs
    if (o->lanes_per_chain > 1 && (st = choose_lanes(mc, o, n_vox, &lanes)) != GAC_OK) return st;
    if (n_vox == 0) return GAC_OK;
    if (o->lanes_per_chain == 0 && (st = choose_lanes(mc, o, n_vox, &lanes)) != GAC_OK) return st;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    keep_staging_pool();
    const int P = mc.n_par, C = o->n_chains, M = mc.n_meas;
    const int S = n_samples(o->iterations, o->burnin, o->thin);
    const size_t N = static_cast<size_t>(n_vox);

    DevBuf d_data, d_sigma, d_x0, d_mean, d_std, d_samples, d_acc, d_bad, d_trace, d_rhat, d_scale;
    if ((st = d_data.make(const_cast<void *>(data), N * M * sizeof(float), true, s, "data")) != GAC_OK) return st;
    if ((st = d_sigma.make(const_cast<float *>(sigma), sigma ? N * sizeof(float) : 0, true, s, "sigma")) != GAC_OK) return st;
    if ((st = d_x0.make(const_cast<float *>(x0), x0 ? N * C * P * sizeof(float) : 0, true, s, "x0")) != GAC_OK) return st;
    if ((st = d_mean.make(out->mean, P * N * sizeof(double), false, s, "mean")) != GAC_OK) return st;
    if ((st = d_std.make(out->std, P * N * sizeof(double), false, s, "std")) != GAC_OK) return st;
    if ((st = d_samples.make(out->samples, static_cast<size_t>(S) * C * P * N * sizeof(float), false, s, "samples")) != GAC_OK) return st;
    if ((st = d_acc.make(out->accept_rate, C * N * sizeof(float), false, s, "accept_rate")) != GAC_OK) return st;
    if ((st = d_bad.make(out->nonfinite, C * N * sizeof(int32_t), false, s, "nonfinite")) != GAC_OK) return st;
    if ((st = d_trace.make(out->trace, static_cast<size_t>(o->trace_n_vox) * C * o->iterations * sizeof(gac_trace_rec), false, s, "trace")) != GAC_OK) return st;
    if ((st = d_rhat.make(out->rhat, P * N * sizeof(double), false, s, "rhat")) != GAC_OK) return st;
    if ((st = d_scale.make(out->step_scale, C * N * sizeof(float), false, s, "step_scale")) != GAC_OK) return st;

    const bool trace = o->trace_n_vox > 0;
    LaunchCfg cfg{};
    int64_t n_tiles = 0;
    int vb = 0;
    const int depth = choose_depth(mc, o, n_vox, lanes > 1);
    st = depth > 0 ? plan_spec(mc, depth, C, n_vox, o->moments_mode, &cfg, &n_tiles, &vb)
       : lanes > 1 ? plan_split(mc, lanes, C, n_vox, o->moments_mode, &cfg, &n_tiles, &vb)
                   : plan_launch(mc, o->precision, trace, C, n_vox, o->moments_mode, &cfg, &n_tiles, &vb);
    if (st != GAC_OK) return st;
    // slices read the data once each: not over the link from host memory
    SlicePlan sp;
    if (depth == 0 && lanes == 1 && is_device_ptr(d_data.ptr) &&
        (st = plan_slices(mc, o, n_vox, cfg, n_tiles, &sp)) != GAC_OK)
        return st;
    const bool all = o->moments_mode == GAC_MOMENTS_ALL_POSTBURNIN;
    SliceState ss{};
    DevBuf d_state;  // freed in stream order
    if (sp.fn) {
        d_state.stream = s;
        if (cudaMallocAsync(&d_state.ptr, slice_state(mc, n_vox * C, all, nullptr, nullptr), s) == cudaSuccess) {
            d_state.owned = true;
            slice_state(mc, n_vox * C, all, static_cast<char *>(d_state.ptr), &ss);
            n_tiles = sp.n_tiles;
            vb = sp.vb;
        } else {  // no memory for the state: one launch
            cudaGetLastError();
            d_state.ptr = nullptr;
            sp.fn = nullptr;
        }
    }

    RunArgs ra;
    std::memset(&ra, 0, sizeof ra);
    ra.data = static_cast<const float *>(d_data.ptr);
    ra.sigma = static_cast<const float *>(d_sigma.ptr);
    ra.sigma_scalar = sigma_scalar;
    ra.x0 = static_cast<const float *>(d_x0.ptr);
    ra.mean = static_cast<double *>(d_mean.ptr);
    ra.std = static_cast<double *>(d_std.ptr);
    ra.samples = static_cast<float *>(d_samples.ptr);
    ra.accept = static_cast<float *>(d_acc.ptr);
    ra.nonfinite = static_cast<int32_t *>(d_bad.ptr);
    ra.trace = static_cast<gac_trace_rec *>(d_trace.ptr);
    ra.n_vox = n_vox;
    ra.C = C;
    ra.I = o->iterations;
    ra.B = o->burnin;
    ra.T = o->thin;
    ra.S = S;
    ra.k0 = static_cast<uint32_t>(o->seed & 0xFFFFFFFFu);
    ra.k1 = static_cast<uint32_t>(o->seed >> 32);
    ra.voxel_base = o->voxel_base;
    ra.moments_mode = o->moments_mode;
    ra.trace_n = o->trace_n_vox;
    ra.vox_per_block = vb;
    ra.row_stride = row_stride_for(mc.kind, M);
    ra.data_vec4 = (M % 4 == 0) && ((reinterpret_cast<uintptr_t>(ra.data) & 15) == 0);
    ra.n_tiles = n_tiles;
    ra.sampling_threads = cfg.sampling;
    set_adaptation(ra, o);
    ra.rhat = static_cast<double *>(d_rhat.ptr);
    ra.step_scale = static_cast<float *>(d_scale.ptr);

    cudaError_t e = cudaSuccess;
    if (sp.fn) {
        const int64_t end = sp.count * sp.n_tiles;
        for (int64_t pos = 0; pos < end && e == cudaSuccess; pos += sp.slots) {
            void *args[] = {&mc, &ra, &ss, &pos, &sp.q};
            e = cudaLaunchKernel(sp.fn, dim3(static_cast<unsigned>(std::min<int64_t>(sp.slots, end - pos))), dim3(kBlock), args, sp.smem, s);
        }
    } else {
        void *args[] = {&mc, &ra};
        e = cudaLaunchKernel(cfg.fn, dim3(cfg.grid), dim3(cfg.block), args, cfg.smem, s);
    }
    if (e != cudaSuccess) return cuda_fail(e, "MH kernel launch");
    for (DevBuf *b : {&d_mean, &d_std, &d_samples, &d_acc, &d_bad, &d_trace, &d_rhat, &d_scale})
        if ((st = b->copy_out()) != GAC_OK) return st;
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "MH kernel");
    return GAC_OK;
}

}  // extern "C"
