// Test and data-synthesis entry points of the C ABI: the forward model and
// likelihood at given parameters, and the random-number layer.  They run the
// same device functions as the sampler.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "gac.h"
#include "gac_internal.h"
#include "mh_kernel.cuh"

namespace gac {

// FP64: a thread per parameter vector, which writes its row as it evaluates.
template <int KIND>
__global__ void forward_d_kernel(const ModelConst mc, const double *theta, int64_t n, double *s) {
    constexpr int P = model_n_par(KIND);
    const int M = mc.n_meas;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double *out = s + i * M;
        double th[P];
        for (int p = 0; p < P; ++p) th[p] = theta[i * P + p];
        if constexpr (model_complex(KIND))
            eval_d<KIND>(th, mc, [&](int k, double re, double im) { out[2 * k] = re; out[2 * k + 1] = im; });
        else
            eval_d<KIND>(th, mc, [&](int k, double v) { out[k] = v; });
    }
}

// FP32 arithmetic (the MIXED and FP32 paths share the forward model): bound by
// the bytes of its rows, so they cross shared memory.  A warp takes 32
// consecutive parameter vectors: it reads them as one contiguous piece, each
// lane evaluates one of them into its row of the warp's tile, and the warp
// writes the 32 rows as one contiguous piece.  (A thread writing its own row
// touched 32 lines with every store: 3-pool, 24 echoes, 500,000 vectors took
// 292 us a call, 73 so, of which about 20 are the launch and the wait of any
// call; their 228 MB cross HBM in 34.)
constexpr int kFwdBlock = 128;
template <int KIND>
__global__ void __launch_bounds__(kFwdBlock) forward_f_kernel(const ModelConst mc, const double *theta, int64_t n,
                                                              double *s, int row_stride) {
    constexpr int P = model_n_par(KIND);
    extern __shared__ __align__(16) float fwd_rows[];
    const int M = mc.n_meas;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *tile = fwd_rows + warp * 32 * row_stride;
    model_smem_load<KIND, 1>(mc);
    __syncthreads();
    const int64_t tiles = (n + 31) / 32;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(kFwdBlock / 32) + warp; t < tiles;
         t += static_cast<int64_t>(gridDim.x) * (kFwdBlock / 32)) {
        const int64_t left = n - t * 32;
        const int rows = left < 32 ? static_cast<int>(left) : 32;
        const double *src = theta + t * 32 * P;
        float th[P];
#pragma unroll
        for (int p = 0; p < P; ++p)  // row_stride >= P (the host sees to it)
            if (lane + 32 * p < rows * P) tile[lane + 32 * p] = static_cast<float>(src[lane + 32 * p]);
        __syncwarp();
        const int r = min(lane, rows - 1);  // a lane without a vector repeats the last
#pragma unroll
        for (int p = 0; p < P; ++p) th[p] = tile[r * P + p];
        __syncwarp();
        float *row = tile + lane * row_stride;
        if constexpr (model_complex(KIND))
            eval_f<KIND, 1>(th, mc, [&](int k, float re, float im) { reinterpret_cast<float2 *>(row)[k] = make_float2(re, im); });
        else
            eval_f<KIND, 1>(th, mc, [&](int k, float v) { row[k] = v; });
        __syncwarp();
        double *out = s + t * 32 * M;
        int q = lane / M, col = lane - q * M;  // element e = lane + 32 i of the rows as one piece
        const int dq = 32 / M, dc = 32 - dq * M;
        for (int e = lane; e < rows * M; e += 32) {
            out[e] = static_cast<double>(tile[q * row_stride + col]);
            q += dq;
            col += dc;
            if (col >= M) {
                col -= M;
                ++q;
            }
        }
        __syncwarp();
    }
}

template <int KIND, int PREC>
__global__ void loglik_kernel(const ModelConst mc, const double *theta, int64_t n, const float *y,
                              const float *sigma, double *L) {
    constexpr int P = model_n_par(KIND);
    using R = typename PrecTraits<PREC>::R;
    const int M = mc.n_meas;
    model_smem_load<KIND, 1>(mc);
    __syncthreads();
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        R th[P];
        for (int p = 0; p < P; ++p) th[p] = static_cast<R>(theta[i * P + p]);
        const R sg = static_cast<R>(sigma[i]);
        L[i] = static_cast<double>(loglik_any<KIND, PREC, 1>(th, y + i * M, R(1) / (sg * sg), mc));
    }
}

__global__ void philox_kernel(uint32_t k0, uint32_t k1, const uint32_t *t, const uint32_t *v,
                              const uint32_t *c, int64_t n, int nw, uint32_t *out) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        for (int k = 0; 4 * k < nw; ++k) {
            Words4 o = philox4x32_10(t[i], v[i], (c[i] << 8) | static_cast<uint32_t>(k), 0u, k0, k1);
            for (int j = 0; j < 4 && 4 * k + j < nw; ++j) out[i * nw + 4 * k + j] = o.w[j];
        }
    }
}

template <int P, int PREC>
__global__ void normals_kernel(uint32_t k0, uint32_t k1, const uint32_t *t, const uint32_t *v,
                               const uint32_t *c, int64_t n, double *z, uint32_t *w_acc) {
    constexpr int NW = n_words(P);
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        uint32_t w[4 * n_calls(P)];
        draw_words(w, t[i], v[i], c[i], k0, k1);
        for (int j = 0; 2 * j < P; ++j) {
            if constexpr (PREC == GAC_PREC_FP64) {
                double a, b;
                box_muller_d(w[2 * j], w[2 * j + 1], a, b);
                z[i * P + 2 * j] = a;
                if (2 * j + 1 < P) z[i * P + 2 * j + 1] = b;
            } else {
                float a, b;
                box_muller_f(w[2 * j], w[2 * j + 1], a, b);
                z[i * P + 2 * j] = a;
                if (2 * j + 1 < P) z[i * P + 2 * j + 1] = b;
            }
        }
        w_acc[i] = w[NW - 1];
    }
}

static int grid_for(int64_t n) {
    const int64_t blocks = (n + 255) / 256;
    return static_cast<int>(blocks < 4096 ? (blocks > 0 ? blocks : 1) : 4096);
}

template <int KIND>
static cudaError_t launch_forward(int prec, const ModelConst &mc, const double *th, int64_t n, double *s,
                                  cudaStream_t st) {
    if (prec == GAC_PREC_FP64) {
        forward_d_kernel<KIND><<<grid_for(n), 256, 0, st>>>(mc, th, n, s);
        return cudaGetLastError();
    }
    const int row_stride = row_stride_for(KIND, std::max(mc.n_meas, mc.n_par));
    const size_t smem = static_cast<size_t>(kFwdBlock) * row_stride * sizeof(float);
    if (smem > 44 * 1024) {  // beside the model's tables, past the default 48 KB
        const cudaError_t lim = allow_smem(reinterpret_cast<const void *>(&forward_f_kernel<KIND>), smem);
        if (lim != cudaSuccess) return lim;
    }
    // one wave: 8 blocks an SM, or as many as its shared memory holds (long rows, the
    // models' tables and the system's kilobyte)
    constexpr int kBeside = KIND == GAC_MODEL_SMT || KIND == GAC_MODEL_AXCAL_SMT ? 6 * 1024 : 1024;
    int dev = 0, sms = 0, smem_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e != cudaSuccess) return e;
    const int64_t per_sm = std::min<int64_t>(8, std::max<int64_t>(1, smem_sm / static_cast<int64_t>(smem + kBeside)));
    const int64_t blocks = (n + kFwdBlock - 1) / kFwdBlock;
    const int grid = static_cast<int>(std::min<int64_t>(blocks, sms * per_sm));
    forward_f_kernel<KIND><<<grid, kFwdBlock, smem, st>>>(mc, th, n, s, row_stride);
    return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_loglik(int prec, const ModelConst &mc, const double *th, int64_t n, const float *y,
                                 const float *sg, double *L, cudaStream_t st) {
    switch (prec) {
    case GAC_PREC_MIXED: loglik_kernel<KIND, GAC_PREC_MIXED><<<grid_for(n), 256, 0, st>>>(mc, th, n, y, sg, L); break;
    case GAC_PREC_FP32: loglik_kernel<KIND, GAC_PREC_FP32><<<grid_for(n), 256, 0, st>>>(mc, th, n, y, sg, L); break;
    default: loglik_kernel<KIND, GAC_PREC_FP64><<<grid_for(n), 256, 0, st>>>(mc, th, n, y, sg, L); break;
    }
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_normals_p(int prec, uint64_t seed, const uint32_t *t, const uint32_t *v, const uint32_t *c,
                                   int64_t n, double *z, uint32_t *w, cudaStream_t cs) {
    const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    if (prec == GAC_PREC_FP64) normals_kernel<P, GAC_PREC_FP64><<<grid_for(n), 256, 0, cs>>>(k0, k1, t, v, c, n, z, w);
    else normals_kernel<P, GAC_PREC_MIXED><<<grid_for(n), 256, 0, cs>>>(k0, k1, t, v, c, n, z, w);
    return cudaGetLastError();
}

}  // namespace gac

using namespace gac;

extern "C" {

gac_status gac_forward(int model_id, const double *theta, int64_t n, int precision, double *s, void *stream) {
    clear_error();
    ModelConst mc;
    gac_status st = model_get(model_id, &mc);
    if (st != GAC_OK) return st;
    if (n < 0 || (n > 0 && (!theta || !s))) return fail(GAC_ERR_INVALID_ARG, "bad theta/s/n");
    if (precision < GAC_PREC_MIXED || precision > GAC_PREC_FP64)
        return fail(GAC_ERR_INVALID_ARG, "unknown precision %d", precision);
    if (n == 0) return GAC_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    DevBuf dth, ds;
    if ((st = dth.make(const_cast<double *>(theta), n * mc.n_par * sizeof(double), true, cs, "theta")) != GAC_OK) return st;
    if ((st = ds.make(s, n * mc.n_meas * sizeof(double), false, cs, "s")) != GAC_OK) return st;
    const double *th = static_cast<const double *>(dth.ptr);
    double *out = static_cast<double *>(ds.ptr);
    cudaError_t e;
    switch (mc.kind) {
    case GAC_MODEL_MONOEXP: e = launch_forward<GAC_MODEL_MONOEXP>(precision, mc, th, n, out, cs); break;
    case GAC_MODEL_MWI3: e = launch_forward<GAC_MODEL_MWI3>(precision, mc, th, n, out, cs); break;
    case GAC_MODEL_SMT: e = launch_forward<GAC_MODEL_SMT>(precision, mc, th, n, out, cs); break;
    case GAC_MODEL_AXCAL_SMT: e = launch_forward<GAC_MODEL_AXCAL_SMT>(precision, mc, th, n, out, cs); break;
    default: e = launch_forward<GAC_MODEL_LINEAR_TEST>(precision, mc, th, n, out, cs); break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "forward kernel launch");
    if ((st = ds.copy_out()) != GAC_OK) return st;
    e = cudaStreamSynchronize(cs);
    return e == cudaSuccess ? GAC_OK : cuda_fail(e, "forward kernel");
}

gac_status gac_loglik(int model_id, const double *theta, int64_t n, const float *data, const float *sigma,
                      int precision, double *L, void *stream) {
    clear_error();
    ModelConst mc;
    gac_status st = model_get(model_id, &mc);
    if (st != GAC_OK) return st;
    if (n < 0 || (n > 0 && (!theta || !data || !sigma || !L))) return fail(GAC_ERR_INVALID_ARG, "bad arguments");
    if (precision < GAC_PREC_MIXED || precision > GAC_PREC_FP64)
        return fail(GAC_ERR_INVALID_ARG, "unknown precision %d", precision);
    if (n == 0) return GAC_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    DevBuf dth, dy, dsg, dl;
    if ((st = dth.make(const_cast<double *>(theta), n * mc.n_par * sizeof(double), true, cs, "theta")) != GAC_OK) return st;
    if ((st = dy.make(const_cast<float *>(data), n * mc.n_meas * sizeof(float), true, cs, "data")) != GAC_OK) return st;
    if ((st = dsg.make(const_cast<float *>(sigma), n * sizeof(float), true, cs, "sigma")) != GAC_OK) return st;
    if ((st = dl.make(L, n * sizeof(double), false, cs, "L")) != GAC_OK) return st;
    const double *th = static_cast<const double *>(dth.ptr);
    const float *y = static_cast<const float *>(dy.ptr);
    const float *sg = static_cast<const float *>(dsg.ptr);
    double *out = static_cast<double *>(dl.ptr);
    cudaError_t e;
    switch (mc.kind) {
    case GAC_MODEL_MONOEXP: e = launch_loglik<GAC_MODEL_MONOEXP>(precision, mc, th, n, y, sg, out, cs); break;
    case GAC_MODEL_MWI3: e = launch_loglik<GAC_MODEL_MWI3>(precision, mc, th, n, y, sg, out, cs); break;
    case GAC_MODEL_SMT: e = launch_loglik<GAC_MODEL_SMT>(precision, mc, th, n, y, sg, out, cs); break;
    case GAC_MODEL_AXCAL_SMT: e = launch_loglik<GAC_MODEL_AXCAL_SMT>(precision, mc, th, n, y, sg, out, cs); break;
    default: e = launch_loglik<GAC_MODEL_LINEAR_TEST>(precision, mc, th, n, y, sg, out, cs); break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "loglik kernel launch");
    if ((st = dl.copy_out()) != GAC_OK) return st;
    e = cudaStreamSynchronize(cs);
    return e == cudaSuccess ? GAC_OK : cuda_fail(e, "loglik kernel");
}

gac_status gac_philox_words(uint64_t seed, const uint32_t *t, const uint32_t *v, const uint32_t *c, int64_t n,
                            int n_words_, uint32_t *out, void *stream) {
    clear_error();
    if (n < 0 || n_words_ < 1 || n_words_ > 1024 || (n > 0 && (!t || !v || !c || !out)))
        return fail(GAC_ERR_INVALID_ARG, "bad arguments");
    if (n == 0) return GAC_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    DevBuf dt, dv, dc, dout;
    gac_status st;
    if ((st = dt.make(const_cast<uint32_t *>(t), n * 4, true, cs, "t")) != GAC_OK) return st;
    if ((st = dv.make(const_cast<uint32_t *>(v), n * 4, true, cs, "v")) != GAC_OK) return st;
    if ((st = dc.make(const_cast<uint32_t *>(c), n * 4, true, cs, "c")) != GAC_OK) return st;
    if ((st = dout.make(out, n * n_words_ * 4, false, cs, "out")) != GAC_OK) return st;
    philox_kernel<<<grid_for(n), 256, 0, cs>>>(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32),
                                              static_cast<const uint32_t *>(dt.ptr), static_cast<const uint32_t *>(dv.ptr),
                                              static_cast<const uint32_t *>(dc.ptr), n, n_words_,
                                              static_cast<uint32_t *>(dout.ptr));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "philox kernel launch");
    if ((st = dout.copy_out()) != GAC_OK) return st;
    e = cudaStreamSynchronize(cs);
    return e == cudaSuccess ? GAC_OK : cuda_fail(e, "philox kernel");
}

gac_status gac_normals(uint64_t seed, const uint32_t *t, const uint32_t *v, const uint32_t *c, int64_t n,
                       int n_par, int precision, double *z, uint32_t *w_acc, void *stream) {
    clear_error();
    if (n < 0 || (n > 0 && (!t || !v || !c || !z || !w_acc)))
        return fail(GAC_ERR_INVALID_ARG, "bad arguments");
    if (n_par != 2 && n_par != 4 && n_par != 9)
        return fail(GAC_ERR_INVALID_ARG, "n_par must be 2, 4 or 9 (the registered kinds)");
    if (precision < GAC_PREC_MIXED || precision > GAC_PREC_FP64)
        return fail(GAC_ERR_INVALID_ARG, "unknown precision %d", precision);
    if (n == 0) return GAC_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    DevBuf dt, dv, dc, dz, dw;
    gac_status st;
    if ((st = dt.make(const_cast<uint32_t *>(t), n * 4, true, cs, "t")) != GAC_OK) return st;
    if ((st = dv.make(const_cast<uint32_t *>(v), n * 4, true, cs, "v")) != GAC_OK) return st;
    if ((st = dc.make(const_cast<uint32_t *>(c), n * 4, true, cs, "c")) != GAC_OK) return st;
    if ((st = dz.make(z, n * n_par * sizeof(double), false, cs, "z")) != GAC_OK) return st;
    if ((st = dw.make(w_acc, n * 4, false, cs, "w_acc")) != GAC_OK) return st;
    const uint32_t *pt = static_cast<const uint32_t *>(dt.ptr), *pv = static_cast<const uint32_t *>(dv.ptr),
                   *pc = static_cast<const uint32_t *>(dc.ptr);
    double *pz = static_cast<double *>(dz.ptr);
    uint32_t *pw = static_cast<uint32_t *>(dw.ptr);
    cudaError_t e = n_par == 2 ? launch_normals_p<2>(precision, seed, pt, pv, pc, n, pz, pw, cs)
                  : n_par == 4 ? launch_normals_p<4>(precision, seed, pt, pv, pc, n, pz, pw, cs)
                               : launch_normals_p<9>(precision, seed, pt, pv, pc, n, pz, pw, cs);
    if (e != cudaSuccess) return cuda_fail(e, "normals kernel launch");
    if ((st = dz.copy_out()) != GAC_OK) return st;
    if ((st = dw.copy_out()) != GAC_OK) return st;
    e = cudaStreamSynchronize(cs);
    return e == cudaSuccess ? GAC_OK : cuda_fail(e, "normals kernel");
}

}  // extern "C"
