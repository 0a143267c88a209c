// A stand-in for the CUDA runtime, so that the library's host code runs on a
// machine without a GPU: "device" memory is host memory, kernels are not run.  The
// calls that a test wants to see or to fail go to one callback; everything else
// succeeds and does nothing.  Linked with the library's object files in the
// runtime's place (fake_gpu.py).
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

// op: "malloc" (x: bytes), "free" (x: bytes), "attr" (x: attribute, value), "launch" (x: grid
// x, grid y, block, dynamic shared bytes; args: the kernel's) return an error code or 0;
// ("attr" once it is set); "occupancy" (x: block, dynamic shared bytes) returns resident blocks an SM.
using Hook = int (*)(const char *op, const char *kernel, const long long *x, void **args);

namespace {
Hook g_hook = nullptr;
std::map<const void *, std::string> &names() {
    static std::map<const void *, std::string> m;
    return m;
}
std::map<const void *, size_t> g_limit;  // a kernel's dynamic shared-memory limit
std::map<const void *, size_t> g_alloc;  // device allocations and marked buffers
constexpr size_t kStatic = 1024;         // every kernel's static shared memory
cudaError_t call(const char *op, const void *fn, long long a, long long b, long long c = 0, long long d = 0, void **args = nullptr) {
    const long long x[4] = {a, b, c, d};
    return g_hook ? static_cast<cudaError_t>(g_hook(op, fn ? names()[fn].c_str() : "", x, args)) : cudaSuccess;
}
thread_local cudaError_t t_last = cudaSuccess;  // of the last failed launch
size_t limit(const void *fn) { return g_limit.count(fn) ? g_limit[fn] : 48 * 1024 - kStatic; }
cudaError_t alloc(void **p, size_t n) {
    const cudaError_t e = call("malloc", nullptr, static_cast<long long>(n), 0);
    if (e != cudaSuccess) return e;
    *p = std::malloc(n + 256);
    g_alloc[*p] = n;
    return cudaSuccess;
}
cudaError_t release(void *p) {
    if (!g_alloc.count(p)) return cudaErrorInvalidValue;
    call("free", nullptr, static_cast<long long>(g_alloc[p]), 0);
    g_alloc.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t launch(const void *fn, dim3 grid, dim3 block, void **args, size_t smem) {
    const bool bad = smem > limit(fn) || grid.x < 1 || grid.x > 2147483647u || block.x < 1 || block.x > 1024;
    const cudaError_t e = bad ? cudaErrorInvalidValue : call("launch", fn, grid.x, grid.y, block.x, static_cast<long long>(smem), args);
    if (e != cudaSuccess) t_last = e;
    return e;
}
}  // namespace

extern "C" {
void fake_set_hook(Hook h) { g_hook = h; }
void fake_forget_limits() { g_limit.clear(); }
void fake_mark_device(void *p, int on) {
    if (on) g_alloc[p] = 0;
    else g_alloc.erase(p);
}

void **__cudaRegisterFatBinary(void *) { return reinterpret_cast<void **>(&g_hook); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) { names()[host] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(fn));
    return cudaSuccess;
}
static thread_local struct { dim3 grid, block; size_t smem; void *stream; } t_cfg;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *stream) {
    t_cfg = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = t_cfg.grid;
    *block = t_cfg.block;
    *smem = t_cfg.smem;
    *static_cast<void **>(stream) = t_cfg.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t fn, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t) { return launch(fn, grid, block, args, smem); }
cudaError_t cudaLaunchKernel(const void *fn, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t) { return launch(fn, grid, block, args, smem); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) { return launch(fn, c->gridDim, c->blockDim, args, c->dynamicSmemBytes); }

cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (v < 0 || v + kStatic > 227 * 1024) return cudaErrorInvalidValue;
        g_limit[fn] = v;
    }
    return call("attr", fn, a, v);
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *fn) {
    std::memset(a, 0, sizeof *a);
    a->sharedSizeBytes = kStatic;
    a->maxDynamicSharedSizeBytes = static_cast<int>(limit(fn));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *fn, int block, size_t smem) {
    *n = call("occupancy", fn, block, static_cast<long long>(smem));
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024
         : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor                       ? 228 * 1024
                                                                                 : 0;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    std::memset(a, 0, sizeof *a);
    if (g_alloc.count(p)) a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaMalloc(void **p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return (*p = std::malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return release(p); }
cudaError_t cudaFree(void *p) { return p ? release(p) : cudaSuccess; }
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = t_last;
    t_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t *, int) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
}
