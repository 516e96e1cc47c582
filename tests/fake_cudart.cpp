// fake_cudart.cpp -- a CUDA runtime without a GPU, preloaded by
// test_launches_cpu.py: memory is host memory, kernels do not run, and every
// copy, launch and shared-memory limit is written down in order.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
std::mutex mu;
std::string text, given;
std::map<const void *, std::string> names;  // host stub -> kernel
std::map<const void *, size_t> limits;      // dynamic shared memory a kernel may have
struct Call {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local std::vector<Call> calls;
uintptr_t handles = 0;

void put(const std::string &line) {
    std::lock_guard<std::mutex> lock(mu);
    text += line + "\n";
}
std::string at(const void *s) {
    char b[32];
    std::snprintf(b, sizeof b, "%p", s);
    return b;
}
cudaError_t launch(const void *fun, dim3 g, size_t smem, cudaStream_t s) {
    put("launch " + names[fun] + " grid=" + std::to_string(g.x) + "," + std::to_string(g.y) +
        " smem=" + std::to_string(smem) + " stream=" + at(s));
    std::lock_guard<std::mutex> lock(mu);
    return smem > 48 * 1024 && smem > limits[fun] ? cudaErrorInvalidValue : cudaSuccess;
}
template <typename T>
cudaError_t handle(T *out) {
    *out = reinterpret_cast<T>(++handles << 8);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// What was written down so far; starts anew.
const char *fake_cudart_log() {
    std::lock_guard<std::mutex> lock(mu);
    given.swap(text);
    text.clear();
    return given.c_str();
}

void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *stub, char *, const char *name, int, uint3 *, uint3 *, dim3 *,
                            dim3 *, int *) {
    names[stub] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
    calls.push_back({g, b, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    const Call c = calls.back();
    calls.pop_back();
    *g = c.grid;
    *b = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t *>(s) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *stub) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(stub));
    return cudaSuccess;
}
static thread_local cudaError_t last = cudaSuccess;
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void **, size_t smem, cudaStream_t s) {
    return last = launch(k, g, smem, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fun, void **) {
    return last = launch(fun, c->gridDim, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaFuncSetAttribute(const void *fun, cudaFuncAttribute, int value) {
    put("limit " + names[fun] + " " + std::to_string(value));
    std::lock_guard<std::mutex> lock(mu);
    limits[fun] = (size_t)value;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 3;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t n) { return (*p = std::aligned_alloc(256, (n + 255) / 256 * 256)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    put("copy bytes=" + std::to_string(n));
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    put("copy bytes=" + std::to_string(n) + " stream=" + at(st));
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidSymbol; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
    std::memset(a, 0, sizeof *a);
    return cudaSuccess;
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b) { *a = 0; *b = -5; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return handle(s); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
}
