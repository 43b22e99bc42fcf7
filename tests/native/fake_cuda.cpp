// The stand-in CUDA runtime of fake_cuda.h.
#include "fake_cuda.h"

#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace fake {

struct State {
    std::recursive_mutex mu;
    std::map<const void*, std::string> names;  // kernels, by host function
    std::map<std::string, long> launched;
    std::map<void*, size_t> live;              // device allocations
    long memsets = 0;
    long waits = 0;                             // cudaMalloc and cudaFree
    long fail_from = 0, fail_to = 0;           // device allocations [fail_from, fail_to) from now on fail (1: the next)
    cudaError_t last = cudaSuccess;
};
State& st() {
    static State* s = new State();  // outlives the static registrations
    return *s;
}
using Lock = std::lock_guard<std::recursive_mutex>;

void fail_after(long skip, long count) {
    Lock l(st().mu);
    st().fail_from = skip + 1;
    st().fail_to = skip + 1 + count;
}
void fail_none() { fail_after(-1, 0); }

size_t live_bytes() {
    Lock l(st().mu);
    size_t b = 0;
    for (const auto& kv : st().live) b += kv.second;
    return b;
}
long launches(const char* part) {
    Lock l(st().mu);
    long n = 0;
    for (const auto& kv : st().launched)
        if (kv.first.find(part) != std::string::npos) n += kv.second;
    return n;
}

bool last_error() {
    Lock l(st().mu);
    return st().last != cudaSuccess;
}
long memsets() {
    Lock l(st().mu);
    return st().memsets;
}
std::function<void(void*, size_t)> on_read;

long device_waits() {
    Lock l(st().mu);
    return st().waits;
}

cudaError_t alloc(void** p, size_t bytes, bool device) {
    Lock l(st().mu);
    *p = nullptr;
    if (device) {
        if (st().fail_from > 0) --st().fail_from;
        if (st().fail_to > 0) --st().fail_to;
        if (st().fail_from <= 0 && st().fail_to > 0) return st().last = cudaErrorMemoryAllocation;
    }
    *p = std::calloc(bytes ? bytes : 1, 1);
    if (device) st().live[*p] = bytes;
    return cudaSuccess;
}
cudaError_t release(void* p) {
    Lock l(st().mu);
    if (p && st().live.erase(p) == 0) return st().last = cudaErrorInvalidValue;
    std::free(p);
    return cudaSuccess;
}
cudaError_t launch(const void* f) {
    Lock l(st().mu);
    ++st().launched[st().names[f]];
    return cudaSuccess;
}
template <typename T>
T token() {
    return reinterpret_cast<T>(std::malloc(8));
}

}  // namespace fake

static void wait_all() {
    fake::Lock l(fake::st().mu);
    ++fake::st().waits;
}

extern "C" {

void** __cudaRegisterFatBinary(void*) {
    static void* h[1];
    return h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    fake::st().names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) { return fake::launch(k); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void**) { return fake::launch(f); }

cudaError_t cudaMalloc(void** p, size_t bytes) {
    wait_all();
    return fake::alloc(p, bytes, true);
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) {
    return fake::alloc(p, bytes, true);
}
cudaError_t cudaMallocHost(void** p, size_t bytes) { return fake::alloc(p, bytes, false); }
cudaError_t cudaFree(void* p) {
    wait_all();
    return fake::release(p);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
    return fake::release(p);
}
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    if (n) std::memcpy(d, s, n);
    if (k == cudaMemcpyDeviceToHost && fake::on_read) fake::on_read(d, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void* d, int v, size_t n) {
    {
        fake::Lock l(fake::st().mu);
        ++fake::st().memsets;
    }
    if (n) std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaMemGetInfo(size_t* fr, size_t* tot) {
    *fr = *tot = (size_t)1 << 38;
    return cudaSuccess;
}

cudaError_t cudaGetLastError() {
    fake::Lock l(fake::st().mu);
    const cudaError_t e = fake::st().last;
    fake::st().last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 129 << 20;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) {
    *lo = *hi = 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) {
    *s = fake::token<cudaStream_t>();
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    std::free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = fake::token<cudaGraph_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    std::free(g);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = fake::token<cudaGraphExec_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = fake::token<cudaEvent_t>();
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}

}  // extern "C"
