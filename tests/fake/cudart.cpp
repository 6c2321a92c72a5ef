// A CUDA runtime for tests of the library's host code without a GPU: several devices whose
// memory is host memory, kernels that are checked against their launch limits and not run,
// streams, events and graphs that do nothing, and allocations that fail on request.  Linked
// with the library's objects in place of the real runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <utility>

namespace {

constexpr int kDevices = 2, kStaticLimit = 48 * 1024;
std::mutex mu;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
std::map<std::pair<int, const void*>, int> limit;   // dynamic shared memory per (device, kernel)
std::set<void*> live;
int bad_frees = 0, fail_after = -1, capturing_error = 0, refuse_attr = 0;
long launches = 0;
bool capturing = false;
int instantiated = 0;
int first_in_capture = 0;                           // kernels first launched inside a capture
std::set<std::pair<int, const void*>> seen;
struct Config {
    dim3 grid, block;
    size_t shared;
    void* stream;
};
thread_local Config pushed;

cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t launch(const void* k, size_t shared) {
    std::lock_guard<std::mutex> l(mu);
    auto it = limit.find({device, k});
    const size_t most = it == limit.end() ? kStaticLimit : it->second;
    if (shared > most && shared > (size_t)kStaticLimit) return done(cudaErrorInvalidValue);
    ++launches;
    if (seen.insert({device, k}).second && capturing) ++first_in_capture;
    return cudaSuccess;
}

}  // namespace

extern "C" {

// the tests' controls
int fake_bad_frees() { return bad_frees; }
int fake_live() { return (int)live.size(); }
long fake_launches() { return launches; }
void fake_fail_malloc(int after) { fail_after = after; }
void fake_capture_query_error(int on) { capturing_error = on; }
void fake_refuse_attribute(int on) { refuse_attr = on; }
int fake_set_device(int d) { return cudaSetDevice(d); }
int fake_last_error() { return last; }
int fake_instantiated() { return instantiated; }
int fake_first_in_capture() { return first_in_capture; }

cudaError_t cudaGetDeviceCount(int* n) { *n = kDevices; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) {
    if (d < 0 || d >= kDevices) return done(cudaErrorInvalidDevice);
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }

cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> l(mu);
    if (fail_after >= 0 && fail_after-- == 0) return done(cudaErrorMemoryAllocation);   // *p untouched
    *p = calloc(n ? n : 1, 1);
    live.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> l(mu);
    if (!p) return cudaSuccess;
    if (!live.erase(p)) { ++bad_frees; return done(cudaErrorInvalidValue); }
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return done(cudaErrorInvalidSymbol); }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long, cudaDriverEntryPointQueryResult*) {
    return done(cudaErrorNotSupported);
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    *c = cudaStreamCaptureStatusNone;
    return capturing_error ? done(cudaErrorStreamCaptureImplicit) : cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { capturing = true; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { capturing = false; *g = (cudaGraph_t)malloc(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { ++instantiated; *x = (cudaGraphExec_t)malloc(1); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { free(x); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }

cudaError_t cudaFuncSetAttribute(const void* k, cudaFuncAttribute a, int v) {
    std::lock_guard<std::mutex> l(mu);
    if (refuse_attr) return done(cudaErrorInvalidValue);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[{device, k}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* k, void**) { return launch(k, c->dynamicSmemBytes); }
cudaError_t __cudaGetKernel(cudaKernel_t* h, const void* k) { *h = (cudaKernel_t)k; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t shared, cudaStream_t) { return launch((const void*)k, shared); }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sh, void* s) { pushed = Config{g, b, sh, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sh, void* s) {
    *g = pushed.grid;
    *b = pushed.block;
    *sh = pushed.shared;
    *(void**)s = pushed.stream;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

}  // extern "C"
