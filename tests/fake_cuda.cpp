// A CUDA runtime on the host, for tests of the library's error paths without a
// GPU: the library's objects are linked against it instead of libcudart.
// Memory is host memory, copies copy at once, kernels are named and counted but
// do nothing, and any call or launch can be made to fail with an error code.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::map<const void*, std::string>& kernels() {   // filled before main, by the other objects
    static std::map<const void*, std::string> k;
    return k;
}
std::map<char*, size_t> device;          // allocations by base
std::string log_, fail_what;
int fail_in = 0, hits = 0;               // the fail_in-th match from now on fails
cudaError_t last = cudaSuccess;
dim3 cfg_grid, cfg_block;
size_t cfg_sm;
cudaStream_t cfg_stream;
bool capturing = false;
cudaStream_t captured;

cudaError_t call(const std::string& what, const void* on = nullptr) {
    log_ += what;
    if (on) log_ += " " + std::to_string((size_t)on);
    if (fail_in > 0 && what.find(fail_what) != std::string::npos && --fail_in == 0) {
        ++hits;
        log_ += " FAILS\n";
        return last = cudaErrorMemoryAllocation;
    }
    log_ += "\n";
    return cudaSuccess;
}
template <typename T>
cudaError_t handle(const char* what, T* out) {
    static size_t next = 16;
    const cudaError_t e = call(what);
    if (e == cudaSuccess) *out = (T)(next += 16);
    return e;
}
cudaError_t alloc(const char* what, void** p, size_t n, bool dev) {
    const cudaError_t e = call(what);
    if (e != cudaSuccess) return e;
    *p = std::calloc(n ? n : 1, 1);
    if (dev) device[(char*)*p] = n;
    return cudaSuccess;
}
cudaError_t launch(const void* f, cudaStream_t st) { return call("launch " + kernels()[f], st); }
}  // namespace

extern "C" {
// ---- for the tests
void fake_fail(const char* what, int nth) {
    fail_what = what;
    fail_in = nth;
    hits = 0;
}
int fake_hits() { return hits; }
void fake_clear() { log_.clear(); }
const char* fake_log() { return log_.c_str(); }

// ---- kernels
void** __cudaRegisterFatBinary(void*) { return (void**)&kernels(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    kernels()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t st) {
    cfg_grid = g;
    cfg_block = b;
    cfg_sm = sm;
    cfg_stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* st) {
    *g = cfg_grid;
    *b = cfg_block;
    *sm = cfg_sm;
    *(cudaStream_t*)st = cfg_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t st) {
    return launch((const void*)k, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->stream); }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = 1;
    return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDeviceCount(int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    std::memset(p, 0, sizeof(*p));
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "an error made by the test"; }

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) { return alloc("cudaMalloc", p, n, true); }
cudaError_t cudaMallocHost(void** p, size_t n) { return alloc("cudaMallocHost", p, n, false); }
cudaError_t cudaFree(void* p) {
    device.erase((char*)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof(*a));
    auto it = device.upper_bound((char*)p);
    if (it != device.begin()) {
        --it;
        if ((const char*)p < it->first + it->second) a->type = cudaMemoryTypeDevice;
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return call("cudaMemcpy");
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (!(capturing && st == captured)) std::memcpy(d, s, n);
    return call("cudaMemcpyAsync", st);
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
    *p = (void*)s;
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) {
    if (!(capturing && st == captured)) std::memset(p, v, n);
    return call("cudaMemsetAsync", st);
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle("cudaStreamCreateWithFlags", s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return call("cudaStreamSynchronize", s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return call("cudaStreamWaitEvent", s); }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = capturing && s == captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    const cudaError_t e = call("cudaStreamBeginCapture", s);
    if (e == cudaSuccess) capturing = true, captured = s;
    return e;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
    capturing = false;
    const cudaError_t e = call("cudaStreamEndCapture", s);
    *g = e == cudaSuccess ? (cudaGraph_t)1 : nullptr;
    return e;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    return handle("cudaGraphInstantiate", x);
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { return call("cudaGraphLaunch", s); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle("cudaEventCreate", e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle("cudaEventCreateWithFlags", e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) { return call("cudaEventRecord", s); }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t s, unsigned) { return call("cudaEventRecordWithFlags", s); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return call("cudaEventSynchronize"); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
}
