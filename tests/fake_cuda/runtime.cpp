// A CUDA runtime without a device, for tests of the library's host code: memory
// is host memory, nothing is executed, and every call that enqueues, orders or
// waits is written to a log, one line each ("op stream operands").  fake_fail
// makes a later call return an error, fake_capturing marks a stream as being
// captured, fake_pin marks host memory as page-locked.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {

std::string g_log;
// host stub -> device name (made on first use: kernels are registered before this file's variables are set up)
std::map<const void*, std::string>& kernels() {
    static auto* k = new std::map<const void*, std::string>;
    return *k;
}
std::map<uintptr_t, size_t> g_pinned;              // page-locked ranges
std::map<std::string, int> g_fail;                 // op -> calls until it fails
cudaStream_t g_capturing = nullptr;
bool g_any_capture = false;
cudaStream_t g_begun = nullptr;                    // stream whose work the library itself captures
uintptr_t g_next = 1;
struct { dim3 grid, block; size_t smem; cudaStream_t stream; } g_config;

template <typename... T>
void note(const char* fmt, T... v) {
    char line[512];
    std::snprintf(line, sizeof line, fmt, v...);
    g_log += line;
    g_log += '\n';
}

// Counts a call of `op`; true when it is the one that has to fail.
bool fails(const char* op) {
    auto it = g_fail.find(op);
    if (it == g_fail.end() || --it->second > 0) return false;
    g_fail.erase(it);
    return true;
}

bool pinned(const void* p) {
    auto it = g_pinned.upper_bound((uintptr_t)p);
    if (it == g_pinned.begin()) return false;
    --it;
    return (uintptr_t)p < it->first + it->second;
}

void* room(size_t n) {
    void* p = nullptr;
    return posix_memalign(&p, 512, n < 512 ? 512 : n) == 0 ? p : nullptr;
}

cudaError_t launch(const void* f, cudaStream_t s) {
    if (fails("launch")) return cudaErrorLaunchFailure;
    note(s == g_begun && s ? "captured %p %s" : "launch %p %s", (void*)s, kernels().count(f) ? kernels()[f].c_str() : "?");
    return cudaSuccess;
}

bool capturing(cudaStream_t s) { return g_any_capture && s == g_capturing; }

CUresult encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
    std::memset(m, 0, sizeof *m);
    return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- for the tests ----
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_fail(const char* op, int nth) { g_fail[op] = nth; }
void fake_pin(const void* p, size_t n) { g_pinned[(uintptr_t)p] = n; }
void fake_capturing(cudaStream_t s, int on) {
    g_capturing = s;
    g_any_capture = on;
}

// ---- what compiled kernels register ----
void** __cudaRegisterFatBinary(void*) { return (void**)room(8); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    kernels()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
    g_config = {g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = g_config.grid;
    *b = g_config.block;
    *smem = g_config.smem;
    *(cudaStream_t*)s = g_config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) {
    return launch((const void*)k, s);
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) { return launch(f, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->stream); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}

// ---- device ----
cudaError_t cudaGetDeviceCount(int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    std::memset(p, 0, sizeof *p);
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    note("device_sync %s", "-");
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "an error of the fake runtime"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *f = (void*)encode;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = room(1 << 20);
    return cudaSuccess;
}

// ---- memory (never reused, so that an address names one buffer) ----
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = room(n);
    note("malloc - %p %zu", *p, n);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    note("free - %p", p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    *p = room(n);
    fake_pin(*p, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    g_pinned.erase((uintptr_t)p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    a->type = pinned(p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    a->devicePointer = pinned(p) ? const_cast<void*>(p) : nullptr;
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
    std::memset(p, v, n);
    note("memset legacy %p %zu", p, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    std::memset(p, v, n);
    note("memset %p %p %zu", (void*)s, p, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) {
    if (fails("copy")) return cudaErrorInvalidValue;
    note("copy %p %p %p %zu", (void*)s, d, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* src, size_t, size_t, size_t h, cudaMemcpyKind,
                              cudaStream_t s) {
    if (fails("copy")) return cudaErrorInvalidValue;
    note("copy %p %p %p %zu", (void*)s, d, src, dp * h);
    return cudaSuccess;
}

// ---- streams and events ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)(0x10000 + 16 * g_next++);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    note("stream_sync %p", (void*)s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    note("wait %p %p", (void*)s, (void*)e);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = capturing(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    g_begun = s;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    g_begun = nullptr;
    *g = (cudaGraph_t)g_next++;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = (cudaGraphExec_t)g_next++;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
    if (fails("launch")) return cudaErrorLaunchFailure;
    if (capturing(s)) return cudaErrorStreamCaptureUnsupported;
    note("launch %p graph", (void*)s);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)(0x20000000 + 16 * g_next++);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    note("record %p %p", (void*)s, (void*)e);
    return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    if (g_any_capture) return cudaErrorStreamCaptureUnsupported;
    note("event_sync - %p", (void*)e);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}

}  // extern "C"
