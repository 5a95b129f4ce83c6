// A CUDA runtime without a device, for tests of the library's host code: two
// "GPUs" whose memory is host memory and whose kernels do nothing.  Every call
// that matters to a test is written to a log (fake_log):
//
//   launch <kernel> dev <current device> stream <stream>
//   malloc dev <current device> <bytes>
//   sync <call>                      a call that waits for the device
//   attr <kernel> <bytes>            a dynamic shared memory limit
//   graph                            a graph launch
//
// Built as libcudart.so.13 with that version on its symbols and put in front of
// the real one (test_host_calls.py).
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::recursive_mutex g_mu;
std::string g_text;
std::map<const void*, std::string> g_name;
std::map<const void*, std::pair<void*, size_t>> g_var;
std::map<long, std::pair<void*, size_t>> g_alloc;    // by number
long g_allocs = 0;
size_t g_limit = SIZE_MAX;              // larger allocations fail
uint32_t* g_count = nullptr;            // the raster count that was read last
thread_local int g_dev = 0;
thread_local cudaError_t g_last = cudaSuccess;
struct Call { dim3 grid, block; size_t smem; cudaStream_t s; };
thread_local Call g_call;

void note(const std::string& line) {
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    g_text += line + "\n";
}

cudaError_t launch(const void* fn, void** args, cudaStream_t s) {
    const std::string name = g_name.count(fn) ? g_name[fn] : "?";
    note("launch " + name + " dev " + std::to_string(g_dev) + " stream " + std::to_string((uintptr_t)s));
    // the one kernel whose result the host code branches on: it reports the
    // number of recorded spikes (above its own limit nothing else); a test
    // sets that of the first list (fake_raster_count)
    if (name.find("k_sort_small") != std::string::npos) {
        g_count = *reinterpret_cast<uint32_t**>(args[1]);
        uint32_t* head = *reinterpret_cast<uint32_t**>(args[2]);
        head[0] = *g_count;
        head[1] = head[2] = 0u;
    }
    return cudaSuccess;
}
}  // namespace

extern "C" {
const char* fake_log() { return g_text.c_str(); }
void fake_clear() { g_text.clear(); }
uint32_t* fake_raster_count() { return g_count; }
// the k-th of the live allocations of n bytes, in the order they were made
void* fake_alloc(size_t n, int k) {
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    for (const auto& a : g_alloc)
        if (a.second.second == n && k-- == 0) return a.second.first;
    return nullptr;
}
void fake_alloc_limit(size_t bytes) { g_limit = bytes; }
void fake_set_device(int d) { g_dev = d; }
int fake_device() { return g_dev; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    g_name[host] = name;
}
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t size, int, int) {
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    g_var[host] = {calloc(1, size), size};
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
    g_call = {g, b, m, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
    *g = g_call.grid;
    *b = g_call.block;
    *m = g_call.smem;
    *static_cast<cudaStream_t*>(s) = g_call.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fn));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t s) {
    return launch(reinterpret_cast<const void*>(k), args, s);
}
cudaError_t cudaLaunchCooperativeKernel(const void* fn, dim3, dim3, void** args, size_t, cudaStream_t s) {
    return launch(fn, args, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
    return launch(fn, args, c->stream);
}

cudaError_t cudaMalloc(void** p, size_t n) {
    note("malloc dev " + std::to_string(g_dev) + " " + std::to_string(n));
    if (n > g_limit) return g_last = cudaErrorMemoryAllocation;
    *p = calloc(1, n ? n : 1);
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    g_alloc[g_allocs++] = {*p, n};
    return *p ? cudaSuccess : (g_last = cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::recursive_mutex> hold(g_mu);
    for (auto a = g_alloc.begin(); a != g_alloc.end(); ++a)
        if (a->second.first == p) {
            g_alloc.erase(a);
            break;
        }
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    note("sync cudaMemcpy");
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)280 << 30; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { *p = g_var[sym].first; return cudaSuccess; }

cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    memset(p, 0, sizeof(*p));
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    p->sharedMemPerBlockOptin = 232448;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) note("attr " + g_name[fn] + " " + std::to_string(v));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 8; return cudaSuccess; }

cudaError_t cudaStreamSynchronize(cudaStream_t) { note("sync cudaStreamSynchronize"); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(0x77); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = reinterpret_cast<cudaGraph_t>(0x88); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = reinterpret_cast<cudaGraphExec_t>(0x99); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { note("graph"); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(0x66); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { note("sync cudaEventSynchronize"); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
}
