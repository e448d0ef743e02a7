// A CUDA runtime that runs nothing: the library's object files linked against it execute their whole host
// path on the CPU.  Kernel launches are listed (name, grid, block), allocations are addresses that are never
// read, copies to the host give zeros.  What the host path is checked for:
//   order:    every stream carries a vector clock (how many launches, copies and fills of each stream come
//             before what is enqueued on it now), moved on by records, waits and synchronisations; a
//             cudaFreeAsync with work on any stream that is not ordered before it is a bad free
//   failures: the n-th event call (create, record or wait) can be made to fail; launches after it are counted
// Test infrastructure only.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
using Clock = std::map<void*, unsigned long>;          // stream -> operations seen
std::map<void*, Clock> g_view;                         // per stream
std::map<void*, Clock> g_event;
std::map<void*, std::string> g_name;                   // kernel handles
Clock g_host, g_done;                                  // what the host has waited for; what each stream has been given
std::string g_log;
long g_fail_at = -1, g_calls = 0, g_bad_frees = 0, g_late = 0;
bool g_failed = false;
cudaError_t g_last = cudaSuccess;
uintptr_t g_next = 1 << 20;
struct Config { dim3 grid, block; size_t smem; void* stream; } g_cfg;

void join(Clock& a, const Clock& b) {
    for (auto& e : b)
        if (a[e.first] < e.second) a[e.first] = e.second;
}
Clock& view(void* s) {                                 // what is enqueued now on s comes after all of this
    join(g_view[s], g_host);
    return g_view[s];
}
template <class T>
T fresh() { return reinterpret_cast<T>(g_next += 256); }
bool event_call() {                                    // false: this one fails
    if (g_calls++ == g_fail_at) {
        g_failed = true;
        g_last = cudaErrorUnknown;
        return false;
    }
    return true;
}
cudaError_t take(void** p, size_t n) {
    *p = reinterpret_cast<void*>(g_next += 512);
    g_next += (n + 255) & ~(size_t)255;
    return cudaSuccess;
}
cudaError_t work(void* s) {                            // a launch, copy or fill
    view(s)[s] = ++g_done[s];
    return cudaSuccess;
}
cudaError_t copied(void* dst, size_t n, cudaMemcpyKind k) {
    if (k == cudaMemcpyDeviceToHost) memset(dst, 0, n);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- for the tests
void fake_reset(long fail_at) {
    g_fail_at = fail_at;
    g_calls = g_bad_frees = g_late = 0;
    g_failed = false;
    g_log.clear();
}
long fake_event_calls() { return g_calls; }
long fake_bad_frees() { return g_bad_frees; }
long fake_late_launches() { return g_late; }
const char* fake_log() { return g_log.c_str(); }       // "mangled_name grid block" per launch

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_name[const_cast<char*>(host)] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(host));
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
    g_cfg = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = g_cfg.grid;
    *block = g_cfg.block;
    *smem = g_cfg.smem;
    *static_cast<void**>(s) = g_cfg.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t, cudaStream_t s) {
    g_log += g_name[k] + " " + std::to_string(grid.x) + " " + std::to_string(block.x) + "\n";
    if (g_failed) g_late++;
    work(s);
    if (!grid.x || !block.x) return g_last = cudaErrorInvalidConfiguration;
    return cudaSuccess;
}

// ---- devices, streams, events
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { *lo = 0; *hi = -5; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = fresh<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { *s = fresh<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { join(g_host, g_view[s]); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { join(g_host, g_done); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) { *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    if (!event_call()) return cudaErrorUnknown;
    *e = fresh<cudaEvent_t>();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return e ? cudaSuccess : g_last = cudaErrorInvalidResourceHandle; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (!event_call()) return cudaErrorUnknown;
    if (!e) return g_last = cudaErrorInvalidResourceHandle;
    g_event[e] = view(s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (!event_call()) return cudaErrorUnknown;
    if (!e) return g_last = cudaErrorInvalidResourceHandle;
    join(view(s), g_event[e]);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { join(g_host, g_event[e]); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFreeAsync(void*, cudaStream_t s) {
    const Clock& v = view(s);
    for (auto& e : g_done) {
        const auto it = v.find(e.first);
        if (it == v.end() || it->second < e.second) {
            g_bad_frees++;
            break;
        }
    }
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return take(p, 256); }
cudaError_t cudaMemcpy(void* d, const void*, size_t n, cudaMemcpyKind k) { work(nullptr); join(g_host, g_view[nullptr]); return copied(d, n, k); }
cudaError_t cudaMemcpyAsync(void* d, const void*, size_t n, cudaMemcpyKind k, cudaStream_t s) { work(s); return copied(d, n, k); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) { return work(s); }

// ---- graphs (not run here)
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
}
