// fake_cudart.cpp -- a stand-in for the CUDA runtime, for tests of the host
// code without a GPU: libgpm's objects are linked against it, "device" memory
// is host memory (zeroed), launches are written to a log and do nothing, and
// any call can be made to fail.  It keeps the rules that the host code has to
// keep: a copy from pageable memory may still be in flight when the call
// returns, so a launch on a stream that is not ordered behind it is counted as
// a violation; a launch with more dynamic shared memory than its kernel's
// attribute allows, and the launch of a graph that was never instantiated,
// fail.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

struct CUstream_st {
    bool nonblocking = false, capturing = false;
};
struct CUevent_st {};
struct CUgraph_st {};
struct CUgraphExec_st {};

namespace {

CUstream_st g_legacy;
std::map<void*, size_t> g_mem;                    // device allocations
size_t g_in_use = 0, g_limit = ~size_t(0);
std::set<CUstream_st*> g_in_flight;               // streams with a pageable copy that may not have landed
int g_violations = 0;
std::map<const void*, std::string> g_names;       // kernels by host function
std::map<const void*, int> g_smem;                // their dynamic shared-memory attribute
std::string g_log;
std::map<std::string, int> g_calls;
std::string g_fail_call;
int g_fail_at = 0, g_failed = 0;
cudaError_t g_last = cudaSuccess;
void (*g_hook)() = nullptr;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
std::vector<Config> g_config;

cudaError_t err(cudaError_t e) {
    if (e != cudaSuccess) g_last = e;
    return e;
}

// whether this call is the one that was asked to fail
bool fails(const char* what) {
    const int n = ++g_calls[what];
    if (g_fail_call == "alloc" && (!strcmp(what, "cudaMalloc") || !strcmp(what, "cudaHostAlloc") ||
                                   !strcmp(what, "cudaGraphInstantiate") || !strcmp(what, "cudaStreamBeginCapture"))) {
        if (--g_fail_at == 0) return g_failed = 1;
        return false;
    }
    if (g_fail_call == what && n == g_fail_at) return g_failed = 1;
    return false;
}

CUstream_st* real(cudaStream_t s) {
    return s == nullptr || s == cudaStreamLegacy ? &g_legacy : s;
}

// a launch on s: every pageable copy in flight elsewhere has to be ordered before it
void ordered(cudaStream_t s) {
    CUstream_st* t = real(s);
    for (CUstream_st* c : g_in_flight) {
        const bool implicit = c == t || ((c == &g_legacy || t == &g_legacy) && !c->nonblocking && !t->nonblocking);
        if (!implicit) g_violations++;
    }
}

cudaError_t launch(const void* f, dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    if (fails("cudaLaunchKernel")) return err(cudaErrorLaunchOutOfResources);
    ordered(s);
    char line[64];
    snprintf(line, sizeof line, " %u %u %zu\n", grid.x, block.x, smem);
    g_log += g_names[f] + line;
    if (smem > 48 * 1024 && (int)smem > g_smem[f]) return err(cudaErrorInvalidValue);
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the test's side
void fake_reset() {
    g_limit = ~size_t(0);
    g_in_flight.clear();
    g_violations = 0;
    g_log.clear();
    g_calls.clear();
    g_fail_call.clear();
    g_fail_at = g_failed = 0;
    g_last = cudaSuccess;
    g_hook = nullptr;
}
void fake_fail(const char* call, int at) {
    g_calls.clear();
    g_fail_call = call;
    g_fail_at = at;
    g_failed = 0;
}
int fake_failed() { return g_failed; }
void fake_memory_limit(size_t bytes) { g_limit = bytes; }
size_t fake_memory_in_use() { return g_in_use; }
int fake_calls(const char* call) { return g_calls[call]; }
int fake_violations() { return g_violations; }
const char* fake_log() { return g_log.c_str(); }
void fake_clear_log() { g_log.clear(); }
void fake_on_event_record(void (*f)()) { g_hook = f; }      // called once, at the next cudaEventRecord
void* fake_stream(int nonblocking) {
    auto* s = new CUstream_st;
    s->nonblocking = nonblocking != 0;
    return s;
}

// ---- registration
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_config.push_back({grid, block, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    const Config c = g_config.back();
    g_config.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t*>(s) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t s) {
    return launch((const void*)k, grid, block, smem, s);
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t s) {
    return launch(f, grid, block, smem, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t bytes) {
    if (fails("cudaMalloc") || bytes > g_limit || g_in_use > g_limit - bytes) return err(cudaErrorMemoryAllocation);
    *p = calloc(1, bytes);
    g_mem[*p] = bytes;
    g_in_use += bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    auto it = g_mem.find(p);
    if (it == g_mem.end()) return err(cudaErrorInvalidValue);
    g_in_use -= it->second;
    g_mem.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
    if (fails("cudaHostAlloc")) return err(cudaErrorMemoryAllocation);
    *p = calloc(1, bytes);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) { return cudaHostAlloc(p, bytes, 0); }
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
    memcpy(d, s, n);
    if (kind == cudaMemcpyHostToDevice) g_in_flight.insert(&g_legacy);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t t) {
    if (real(t)->capturing) return cudaSuccess;
    memcpy(d, s, n);
    if (kind == cudaMemcpyHostToDevice) g_in_flight.insert(real(t));
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    memset(d, v, n);
    return cudaSuccess;
}
// (zeros stay unwritten pages: large scratch costs nothing here)
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    if (v || n < (16u << 20)) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static void* scratch = calloc(1, 4 << 20);
    *p = scratch;
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
    *s = static_cast<cudaStream_t>(fake_stream(flags == cudaStreamNonBlocking));
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    g_in_flight.erase(s);
    delete s;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    g_in_flight.erase(real(s));
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    g_in_flight.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    if (fails("cudaStreamBeginCapture")) return err(cudaErrorMemoryAllocation);
    real(s)->capturing = true;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
    real(s)->capturing = false;
    *g = new CUgraph_st;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    if (fails("cudaGraphInstantiate")) return err(cudaErrorMemoryAllocation);
    *e = new CUgraphExec_st;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    delete e;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
    if (!e) return err(cudaErrorInvalidValue);
    ordered(s);
    g_log += "graph\n";
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = new CUevent_st;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) {
    if (g_hook) {
        void (*f)() = g_hook;
        g_hook = nullptr;
        f();
    }
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    if (v > 227 * 1024) return err(cudaErrorInvalidValue);
    g_smem[f] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int threads, size_t smem) {
    const size_t by_smem = (228 * 1024) / (smem + 1024);
    *n = (int)(by_smem < 2048u / threads ? by_smem : 2048u / threads);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem,
                                                                   unsigned) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, threads, smem);
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }

}  // extern "C"
