// A stand-in for the CUDA runtime, for tests of libgear's host code on machines without a GPU (tests/test_host_paths.py): nothing
// runs, every call is written down, and a chosen call can be made to fail.  It follows which work the host knows to be finished:
// every stream carries a clock per stream, which events take along and waits merge, so that fake_unfinished() can say whether a
// call left work behind that its caller cannot wait for.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <map>
#include <new>
#include <set>
#include <string>
#include <vector>

namespace {

long g_news = 0, g_no_memory_at = -1;                // allocations of the library; which one fails
bool g_own = false;                                  // the stand-in's own allocations do not count
struct Own { bool before = g_own; Own() { g_own = true; } ~Own() { g_own = before; } };

typedef std::map<void*, long> Clock;                 // stream -> how much of its work
std::map<void*, Clock> g_stream;
std::map<void*, Clock> g_event;
Clock g_done;                                        // what the host has waited for
std::set<void*> g_capturing, g_captured_events;      // streams of a capture; events recorded in one
void* g_capture_origin = nullptr;
std::vector<std::string> g_log;
std::map<const void*, std::string> g_kernel;
long g_calls = 0, g_fail_at = -1, g_handles = 0, g_live = 0;
int g_device = 0;
std::map<std::pair<int, const void*>, int> g_smem;   // dynamic shared memory that a kernel has been allowed on a device
int g_nodes[4096];
int g_n_nodes = 0;

void note(const char* what, void* stream, const char* detail = "") {
    Own own;
    char line[512];
    snprintf(line, sizeof(line), "%s %llx %s", what, (unsigned long long)stream, detail);
    g_log.push_back(line);
}
// A call that can be made to fail.  Work on a stream that is being captured becomes a node of the graph.
cudaError_t work(const char* what, void* stream, const char* detail = "") {
    Own own;
    if (++g_calls == g_fail_at) { note("FAIL", stream, what); return cudaErrorMemoryAllocation; }
    if (g_capturing.count(stream)) { ++g_n_nodes; note("node", stream, detail[0] ? detail : what); }
    else { ++g_stream[stream][stream]; note(what, stream, detail); }
    return cudaSuccess;
}
void merge(Clock& to, const Clock& from) {
    for (const auto& c : from) if (to[c.first] < c.second) to[c.first] = c.second;
}
template <typename T> T handle() { ++g_live; return reinterpret_cast<T>((size_t)(0x10000 + 16 * ++g_handles)); }
CUresult encode_tiled(...) { return CUDA_SUCCESS; }

}  // namespace

// (the library is linked so that its allocations come here)
void* operator new(size_t n) {
    if (!g_own && ++g_news == g_no_memory_at) throw std::bad_alloc();
    void* p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

extern "C" {

// ---- what the tests ask
void fake_reset() { g_stream.clear(); g_event.clear(); g_done.clear(); g_capturing.clear(); g_captured_events.clear(); g_log.clear(); g_calls = 0; g_fail_at = -1; }
void fake_fail_at(long k) { g_calls = 0; g_fail_at = k; }        // the k-th call from now (1, 2, ...) fails; -1: none
long fake_calls() { return g_calls; }
void fake_no_memory_at(long k) { g_news = 0; g_no_memory_at = k; }         // the k-th allocation from now fails; -1: none
long fake_news() { return g_news; }
long fake_live() { return g_live; }                              // streams, events, graphs and pinned blocks not given back
void fake_user_capture(void* stream, int on) { if (on) g_capturing.insert(stream); else g_capturing.clear(); }
// streams with work that the host has not waited for
int fake_unfinished() {
    int n = 0;
    for (const auto& s : g_stream) {
        const auto own = s.second.find(s.first);
        if (own != s.second.end() && own->second > g_done[s.first]) ++n;
    }
    return n;
}
void fake_device(int d) { g_device = d; }
long fake_log(char* out, long cap) {
    std::string all;
    for (const auto& l : g_log) all += l + "\n";
    g_log.clear();
    if ((long)all.size() + 1 > cap) return -1;
    memcpy(out, all.c_str(), all.size() + 1);
    return (long)all.size();
}

// ---- the runtime
void** __cudaRegisterFatBinary(void*) { static void* p; return &p; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { g_kernel[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }

cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int bytes) { Own own;
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = bytes;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** p, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *p = reinterpret_cast<void*>(&encode_tiled);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = reinterpret_cast<void*>(0x1000); return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }

cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) { Own own; return work("launch", s, g_kernel[f].c_str()); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { Own own;
    if (c->dynamicSmemBytes > 48 * 1024 && (int)c->dynamicSmemBytes > g_smem[{g_device, f}]) return cudaErrorInvalidValue;
    if (c->gridDim.x == 0 || c->gridDim.y > 65535 || c->gridDim.z > 65535) return cudaErrorInvalidConfiguration;
    return work("launch", c->stream, g_kernel[f].c_str());
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t s) { Own own; return work("copy", s); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) { Own own; return work("memset", s); }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); ++g_live; note("pinned", nullptr); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); --g_live; return cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { --g_live; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { Own own;
    if (g_capturing.count(s)) return cudaErrorStreamCaptureUnsupported;
    merge(g_done, g_stream[s]);
    note("sync", s);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { --g_live; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { Own own;
    if (++g_calls == g_fail_at) { note("FAIL", s, "record"); return cudaErrorMemoryAllocation; }
    if (g_capturing.count(s)) g_captured_events.insert(e); else { g_captured_events.erase(e); g_event[e] = g_stream[s]; }
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { Own own;
    if (++g_calls == g_fail_at) { note("FAIL", nullptr, "event sync"); return cudaErrorMemoryAllocation; }
    if (g_captured_events.count(e)) return cudaErrorCapturedEvent;
    merge(g_done, g_event[e]);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { Own own;
    if (++g_calls == g_fail_at) { note("FAIL", s, "wait"); return cudaErrorMemoryAllocation; }
    if (g_captured_events.count(e)) g_capturing.insert(s); else merge(g_stream[s], g_event[e]);
    return cudaSuccess;
}

cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) { Own own;
    *st = g_capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { Own own; g_capturing.insert(s); g_capture_origin = s; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { Own own; g_capturing.clear(); g_captured_events.clear(); *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo_v3(cudaStream_t, cudaStreamCaptureStatus* st, unsigned long long*, cudaGraph_t*, const cudaGraphNode_t** deps,
                                        const cudaGraphEdgeData** edges, size_t* n) {
    static cudaGraphNode_t last;
    last = reinterpret_cast<cudaGraphNode_t>(&g_nodes[g_n_nodes % 4096]);
    *st = cudaStreamCaptureStatusActive; *deps = &last; *edges = nullptr; *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { Own own;
    if (++g_calls == g_fail_at) { note("FAIL", nullptr, "instantiate"); return cudaErrorMemoryAllocation; }
    *x = handle<cudaGraphExec_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { Own own; return work("graph", s); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { --g_live; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { --g_live; return cudaSuccess; }
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, const cudaKernelNodeParams* p) { Own own;
    if (++g_calls == g_fail_at) { note("FAIL", nullptr, "node"); return cudaErrorMemoryAllocation; }
    note("update", nullptr, g_kernel[p->func].c_str());
    return cudaSuccess;
}
cudaError_t cudaGraphExecMemsetNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, const cudaMemsetParams*) { return cudaSuccess; }
cudaError_t cudaGraphExecMemcpyNodeSetParams1D(cudaGraphExec_t, cudaGraphNode_t, void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }

}  // extern "C"
