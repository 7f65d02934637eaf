// A CUDA runtime without a GPU, for tests of the library's host side: the library's own objects are linked
// against it.  Device memory is host memory, nothing runs on it, and every launch, event and asynchronous
// copy is written to a log that the test reads, one line each:
//   launch <kernel symbol> <stream> <priority of the stream> <1 with the programmatic attribute>
//   record <event> <stream>      wait <stream> <event>      memset <stream> <bytes>
// fake_refuse(n) makes the n-th launch from now on (0: the next one) return an error once.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

namespace {
struct Stream {
    int id, priority;
};
std::vector<std::string> g_log;
int g_ids = 0, g_refuse = -1, g_streams = 0;
cudaError_t g_last = cudaSuccess;
std::map<const void*, void*>& symbols() {
    static std::map<const void*, void*> m;
    return m;
}
std::map<const void*, std::string>& kernels() {
    static std::map<const void*, std::string> m;
    return m;
}
int sid(cudaStream_t s) { return s ? ((Stream*)s)->id : 0; }
int spri(cudaStream_t s) { return s ? ((Stream*)s)->priority : 0; }
cudaError_t launch(const void* f, cudaStream_t s, bool early) {
    if (g_refuse >= 0 && g_refuse-- == 0) return g_last = cudaErrorLaunchOutOfResources;
    g_log.push_back("launch " + kernels()[f] + " " + std::to_string(sid(s)) + " " + std::to_string(spri(s)) + " " +
                    (early ? "1" : "0"));
    return cudaSuccess;
}
void note(const char* what, int a, long long b) { g_log.push_back(std::string(what) + " " + std::to_string(a) + " " + std::to_string(b)); }
}  // namespace

extern "C" {
void fake_clear() { g_log.clear(); }
int fake_count() { return (int)g_log.size(); }
const char* fake_line(int i) { return g_log[i].c_str(); }
void fake_refuse(int n) { g_refuse = n; }
int fake_streams() { return g_streams; }
void* fake_stream(int priority) { return new Stream{++g_ids, priority}; }

void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) { kernels()[f] = name; }
void __cudaRegisterVar(void**, char* var, char*, const char*, int, size_t size, int, int) { symbols()[var] = calloc(1, size); }
static dim3 g_grid, g_block;
static size_t g_smem;
static cudaStream_t g_stream;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_grid = grid, g_block = block, g_smem = smem, g_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = g_grid, *block = g_block, *smem = g_smem, *(cudaStream_t*)s = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) { return launch((const void*)k, s, false); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    bool early = false;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        early |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
                 c->attrs[i].val.programmaticStreamSerializationAllowed != 0;
    return launch(f, c->stream, early);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) { return launch(f, s, false); }

cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) { return *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    memset(p, 0, sizeof(*p));
    strcpy(p->name, "fake");
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { return *lo = 0, *hi = -5, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { return *n = 4, cudaSuccess; }

// what a test never writes stays untouched pages
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t k = 0; k < h; ++k) memcpy((char*)d + k * dp, (const char*)s + k * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    note("memset", sid(s), (long long)n);
    return cudaMemset(p, v, n);
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { return *p = symbols()[sym], cudaSuccess; }

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int priority) {
    ++g_streams;
    *s = (cudaStream_t)fake_stream(priority);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { return cudaStreamCreateWithPriority(s, f, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    --g_streams;
    delete (Stream*)s;
    return cudaSuccess;
}
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { return *p = spri(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) { return *c = cudaStreamCaptureStatusNone, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return note("wait", sid(s), *(int*)e), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t) new int(++g_ids), cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (int*)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return note("record", *(int*)e, sid(s)), cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }

cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, const cudaKernelNodeParams*) { return *n = nullptr, cudaSuccess; }
cudaError_t cudaGraphAddMemcpyNode1D(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, void*, const void*, size_t, cudaMemcpyKind) { return *n = nullptr, cudaSuccess; }
cudaError_t cudaGraphAddMemsetNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, const cudaMemsetParams*) { return *n = nullptr, cudaSuccess; }
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t, cudaLaunchAttributeID, const cudaLaunchAttributeValue*) { return cudaSuccess; }
}
