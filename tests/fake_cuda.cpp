// The CUDA runtime calls that csrc/api.cu makes, on a CPU (the kernel launchers are in
// fake_launchers.cu).  Device memory is the heap's; everything enqueued on a stream waits
// in one queue until something synchronises, as late as the runtime allows, so that host
// memory rewritten before its copy has run shows; an allocation can be made to fail.
#include "fake_cuda.h"

#include <cstdlib>
#include <map>
#include <cstring>
#include <set>
#include <vector>

static std::vector<Op> g_queue;
static std::vector<Op>* g_capture = nullptr;
static cudaStream_t g_capture_stream = nullptr;
static std::set<const void*> g_fresh;
static std::map<const void*, size_t> g_size;        // device blocks
static long g_pinned = 0;            // pinned blocks
static long g_allocs = 0, g_fail_at = -1, g_execs = 0;
static cudaError_t g_last = cudaSuccess;

void fake_push(cudaStream_t s, Op op)
{
    if (g_capture && s == g_capture_stream) g_capture->push_back(std::move(op));
    else g_queue.push_back(std::move(op));
}

static void drain()
{
    std::vector<Op> q;
    q.swap(g_queue);
    for (auto& op : q) op();
}

size_t fake_size(const void* p)
{
    const auto i = g_size.find(p);
    return i == g_size.end() ? 0 : i->second;
}

static cudaError_t alloc(void** p, size_t n, bool device)
{
    *p = nullptr;
    if (g_allocs++ == g_fail_at) return g_last = cudaErrorMemoryAllocation;
    *p = calloc(n ? n : 1, 1);
    if (device) g_fresh.insert(*p), g_size[*p] = n;
    return cudaSuccess;
}

extern "C" {

void fake_fail_at(long n) { g_allocs = 0, g_fail_at = n; }      // the n-th allocation from now fails (-1: none)
long fake_allocs() { return g_allocs; }
void fake_drain() { drain(); }
long fake_graphs() { return g_execs; }
long fake_pinned() { return g_pinned; }

// ---- the runtime
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { drain(); return cudaSuccess; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n, true); }
cudaError_t cudaMallocHost(void** p, size_t n)
{
    const cudaError_t e = alloc(p, n, false);
    g_pinned += e == cudaSuccess;
    return e;
}
cudaError_t cudaFree(void* p) { drain(); g_fresh.erase(p); g_size.erase(p); free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { drain(); free(p); --g_pinned; return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n)
{
    drain();
    if (g_fresh.erase(p) && v == 0) return cudaSuccess;             // calloc's zeros, untouched
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s)
{
    fake_push(s, [=] { memset(p, v, n); });
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { drain(); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2D(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind)
{
    drain();
    for (size_t i = 0; i < h; ++i) memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    fake_push(st, [=] { memcpy(d, s, n); });
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*)
{
    memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { drain(); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode)
{
    g_capture = new std::vector<Op>;
    g_capture_stream = s;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g)
{
    *g = (cudaGraph_t)g_capture;
    g_capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long)
{
    *e = (cudaGraphExec_t) new std::vector<Op>(*(std::vector<Op>*)g);
    ++g_execs;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (std::vector<Op>*)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete (std::vector<Op>*)e; --g_execs; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s)
{
    for (const Op& op : *(std::vector<Op>*)e) fake_push(s, op);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { drain(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }

}  // extern "C"
