// A stand-in for the CUDA runtime that runs nothing on a device: memory comes from
// the host, copies and clears are done at once, kernels are left out, and every call
// that matters for order or memory is written down, one line each:
//   malloc <ptr> <bytes> | free <ptr> | sync <stream, or "all"> |
//   memset <stream> <ptr> <bytes> | copy <stream> <kind> <dst> <src> <bytes> |
//   launch <stream> <kernel> <grid> <args as given, only of k_scan_block>
// Streams print as numbers, 0 for the legacy default stream.  Linked with the
// library's own objects in place of libcudart, so that host code runs as built.
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::string log_;
std::map<const void*, std::string> names;
size_t limit = ~(size_t)0, held = 0;
std::map<void*, size_t> blocks;
bool capturing = false;
dim3 cfg_grid, cfg_block;
size_t cfg_smem;
void* cfg_stream;
uintptr_t next_handle = 1000;
cudaGraph_t body;
cudaGraphNode_t node = (cudaGraphNode_t)7;

void say(const char* f, ...)
{
    char b[512];
    va_list a;
    va_start(a, f);
    vsnprintf(b, sizeof b, f, a);
    va_end(a);
    log_ += b;
    log_ += '\n';
}
unsigned long long num(const void* p) { return (unsigned long long)(uintptr_t)p; }
cudaError_t launched(const void* f, dim3 g, void** args, cudaStream_t s)
{
    if (capturing) return cudaSuccess;
    const std::string& n = names[f];
    if (n.find("k_scan_block") != std::string::npos)
        say("launch %llu %s %u %llu %llu %llu %llu", num(s), n.c_str(), g.x, *(unsigned long long*)args[0],
            *(unsigned long long*)args[1], *(unsigned long long*)args[2], *(unsigned long long*)args[3]);
    else
        say("launch %llu %s %u", num(s), n.c_str(), g.x);
    return cudaSuccess;
}
}  // namespace

extern "C" {
const char* rec_log() { return log_.c_str(); }
void rec_clear() { log_.clear(); }
void rec_limit(size_t bytes) { limit = bytes; }
size_t rec_held() { return held; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void* st)
{
    cfg_grid = g; cfg_block = b; cfg_smem = sm; cfg_stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* st)
{
    *g = cfg_grid; *b = cfg_block; *sm = cfg_smem; *(void**)st = cfg_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void** args, size_t, cudaStream_t s)
{
    return launched((const void*)k, g, args, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    return launched(f, c->gridDim, args, c->stream);
}

cudaError_t cudaMalloc(void** p, size_t n)
{
    if (held + n > limit) return cudaErrorMemoryAllocation;
    *p = calloc(1, n);
    blocks[*p] = n;
    held += n;
    say("malloc %llu %zu", num(*p), n);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (!p) return cudaSuccess;
    held -= blocks[p];
    blocks.erase(p);
    free(p);
    say("free %llu", num(p));
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s)
{
    if (capturing) return cudaSuccess;
    memset(p, v, n);
    say("memset %llu %llu %zu", num(s), num(p), n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n, 0); }
cudaError_t cudaMemcpyAsync(void* d, const void* h, size_t n, cudaMemcpyKind k, cudaStream_t s)
{
    memcpy(d, h, n);
    say("copy %llu %d %llu %llu %zu", num(s), (int)k, num(d), num(h), n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* h, size_t n, cudaMemcpyKind k) { return cudaMemcpyAsync(d, h, n, k, 0); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { say("sync %llu", num(s)); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { say("sync all"); return cudaSuccess; }

cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "recorded"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { memset(p, 0, sizeof *p); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)next_handle++; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)next_handle++; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { capturing = true; return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode)
{
    capturing = true;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g)
{
    capturing = false;
    *g = (cudaGraph_t)next_handle++;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* st, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t** d, const cudaGraphEdgeData**, size_t* n)
{
    *st = cudaStreamCaptureStatusActive;
    *d = &node;
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = (cudaGraph_t)next_handle++; return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned)
{
    *h = 1;
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p)
{
    *n = node;
    p->conditional.phGraph_out = &body;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long)
{
    *e = (cudaGraphExec_t)next_handle++;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s)
{
    say("launch %llu graph%llu 0", num(s), num(e));
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
}
