// A stand-in for the CUDA runtime, linked with the library's own objects, so that the host side (routes, workspaces, error
// paths) runs on a machine without a GPU.  Memory is host memory, kernels do nothing but are recorded; allocations can be
// made to fail, the device's size and the outcome of cooperative launches and graph instantiation are set by the test.
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

namespace {
struct Poke { std::string kernel; int arg, offset, value; };
std::map<const void*, std::string> kernels;
std::map<void*, size_t> blocks;
std::vector<Poke> pokes;
std::string watch_kernel, report;
int fail_at = 0, watch_arg = -1, sms = 152, capturing = 0, instantiate_errors = 0;
long long optin = 232448, room = 1ll << 50, watched = -1, held = 0;
cudaError_t coop = cudaSuccess, last = cudaSuccess;
struct Call { dim3 grid, block; size_t smem; void* st; } pending;

cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t launch(const void* f, void** args) {
    const std::string& n = kernels[f];
    report += n + "\n";
    if (!watch_kernel.empty() && n.find(watch_kernel) != std::string::npos) watched = *(long long*)args[watch_arg];
    for (const Poke& p : pokes)
        if (n.find(p.kernel) != std::string::npos) {
            char* dst = *(char**)args[p.arg];
            if (dst) memcpy(dst + p.offset, &p.value, sizeof p.value);
        }
    return cudaSuccess;
}
}  // namespace

extern "C" {
// controls
void fake_reset() {
    pokes.clear();
    watch_kernel.clear();
    report.clear();
    fail_at = 0; watched = -1; sms = 152; capturing = 0; optin = 232448; room = 1ll << 50; instantiate_errors = 0;
    coop = last = cudaSuccess;
}
void fake_device(int n, long long smem) { sms = n; optin = smem; }
void fake_room(long long bytes) { room = bytes; }            // bytes that further allocations may take
void fake_fail_at(int n) { fail_at = n; }                    // the n-th allocation from here fails (1: the next)
int fake_fail_pending() { return fail_at > 0; }
void fake_capturing(int on) { capturing = on; }
void fake_coop_error(int e) { coop = (cudaError_t)e; }
void fake_instantiate_errors(int n) { instantiate_errors = n; }
void fake_watch(const char* kernel, int arg) { watch_kernel = kernel; watch_arg = arg; watched = -1; }
long long fake_watched() { return watched; }                 // 8 bytes of the watched argument in the last such launch
void fake_poke(const char* kernel, int arg, int offset, int value) { pokes.push_back({kernel, arg, offset, value}); }
long long fake_held() { return held; }
const char* fake_report() { return report.c_str(); }         // names of the kernels launched, one a line
void fake_clear_report() { report.clear(); }

// registration and launches
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    kernels[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) { pending = {g, b, s, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = pending.grid; *b = pending.block; *s = pending.smem;
    *(void**)st = pending.st;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) { return launch(k, args); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t) {
    return coop == cudaSuccess ? launch(f, args) : done(coop);
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
    return done(v > optin ? cudaErrorInvalidValue : cudaSuccess);
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}

// memory
cudaError_t cudaMalloc(void** p, size_t n) {
    const bool fail = fail_at > 0 && --fail_at == 0;
    *p = (long long)n <= room && !fail ? calloc(1, n) : nullptr;
    if (!*p) return done(cudaErrorMemoryAllocation);
    room -= n;
    held += n;
    blocks[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = blocks.find(p);
    if (it != blocks.end()) {
        room += it->second;
        held -= it->second;
        blocks.erase(it);
        free(p);
    }
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
// (large blocks are left alone: no test reads them)
cudaError_t cudaMemset(void* p, int v, size_t n) { if (n <= 1 << 20) memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (n <= 1 << 20) memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return cudaSuccess; }

// device, streams, events
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? (int)optin : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

// graphs
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                          cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)&pending; return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* s, unsigned long long*, cudaGraph_t* g,
                                     const cudaGraphNode_t**, const cudaGraphEdgeData**, size_t*) {
    *s = cudaStreamCaptureStatusActive;
    if (g) *g = (cudaGraph_t)&pending;
    return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t, unsigned) {
    return cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
    *h = 0;
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
    static cudaGraph_t body;
    p->conditional.phGraph_out = &body;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    if (instantiate_errors > 0) {
        instantiate_errors--;
        return done(cudaErrorNotSupported);
    }
    report += "instantiate\n";
    *e = (cudaGraphExec_t)&pending;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { report += "graph\n"; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
