// A CUDA runtime for the library's host code on a machine without a GPU:
// device memory is host memory, kernels are counted by name and not run.
// What the tests set and read: the memory there is, the stream that the caller
// captures, and counts of launches, waits, pinned allocations and of
// calls that a capture forbids.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::map<const void *, std::string> names;
std::map<std::string, long long> launched;
std::map<void *, size_t> live;
bool deny = false;
size_t held = 0, room = ~(size_t)0 >> 1;   // bytes allocated, and what there is
cudaStream_t captured = nullptr;
bool relaxed = false;
long long waits = 0, pinned = 0, forbidden = 0, recorded_copies = 0;

cudaError_t get(void **p, size_t n) {
    if (captured && !relaxed) ++forbidden;
    if (deny || n + held > room) return cudaErrorMemoryAllocation;
    *p = calloc(n ? n : 1, 1);
    live[*p] = n;
    held += n;
    return cudaSuccess;
}
cudaError_t put(void *p) {
    if (captured && !relaxed) ++forbidden;
    if (p && !live.count(p)) abort();
    if (p) held -= live[p];
    live.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t wait(cudaStream_t s) {
    ++waits;
    if (captured && s == captured) ++forbidden;
    return s && s == captured ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t launch(const void *f) {
    launched[names.count(f) ? names[f] : "?"]++;
    return cudaSuccess;
}
long long next_id = 1000;
template <class T>
cudaError_t fresh(T *out) {
    *out = (T)(size_t)next_id++;
    return cudaSuccess;
}
dim3 cfg_g, cfg_b;
size_t cfg_m;
cudaStream_t cfg_s;
}  // namespace

#pragma GCC visibility push(default)
extern "C" {
// memory for `more` bytes beside what is held (< 0: no limit)
void fake_room(long long more) { room = more < 0 ? ~(size_t)0 >> 1 : held + (size_t)more; }
void fake_capture(void *s) { captured = (cudaStream_t)s; }
long long fake_waits() { return waits; }
long long fake_pinned() { return pinned; }
long long fake_forbidden() { return forbidden; }
long long fake_recorded_copies() { return recorded_copies; }
void fake_deny(int on) { deny = on; }   // no memory at all
long long fake_held() { return (long long)held; }
// launches since the last call, of kernels whose (mangled) name holds `part`
long long fake_launches(const char *part) {
    long long n = 0;
    for (auto &x : launched)
        if (x.first.find(part) != std::string::npos) n += x.second;
    launched.clear();
    return n;
}
#pragma GCC visibility pop

void **__cudaRegisterFatBinary(void *) { return (void **)&names; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
    cfg_g = g, cfg_b = b, cfg_m = m, cfg_s = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) {
    *g = cfg_g, *b = cfg_b, *m = cfg_m, *(cudaStream_t *)s = cfg_s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t) { return launch(k); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **) { return launch(f); }
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launch(f); }

cudaError_t cudaMalloc(void **p, size_t n) { return get(p, n); }
cudaError_t cudaFree(void *p) { return put(p); }
cudaError_t cudaMallocHost(void **p, size_t n) {
    if (captured && !relaxed) ++forbidden;
    ++pinned;
    *p = calloc(n ? n : 1, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (st && st == captured) ++recorded_copies;
    else memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return wait(s); }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return fresh(s); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { return fresh(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return fresh(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return fresh(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return wait(nullptr); }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st) {
    *st = s && s == captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m) {
    const bool was = relaxed;
    relaxed = *m == cudaStreamCaptureModeRelaxed;
    *m = was ? cudaStreamCaptureModeRelaxed : cudaStreamCaptureModeGlobal;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return fresh(g); }
cudaError_t cudaGraphGetRootNodes(cudaGraph_t, cudaGraphNode_t *n, size_t *k) {
    *k = 1;
    return fresh(n);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { return fresh(x); }
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, const cudaKernelNodeParams *) {
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
    launched["graph"]++;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidSymbol; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi) {
    *lo = 0, *hi = -5;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
    *n = 76;
    return cudaSuccess;
}
}
