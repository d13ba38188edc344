// A CUDA runtime without a GPU, linked with the library's objects for tests of its host code: device memory is
// host memory up to a settable budget, kernels do nothing, copies are made and recorded, and pointers can be
// declared to live on another device.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Copy {
    const void *dst, *src;
    size_t bytes;
};
std::map<char *, size_t> g_live;
std::vector<Copy> g_copies;
std::map<const void *, std::string> g_names;
std::vector<std::string> g_launches;
size_t g_budget = ~(size_t)0, g_used = 0;
unsigned long g_refused = 0;
std::vector<std::pair<std::string, float>> g_times;
const char *g_foreign = nullptr;
size_t g_foreign_bytes = 0;

const char *live_block(const void *p) {
    auto it = g_live.upper_bound((char *)p);
    if (it == g_live.begin()) return nullptr;
    --it;
    return (char *)p < it->first + it->second ? it->first : nullptr;
}
cudaError_t launched(const void *f) {
    g_launches.push_back(g_names[f]);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- the tests' side ----
void fake_budget(size_t bytes) { g_budget = bytes; }
size_t fake_used() { return g_used; }
unsigned long fake_refused() { return g_refused; }
void fake_foreign(const void *p, size_t bytes) { g_foreign = (const char *)p, g_foreign_bytes = bytes; }
// the time of every launch whose kernel's (mangled) name contains `part`; 1 ms for the others
void fake_time(const char *part, float ms) { g_times.push_back({part, ms}); }
void fake_clear_times() { g_times.clear(); }
void fake_clear() { g_copies.clear(), g_launches.clear(); }
int fake_copied(const void *p, int as_source) {
    for (const Copy &c : g_copies)
        if (p == (as_source ? c.src : c.dst)) return 1;
    return 0;
}
int fake_launched(const char *part) {
    int n = 0;
    for (const std::string &s : g_launches) n += s.find(part) != std::string::npos;
    return n;
}

// ---- the library's side ----
cudaError_t cudaMalloc(void **p, size_t n) {
    if (n > g_budget || g_used > g_budget - n) {
        g_refused++;
        return cudaErrorMemoryAllocation;
    }
    char *q = (char *)aligned_alloc(256, (n + 255) / 256 * 256);
    g_live[q] = n;
    g_used += n;
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    auto it = g_live.find((char *)p);
    if (it == g_live.end()) return cudaSuccess;
    g_used -= it->second;
    g_live.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    g_copies.push_back({d, s, n});
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void *d, int v, size_t n) {
    if (n < (size_t)64 << 20) memset(d, v, n);  // not the tuner's flush of a cache that is not there
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof(*a));
    const bool foreign = g_foreign && (const char *)p >= g_foreign && (const char *)p < g_foreign + g_foreign_bytes;
    a->type = foreign || live_block(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    a->device = foreign ? 1 : 0;
    a->devicePointer = (void *)p;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int *n) { return *n = 2, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    memset(p, 0, sizeof(*p));
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 0, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { return *n = 1, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    return *n = 1, cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    for (auto &t : g_times)
        if (!g_launches.empty() && g_launches.back().find(t.first) != std::string::npos) *ms = t.second;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    return *s = cudaStreamCaptureStatusNone, cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "error of the fake runtime"; }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launched(f); }
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launched(f); }
cudaError_t __cudaLaunchKernel(cudaKernel_t f, dim3, dim3, void **, size_t, cudaStream_t) { return launched(f); }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { return *k = (cudaKernel_t)f, cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { return (void **)&g_used; }
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) {
    g_names[host] = name;
}
int fake_nothing() { return 0; }
}

// what the tests do not reach
#define NOTHING(f) asm(".globl " #f "\n.set " #f ", fake_nothing\n")
NOTHING(__cudaRegisterFatBinaryEnd); NOTHING(__cudaRegisterVar); NOTHING(__cudaUnregisterFatBinary);
NOTHING(cudaCtxResetPersistingL2Cache); NOTHING(cudaDeviceGetLimit); NOTHING(cudaDeviceSetLimit);
NOTHING(cudaEventCreate); NOTHING(cudaEventDestroy); NOTHING(cudaEventRecord); NOTHING(cudaEventSynchronize);
NOTHING(cudaFuncSetAttribute); NOTHING(cudaGetLastError); NOTHING(cudaGetSymbolAddress); NOTHING(cudaGraphAddNode);
NOTHING(cudaGraphConditionalHandleCreate); NOTHING(cudaGraphCreate); NOTHING(cudaGraphDestroy);
NOTHING(cudaGraphExecDestroy); NOTHING(cudaGraphInstantiate); NOTHING(cudaGraphLaunch); NOTHING(cudaMemcpy2DAsync);
NOTHING(cudaSetDevice); NOTHING(cudaStreamBeginCaptureToGraph); NOTHING(cudaStreamCreateWithFlags);
NOTHING(cudaStreamDestroy); NOTHING(cudaStreamEndCapture); NOTHING(cudaStreamGetCaptureInfo);
NOTHING(cudaStreamSetAttribute); NOTHING(cudaStreamSynchronize); NOTHING(cudaStreamUpdateCaptureDependencies);
NOTHING(cudaStreamWaitEvent);
