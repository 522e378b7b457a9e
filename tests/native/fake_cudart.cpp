// A stand-in for the CUDA runtime, linked with the library's own object files instead of
// libcudart, so that host logic (which kernel a call launches, what happens on a second device or
// when a launch is refused, what a call allocates) is tested without a GPU.  Device memory is
// host memory; kernels do not run; every launch is recorded by name.  Launch rules that the
// library's host code must respect are enforced per device: more than 48 KiB of dynamic shared
// memory needs the kernel's limit raised on that device, and a cooperative launch must fit.
// Test infrastructure only.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

namespace {

std::mutex g_m;
std::map<const void *, std::string> g_names;
std::map<std::pair<int, const void *>, int> g_smem_limit;
std::map<void *, size_t> g_alloc;
std::string g_log;
thread_local int t_device = 0;
thread_local cudaError_t t_last = cudaSuccess;
int g_sms[8] = {152, 152, 152, 152, 152, 152, 152, 152};
int g_coop = 1;              // the device attribute
int g_refuse = 0;            // cooperative launches fail as too large
size_t g_in_use = 0, g_limit = (size_t)-1;
float g_elapsed = 1.0f;
cudaStream_t g_capturing = (cudaStream_t)-1;  // a stream that a test says is being captured
double g_host[4];            // first values of page-locked memory, where residuals are read
struct Config {
    dim3 g, b;
    size_t smem;
    void *s;
};
thread_local std::vector<Config> t_config;

cudaError_t fail(cudaError_t e) {
    t_last = e;
    return e;
}

int fit(const void *f, int threads, size_t smem) {  // resident blocks per SM
    if (smem > 48 * 1024) {
        auto it = g_smem_limit.find({t_device, f});
        if (it == g_smem_limit.end() || (size_t)it->second < smem) return 0;
    }
    const size_t by_smem = 228 * 1024 / (smem + 1024);
    const size_t by_threads = 2048 / (threads > 0 ? threads : 1);
    return (int)(by_smem < by_threads ? by_smem : by_threads);
}

cudaError_t launch(const void *f, dim3 g, dim3 b, size_t smem, bool coop) {
    std::lock_guard<std::mutex> lock(g_m);
    const int per_sm = fit(f, (int)(b.x * b.y * b.z), smem);
    if (per_sm < 1) return fail(cudaErrorInvalidValue);
    if (coop && !g_coop) return fail(cudaErrorNotSupported);
    if (coop && (g_refuse || (long)g.x * g.y * g.z > (long)per_sm * g_sms[t_device]))
        return fail(cudaErrorCooperativeLaunchTooLarge);
    char line[64];
    std::snprintf(line, sizeof line, " %u %d\n", g.x * g.y * g.z, t_device);
    g_log += (coop ? "cooperative " : "plain ") + g_names[f] + line;
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the tests' controls
void fake_reset() {
    std::lock_guard<std::mutex> lock(g_m);
    g_log.clear();
    for (int &s : g_sms) s = 152;
    g_coop = 1, g_refuse = 0, g_limit = (size_t)-1, g_elapsed = 1.0f;
    g_host[0] = g_host[1] = 1.0, g_host[2] = 0.5, g_host[3] = 0.0;  // rho = 1, max |rt| = 0.5, no status
    t_device = 0, t_last = cudaSuccess;
    g_capturing = (cudaStream_t)-1;
}
void fake_clear_log() { std::lock_guard<std::mutex> lock(g_m); g_log.clear(); }
const char *fake_log() { return g_log.c_str(); }  // "kind kernel blocks device" per line
void fake_set_device(int d) { t_device = d; }
void fake_capture(void *stream) { g_capturing = (cudaStream_t)stream; }
void fake_set_sms(int d, int n) { g_sms[d] = n; }
void fake_cooperative(int attribute, int refuse) { g_coop = attribute, g_refuse = refuse; }
void fake_device_reset() {  // of the current device: raised limits are gone
    std::lock_guard<std::mutex> lock(g_m);
    for (auto &e : g_smem_limit)
        if (e.first.first == t_device) e.second = 48 * 1024;
}
void fake_memory_limit(size_t bytes) { g_limit = bytes; }
size_t fake_memory_in_use() { return g_in_use; }

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    std::lock_guard<std::mutex> lock(g_m);
    g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *s) {
    t_config.push_back({g, b, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    const Config c = t_config.back();
    t_config.pop_back();
    *g = c.g, *b = c.b, *smem = c.smem, *(void **)s = c.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **, size_t smem, cudaStream_t) {
    return launch((const void *)k, g, b, smem, false);
}
cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **, size_t smem, cudaStream_t) { return launch(f, g, b, smem, false); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, false);
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 g, dim3 b, void **, size_t smem, cudaStream_t) {
    return launch(f, g, b, smem, true);
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
    std::lock_guard<std::mutex> lock(g_m);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem_limit[{t_device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int threads, size_t smem, unsigned) {
    std::lock_guard<std::mutex> lock(g_m);
    *n = fit(f, threads, smem);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
    *n = g_sms[t_device] / (int)c->attrs[0].val.clusterDim.x;
    return cudaSuccess;
}

// ---- devices, errors
cudaError_t cudaGetDevice(int *d) { *d = t_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? g_sms[d] : a == cudaDevAttrCooperativeLaunch ? g_coop : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = t_last; t_last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long, enum cudaDriverEntryPointQueryResult *r) {
    *p = nullptr;
    if (r) *r = cudaDriverEntryPointSymbolNotFound;
    return cudaErrorNotSupported;
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::mutex> lock(g_m);
    if (g_in_use + n > g_limit) return fail(cudaErrorMemoryAllocation);
    *p = std::calloc(n ? n : 1, 1);
    g_alloc[*p] = n, g_in_use += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::mutex> lock(g_m);
    auto it = g_alloc.find(p);
    if (it != g_alloc.end()) g_in_use -= it->second, g_alloc.erase(it), std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = std::calloc(n ? n : 1, 1);
    if (n == sizeof g_host) std::memcpy(*p, g_host, n);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, enum cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void *d, const void *, size_t n, size_t, enum cudaMemcpyKind) { std::memset(d, 0, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidSymbol; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p) {
    std::lock_guard<std::mutex> lock(g_m);
    auto it = g_alloc.upper_bound((void *)p);
    const bool dev = it != g_alloc.begin() && (--it, (const char *)p < (const char *)it->first + it->second);
    std::memset(a, 0, sizeof *a);
    a->type = dev ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = (cudaGraph_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, enum cudaStreamCaptureStatus *s) {
    *s = st == g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
    std::lock_guard<std::mutex> lock(g_m);
    g_log += "graph - 0 0\n";
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { std::free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = g_elapsed; return cudaSuccess; }

}  // extern "C"
