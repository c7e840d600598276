// A CUDA runtime for host-side tests on the CPU: device memory is host memory, kernels do
// not run, and every launch is noted with its stream.  Streams and events carry vector
// clocks, so that a test can ask which launches a stream is ordered after.  Named calls can
// be made to fail.  Linked with the library's objects in place of the CUDA runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

typedef std::map<const void *, long> Clock;  // stream -> launches on it

struct Launch {
    std::string kernel;
    const void *stream;
    long seq;
};

std::map<const void *, Clock> g_stream;  // what each stream's next operation is ordered after
std::map<const void *, Clock> g_event;
std::map<const void *, long> g_count;
Clock g_host;  // what the host has waited for
std::vector<Launch> g_launches;
std::map<const void *, std::string> g_names;
std::map<char *, size_t> g_mem;
size_t g_live, g_peak, g_total = (size_t)256 << 30;
cudaError_t g_last = cudaSuccess;
int g_sms = 152, g_streams, g_events;
struct {
    std::string call;
    long first = -1, n = 0, seen = 0;
} g_fail;
struct {
    dim3 grid, block;
    size_t smem;
    void *stream;
} g_config;

void merge(Clock &a, const Clock &b) {
    for (const auto &kv : b)
        if (a[kv.first] < kv.second) a[kv.first] = kv.second;
}

cudaError_t err(cudaError_t e) {
    if (e != cudaSuccess) g_last = e;
    return e;
}

// Whether this call of `name` is one that was asked to fail.
bool fails(const char *name) {
    if (g_fail.call != name) return false;
    const long i = g_fail.seen++;
    return i >= g_fail.first && i < g_fail.first + g_fail.n;
}

void host_waits(const void *stream) {
    merge(g_host, g_stream[stream]);
}

}  // namespace

extern "C" {

// ---- what the tests ask
void fake_sms(int n) { g_sms = n; }
// Calls number first .. first + n - 1 of `call` from now on fail.
void fake_fail(const char *call, long first, long n) {
    g_fail.call = call ? call : "";
    g_fail.first = first;
    g_fail.n = n;
    g_fail.seen = 0;
}
long fake_calls() { return g_fail.seen; }
long fake_launches() { return (long)g_launches.size(); }
const char *fake_kernel(long i) { return g_launches[(size_t)i].kernel.c_str(); }
// Whether everything enqueued on `stream` from now on runs after launch i.
int fake_ordered(void *stream, long i) {
    const Launch &l = g_launches[(size_t)i];
    return g_stream[stream][l.stream] >= l.seq || g_host[l.stream] >= l.seq;
}
size_t fake_live() { return g_live; }
size_t fake_peak() { return g_peak; }
void fake_reset_peak() { g_peak = g_live; }
int fake_streams() { return g_streams; }
int fake_events() { return g_events; }

// ---- kernels
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *stream) {
    g_config.grid = grid;
    g_config.block = block;
    g_config.smem = smem;
    g_config.stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = g_config.grid;
    *block = g_config.block;
    *smem = g_config.smem;
    *(void **)stream = g_config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) {
    *k = (cudaKernel_t)fun;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t s) {
    if (fails("launch")) return err(cudaErrorLaunchOutOfResources);
    const long seq = ++g_count[s];
    g_stream[s][s] = seq;
    g_launches.push_back(Launch{g_names[(const void *)k], s, seq});
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    g_names[fun] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? g_sms : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    memset(p, 0, sizeof(*p));
    p->multiProcessorCount = g_sms;
    return cudaSuccess;
}
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    if (fails("cudaMalloc")) return err(cudaErrorMemoryAllocation);
    char *m = (char *)calloc(n ? n : 1, 1);
    if (!m) return err(cudaErrorMemoryAllocation);
    g_mem[m] = n;
    g_live += n;
    if (g_live > g_peak) g_peak = g_live;
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    auto it = g_mem.find((char *)p);
    if (it != g_mem.end()) {
        g_live -= it->second;
        free(p);
        g_mem.erase(it);
    }
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) {
    *p = calloc(n ? n : 1, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
    if (fails("cudaMemGetInfo")) return err(cudaErrorUnknown);
    *f = g_total - g_live;
    *t = g_total;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof(*a));
    auto it = g_mem.upper_bound((char *)p);
    const bool dev = it != g_mem.begin() && ((--it)->first + it->second > (char *)p);
    a->type = dev ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    a->devicePointer = dev ? (void *)p : nullptr;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (fails("cudaMemcpyAsync")) return err(cudaErrorUnknown);
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    if (fails("cudaMemsetAsync")) return err(cudaErrorUnknown);
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    static char dummy[1 << 16];
    *p = dummy;
    return cudaSuccess;
}

// ---- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    if (fails("cudaStreamCreateWithFlags")) return err(cudaErrorUnknown);
    *s = (cudaStream_t)malloc(1);
    ++g_streams;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    --g_streams;  // the address stays taken: launches are noted by it
    (void)s;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    host_waits(s);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails("cudaStreamWaitEvent")) return err(cudaErrorUnknown);
    merge(g_stream[s], g_event[e]);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    if (fails("cudaEventCreateWithFlags")) return err(cudaErrorUnknown);
    *e = (cudaEvent_t)malloc(1);
    ++g_events;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) {
    --g_events;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails("cudaEventRecord")) return err(cudaErrorUnknown);
    g_event[e] = g_stream[s];
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    merge(g_host, g_event[e]);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}

// ---- graphs: capture is refused, so that every launch is a direct one
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return err(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return err(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) {
    return err(cudaErrorNotSupported);
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return err(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
