// A stand-in for the CUDA runtime on the host's memory, for tests of the library's host logic on a
// machine without a GPU: device memory is malloc'ed, copies happen at once, kernels do nothing, and
// every copy, memset, launch, wait and attribute is written to a log.  Time is counted, not measured:
// a launch advances a clock by the cost that host_cuda_cost gave its kernel.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

namespace {

struct State {
    std::recursive_mutex m;
    std::map<const void *, std::string> names;
    std::string log;
    std::vector<std::pair<std::string, double>> costs;
    double clock = 0.0;
    int device = 0;
    bool capturing = false;
    dim3 grid, block;
    size_t smem = 0;
    void *stream = nullptr;
    cudaError_t last = cudaSuccess;
};
State &st() {
    static State s;
    return s;
}
void note(const char *what, const std::string &name, const void *stream, size_t bytes) {
    std::lock_guard<std::recursive_mutex> lk(st().m);
    char buf[96];
    std::snprintf(buf, sizeof(buf), " %llx %zu\n", (unsigned long long)(uintptr_t)stream, bytes);
    st().log += std::string(what) + " " + name + buf;
}
cudaError_t launched(const void *f, const void *stream) {
    std::lock_guard<std::recursive_mutex> lk(st().m);
    const auto it = st().names.find(f);
    const std::string name = it == st().names.end() ? "?" : it->second;
    double c = 0.0;
    for (const auto &k : st().costs)
        if (name.find(k.first) != std::string::npos) c = k.second;
    st().clock += c;
    note("launch", name, stream, 0);
    return cudaSuccess;
}
const char *kind_name(cudaMemcpyKind k) { return k == cudaMemcpyHostToDevice ? "h2d" : (k == cudaMemcpyDeviceToHost ? "d2h" : "d2d"); }

}  // namespace

extern "C" {

// ---------------------------------------------------------------- control
void host_cuda_reset() { st().log.clear(); }
const char *host_cuda_log() { return st().log.c_str(); }
void host_cuda_cost(const char *part, double ms) { st().costs.push_back({part, ms}); }
void host_cuda_clear_costs() { st().costs.clear(); }
void host_cuda_device(int d) { st().device = d; }
void host_cuda_capture(int on) { st().capturing = on != 0; }

// ---------------------------------------------------------------- registration and launches
void **__cudaRegisterFatBinary(void *) {
    static void *h = nullptr;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    st().names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *s) {
    st().grid = g, st().block = b, st().smem = smem, st().stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = st().grid, *b = st().block, *smem = st().smem, *(void **)s = st().stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t s) { return launched((const void *)k, s); }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t s) { return launched(f, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return launched(f, c->stream); }

// ---------------------------------------------------------------- devices and kernels
cudaError_t cudaGetDevice(int *d) {
    *d = st().device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : (a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 0);
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    std::memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int) {
    const auto it = st().names.find(f);
    note("attribute", it == st().names.end() ? "?" : it->second, nullptr, (size_t)st().device);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    *p = nullptr;
    *q = cudaDriverEntryPointSymbolNotFound;
    return cudaErrorNotSupported;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    *p = nullptr;
    return cudaErrorNotSupported;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = st().last;
    st().last = cudaSuccess;
    return e;
}

// ---------------------------------------------------------------- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    if (st().capturing) {
        note("refused", "cudaMalloc", nullptr, n);
        return st().last = cudaErrorStreamCaptureUnsupported;
    }
    note("malloc", "-", nullptr, n);
    *p = std::calloc(n ? n : 1, 1);
    return *p ? cudaSuccess : (st().last = cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = std::calloc(n ? n : 1, 1);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
    note("memcpy", kind_name(k), nullptr, n);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t q) {
    note("memcpyAsync", kind_name(k), q, n);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    note("memset", "-", nullptr, n);
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t q) {
    note("memsetAsync", "-", q, n);
    std::memset(d, v, n);
    return cudaSuccess;
}

// ---------------------------------------------------------------- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    static uintptr_t next = 0x1000;
    *s = (cudaStream_t)(next += 0x10);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    note("synchronize", "-", s, 0);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = st().capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = (cudaGraph_t)0x1;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
    *x = (cudaGraphExec_t)0x1;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = (cudaEvent_t) new double(0.0);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete (double *)e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    *(double *)e = st().clock;
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
    *ms = (float)(*(double *)b - *(double *)a);
    return cudaSuccess;
}

}  // extern "C"
