// A CUDA runtime without a GPU, for tests of the library's host code (tests/test_host_runtime.py links it with the
// library's objects in place of the real runtime).  Device memory is host memory; kernels do nothing.  Copies
// and sets queue on their stream and run when it is waited for, as with pinned host memory, so that a copy into a
// caller's array that a call leaves behind can be seen.  An allocation can be made to fail, a line solve to
// set its fault word, and a launch that asks for more dynamic shared memory than its kernel's limit is refused,
// as by the real runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <mutex>
#include <set>
#include <string>

struct CUstream_st {
    std::deque<std::function<void()>> ops;
    bool capturing = false;
};
struct CUevent_st {};

namespace {
std::recursive_mutex mu;
std::set<CUstream_st *> streams;
CUstream_st legacy;
std::map<const void *, std::string> names;     // kernels by their host stub
std::map<const void *, size_t> limits, largest, recent;  // dynamic shared memory: the limit set, the largest and the last launch
std::map<const void *, std::pair<void *, size_t>> vars;
thread_local cudaError_t last = cudaSuccess;
int fail_alloc = -1;     // allocations until one fails (-1: none)
int fail_launch = -1;    // launches until one fails (-1: none)
int host_writes = 0;     // queued copies to the host
bool raise_fault = false;
struct Config { dim3 grid, block; size_t smem; cudaStream_t stream; };
thread_local Config config;

cudaError_t set(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
CUstream_st *of(cudaStream_t s) { return s ? s : &legacy; }
void run(CUstream_st *s) {
    while (!s->ops.empty()) {
        auto op = s->ops.front();
        s->ops.pop_front();
        op();
    }
}
void run_all() {
    run(&legacy);
    for (CUstream_st *s : streams) run(s);
}
using Lock = std::lock_guard<std::recursive_mutex>;
}  // namespace

extern "C" {
// ---- the tests' controls ----
void fake_fail_alloc(int k) { Lock l(mu); fail_alloc = k; }
void fake_fail_launch(int k) { Lock l(mu); fail_launch = k; }
void fake_raise_fault(int on) { Lock l(mu); raise_fault = on != 0; }
int fake_host_writes() { Lock l(mu); return host_writes; }
void fake_run_all() { Lock l(mu); run_all(); }
// the dynamic shared memory limit of the kernels whose name contains `part`: the least and, of their launches, the largest
void fake_smem(const char *part, long long *limit, long long *used) {
    Lock l(mu);
    *limit = -1;
    *used = 0;
    for (auto &n : names) {
        if (n.second.find(part) == std::string::npos) continue;
        if (largest.count(n.first) && (long long)largest[n.first] > *used) *used = (long long)largest[n.first];
        if (limits.count(n.first) && (*limit < 0 || (long long)limits[n.first] < *limit)) *limit = (long long)limits[n.first];
    }
}

// the dynamic shared memory of the last launch of the kernel whose name contains `part`
long long fake_last_smem(const char *part) {
    Lock l(mu);
    for (auto &n : names)
        if (n.second.find(part) != std::string::npos && recent.count(n.first)) return (long long)recent[n.first];
    return -1;
}

// ---- the runtime ----
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
    Lock l(mu);
    *p = nullptr;
    if (fail_alloc >= 0 && fail_alloc-- == 0) return set(cudaErrorMemoryAllocation);
    *p = aligned_alloc(256, (n + 255) & ~(size_t)255);
    memset(*p, 0, (n + 255) & ~(size_t)255);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { Lock l(mu); run_all(); free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t st) {
    Lock l(mu);
    if (kind == cudaMemcpyDeviceToHost) {
        ++host_writes;
        of(st)->ops.push_back([=] { memcpy(d, s, n); --host_writes; });
    } else if (kind == cudaMemcpyHostToDevice) {
        std::string staged((const char *)s, n);  // pageable sources are staged at the call
        of(st)->ops.push_back([=] { memcpy(d, staged.data(), n); });
    } else {
        of(st)->ops.push_back([=] { memcpy(d, s, n); });
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { Lock l(mu); run_all(); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { Lock l(mu); run_all(); memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
    Lock l(mu);
    of(st)->ops.push_back([=] { memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { Lock l(mu); streams.insert(*s = new CUstream_st); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { Lock l(mu); run(s); streams.erase(s); delete s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { Lock l(mu); run(of(s)); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { s->capturing = true; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { s->capturing = false; *g = (cudaGraph_t)malloc(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)malloc(1); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { free(x); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = new CUevent_st; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = new CUevent_st; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { Lock l(mu); run_all(); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { Lock l(mu); run_all(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
    memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    Lock l(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limits[f] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *v) {
    Lock l(mu);
    auto &slot = vars[v];
    if (!slot.first) slot.first = calloc(1, slot.second);
    *p = slot.first;
    return cudaSuccess;
}

// ---- what the compiler's host stubs call ----
void **__cudaRegisterFatBinary(void *b) { return (void **)b; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) {
    Lock l(mu);
    names[host] = name;
}
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t size, int, int) { Lock l(mu); vars[host] = {nullptr, size}; }
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) { config = {grid, block, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
    *grid = config.grid;
    *block = config.block;
    *smem = config.smem;
    *(cudaStream_t *)s = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t smem, cudaStream_t s) {
    Lock l(mu);
    if (fail_launch >= 0 && fail_launch-- == 0) return set(cudaErrorLaunchFailure);
    const size_t limit = limits.count(k) ? limits[k] : 48 * 1024;
    if (smem > largest[k]) largest[k] = smem;
    recent[k] = smem;
    if (smem > limit) return set(cudaErrorInvalidValue);
    if (raise_fault && names[k].find("line_solve_factored_kernel") != std::string::npos && !of(s)->capturing) {
        int *fault = *(int **)args[7];  // (descs, groups, ngroups, natural, stage_bytes, stages, q, fault)
        of(s)->ops.push_back([=] { *fault = 1; });
    }
    return cudaSuccess;
}
}  // extern "C"
