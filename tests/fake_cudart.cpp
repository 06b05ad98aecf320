// A CUDA runtime without a device, for tests of the library's host code on the
// CPU: linked with the library's own objects in place of the CUDA runtime.
// Device memory is host memory, copies and fills happen at once, a kernel
// launch is checked against its shared-memory limit, recorded and does
// nothing.  Every device operation is one line of a log (operation, stream and
// what it touches); a test can make an allocation fail and can have itself
// called back inside an operation.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <utility>
#include <vector>

namespace {

typedef void (*Hook)(const char *what, void *ptr, size_t n);

struct Launch {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};

struct State {
    std::recursive_mutex mu;
    std::ostringstream log;
    std::map<const void *, std::string> kernels;        // host function -> name
    std::map<const void *, int> smem_limit;             // as last set
    std::map<const void *, size_t> symbols;             // host variable -> bytes
    std::map<char *, size_t> live;                      // device allocations
    std::vector<std::pair<std::string, int>> watched;   // kernel name part, argument index
    std::string text;
    int fail_in = 0;                                    // 1: the next allocation fails
    Hook hook = nullptr;
};
State &st() {
    static State *s = new State;    // objects register with it before main and release it at exit
    return *s;
}
thread_local Launch g_pushed;
thread_local cudaError_t g_last = cudaSuccess;

void note(const char *what, cudaStream_t s, const void *p, size_t n) {
    Hook hook;
    {
        std::lock_guard<std::recursive_mutex> l(st().mu);
        st().log << what << ' ' << (size_t)s << ' ' << (size_t)p << ' ' << n << '\n';
        hook = st().hook;
    }
    if (hook) hook(what, const_cast<void *>(p), n);
}

cudaError_t launch(const void *fn, dim3 grid, size_t smem, cudaStream_t s, void **args) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    const std::string &name = st().kernels[fn];
    const auto lim = st().smem_limit.find(fn);
    if (smem > 48 * 1024 && (lim == st().smem_limit.end() || smem > (size_t)lim->second))
        return g_last = cudaErrorInvalidValue;
    st().log << "launch " << (size_t)s << ' ' << name << " grid=" << grid.x << ',' << grid.y << ',' << grid.z;
    for (const auto &w : st().watched)
        if (name.find(w.first) != std::string::npos) st().log << " arg=" << *(size_t *)args[w.second];
    st().log << '\n';
    return cudaSuccess;
}

CUresult encode_tiled(CUtensorMap *m, CUtensorMapDataType, cuuint32_t, void *base, const cuuint64_t *,
                      const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    memset(m, 0, sizeof(*m));
    memcpy(m, &base, sizeof(base));
    return base ? CUDA_SUCCESS : CUDA_ERROR_INVALID_VALUE;
}

}  // namespace

extern "C" {

// ---- control by the test
void fake_reset(void) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    st().log.str("");
    st().watched.clear();
    st().fail_in = 0;
    st().hook = nullptr;
}
const char *fake_log(void) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    st().text = st().log.str();
    return st().text.c_str();
}
void fake_watch(const char *part, int arg) { st().watched.push_back({part, arg}); }
void fake_fail_malloc(int n) { st().fail_in = n; }
void fake_hook(Hook h) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    st().hook = h;
}
size_t fake_live(void) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    return st().live.size();
}

// ---- registration and launches of compiled kernels
void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *,
                            dim3 *, int *) {
    st().kernels[host] = name;
}
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t size, int, int) {
    st().symbols[host] = size;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *s) {
    g_pushed = {g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = g_pushed.grid;
    *b = g_pushed.block;
    *smem = g_pushed.smem;
    *(cudaStream_t *)s = g_pushed.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **args, size_t smem, cudaStream_t s) {
    return launch((const void *)k, grid, smem, s, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
    return launch(fn, c->gridDim, c->dynamicSmemBytes, c->stream, args);
}
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        std::lock_guard<std::recursive_mutex> l(st().mu);
        st().smem_limit[fn] = v;
    }
    note("attribute", nullptr, fn, (size_t)v);
    return cudaSuccess;
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    *p = nullptr;
    if (st().fail_in > 0 && --st().fail_in == 0) return cudaErrorMemoryAllocation;
    *p = aligned_alloc(256, (n + 255) / 256 * 256);
    memset(*p, 0, n);
    st().live[(char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    if (p && !st().live.erase((char *)p)) return cudaErrorInvalidValue;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) {
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) {
    memset(p, v, n);
    note("memset", nullptr, p, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
    memset(p, v, n);
    note("memset", s, p, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *src, size_t n, cudaMemcpyKind, cudaStream_t s) {
    memcpy(d, src, n);
    note("memcpy", s, src, n);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    std::lock_guard<std::recursive_mutex> l(st().mu);
    memset(a, 0, sizeof(*a));
    auto it = st().live.upper_bound((char *)p);
    const bool dev = it != st().live.begin() && (--it, (char *)p < it->first + it->second);
    a->type = dev ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol) {
    *p = const_cast<void *>(symbol);        // the host's shadow of the variable
    return st().symbols.count(symbol) ? cudaSuccess : cudaErrorInvalidSymbol;
}

// ---- device, streams, events
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    note("sync", s, nullptr, 0);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = (cudaEvent_t)malloc(1);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    *fn = (void *)encode_tiled;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

}  // extern "C"
