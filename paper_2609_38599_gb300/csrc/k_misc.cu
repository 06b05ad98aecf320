// Elementwise and bookkeeping kernels of the refinement path.
#include <condition_variable>
#include <mutex>

#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kStatusWords = 64;       // calls that hold one at a time
__device__ int g_status_words[kStatusWords];

// Which words are taken.  An index is taken on all devices at once.  Never
// destroyed: a call may still run while the process ends.
struct StatusPool {
    std::mutex mu;
    std::condition_variable freed;
    unsigned long long taken = 0;
};
StatusPool &status_pool() {
    static StatusPool *p = new StatusPool;
    return *p;
}
static_assert(kStatusWords == 64, "one bit of `taken` per word");

// Codes and zero points must lie in [0, qmax] (Sec. 3.1: q in B^{d_i};
// integer zero points kept from the host).
__global__ void validate_kernel(const uint8_t *__restrict__ Q, const int32_t *__restrict__ Z,
                                size_t nq, size_t nz, int qmax, int *status) {
    __shared__ int flag;
    if (threadIdx.x == 0) flag = 0;
    __syncthreads();
    int local = 0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += stride)
        if (Q[i] > qmax) local |= ST_BAD_CODE;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nz; i += stride)
        if (Z[i] < 0 || Z[i] > qmax) local |= ST_BAD_ZERO;
    if (local) atomicOr(&flag, local);
    __syncthreads();
    if (threadIdx.x == 0 && flag) atomicOr(status, flag);
}

// The same check for Q 16-byte aligned and nq a multiple of 16: qmax is 2^b - 1,
// so a code is above it iff it has a bit outside qmax; the codes are OR-ed, 64
// per thread and iteration.
__global__ void validate16_kernel(const uint4 *__restrict__ Q16, const int32_t *__restrict__ Z,
                                  size_t nq16, size_t nz, int qmax, int *status) {
    __shared__ int flag;
    if (threadIdx.x == 0) flag = 0;
    __syncthreads();
    int local = 0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t seen = 0;
    size_t i = i0;
    for (; i + 3 * stride < nq16; i += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = Q16[i + k * stride];
#pragma unroll
        for (int k = 0; k < 4; ++k) seen |= (v[k].x | v[k].y) | (v[k].z | v[k].w);
    }
    for (; i < nq16; i += stride) {
        const uint4 v = Q16[i];
        seen |= (v.x | v.y) | (v.z | v.w);
    }
    if (seen & ~(0x01010101u * (uint32_t)qmax)) local |= ST_BAD_CODE;
    for (size_t k = i0; k < nz; k += stride)
        if (Z[k] < 0 || Z[k] > qmax) local |= ST_BAD_ZERO;
    if (local) atomicOr(&flag, local);
    __syncthreads();
    if (threadIdx.x == 0 && flag) atomicOr(status, flag);
}

// r = w - s (q - z), one rounding (fma) per element (Eq. quantized_group),
// and the code plane c = q - z; with rv.r == nullptr only the code plane.
__global__ void residual_kernel(const float *__restrict__ W, const float *__restrict__ S,
                                const uint8_t *__restrict__ Q, const int32_t *__restrict__ Z,
                                ResidualView rv, int p, int g) {
    const int d = rv.d, G = d / g;
    const size_t n = (size_t)p * d;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += stride) {
        const size_t j = idx / d;
        const int grp = (int)(idx - j * d) / g;
        const int ci = (int)Q[idx] - Z[j * G + grp];
        if (rv.r) store_residual(rv, j, (int)(idx - j * d), fmaf(-S[j * G + grp], (float)ci, W[idx]));
        store_code(rv, j, (int)(idx - j * d), ci);
    }
}

// The same, eight entries per thread (one group: g is a multiple of 8; Q 8-byte,
// W 16-byte aligned; 16-byte accesses); FULL with the residual.  Bound by memory:
// 17 us for the code plane of 4096 x 4096 (3 bytes an entry), 48 us with the
// residual (17 bytes); one entry a thread took 83 us with the residual.
template <bool FULL>
__global__ void __launch_bounds__(256) residual8_kernel(const float *__restrict__ W, const float *__restrict__ S,
                                                        const uint8_t *__restrict__ Q,
                                                        const int32_t *__restrict__ Z, ResidualView rv, int p,
                                                        int g) {
    const int d = rv.d, G = d / g;
    const size_t n8 = (size_t)p * d / 8;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i8 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i8 < n8; i8 += stride) {
        const size_t idx = i8 * 8;
        const size_t j = idx / d;
        const int col = (int)(idx - j * d);
        const int z = Z[j * G + col / g];
        const uint2 q8 = *reinterpret_cast<const uint2 *>(Q + idx);
        const uint32_t w2[2] = {q8.x, q8.y};
        int c[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = (int)((w2[k >> 2] >> (8 * (k & 3))) & 0xFFu) - z;
        const size_t o = j * rv.d_pad + col;
        if constexpr (FULL) {
            const float4 wa = *reinterpret_cast<const float4 *>(W + idx);
            const float4 wb = *reinterpret_cast<const float4 *>(W + idx + 4);
            const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
            const float ns = -S[j * G + col / g];
            float r[8];
            __align__(16) __nv_bfloat16 x[3][8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                r[k] = fmaf(ns, (float)c[k], w[k]);
                split3(r[k], x[0][k], x[1][k], x[2][k]);
            }
            *reinterpret_cast<float4 *>(rv.r + idx) = make_float4(r[0], r[1], r[2], r[3]);
            *reinterpret_cast<float4 *>(rv.r + idx + 4) = make_float4(r[4], r[5], r[6], r[7]);
            const size_t plane = (size_t)rv.p_pad * rv.d_pad;
#pragma unroll
            for (int t = 0; t < 3; ++t)
                *reinterpret_cast<uint4 *>(rv.planes + t * plane + o) = *reinterpret_cast<const uint4 *>(x[t]);
        }
        __align__(16) __half h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) h[k] = __int2half_rn(c[k]);
        *reinterpret_cast<uint4 *>(rv.cplane + o) = *reinterpret_cast<const uint4 *>(h);
    }
}

__global__ void init_rows_kernel(int *active, int *iters, int *accepted, int *ridge, int *rstat,
                                 int p) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < p) {
        active[j] = 1;
        iters[j] = 0;
        accepted[j] = 0;
        ridge[j] = 0;
        rstat[j] = 0;
    }
}

}  // namespace

StatusWord::StatusWord(cudaStream_t s) : s_(s) {
    StatusPool &pool = status_pool();
    {
        std::unique_lock<std::mutex> lock(pool.mu);
        pool.freed.wait(lock, [&] { return pool.taken != ~0ull; });
        index_ = 0;
        while (pool.taken >> index_ & 1) ++index_;
        pool.taken |= 1ull << index_;
    }
    void *base = nullptr;
    if (cudaGetSymbolAddress(&base, g_status_words) != cudaSuccess || !base)
        (void)cudaGetLastError();
    else
        ptr_ = static_cast<int *>(base) + index_;
}

StatusWord::~StatusWord() {
    // an error between clear() and read() leaves work that may use the word
    if (!idle_ && cudaStreamSynchronize(s_) != cudaSuccess) (void)cudaGetLastError();
    StatusPool &pool = status_pool();
    {
        std::lock_guard<std::mutex> lock(pool.mu);
        pool.taken &= ~(1ull << index_);
    }
    pool.freed.notify_one();
}

cudaError_t StatusWord::clear() {
    idle_ = false;
    return cudaMemsetAsync(ptr_, 0, sizeof(int), s_);
}

cudaError_t StatusWord::read(int *bits) {
    cudaError_t e = cudaMemcpyAsync(bits, ptr_, sizeof(int), cudaMemcpyDeviceToHost, s_);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s_);
    idle_ = e == cudaSuccess;
    return e;
}

int num_sms() {
    constexpr int kDevs = 64;
    static std::atomic<int> cache[kDevs];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = 0;
    }
    const bool cached = dev >= 0 && dev < kDevs;
    int n = cached ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    if (n <= 0) n = 1;
    if (cached) cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

cudaError_t set_max_dynamic_smem(const void *func, int bytes,
                                 std::atomic<unsigned long long> &done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

cudaError_t launch_validate(const uint8_t *Q, const int32_t *Z, int p, int d, int G, int qmax,
                            int *status, cudaStream_t s) {
    size_t nq = (size_t)p * d, nz = (size_t)p * G;
    size_t work = nq % 16 == 0 ? nq / 16 : nq;
    if (work < nz) work = nz;
    int blocks = (int)((work + 255) / 256 < (size_t)(8 * num_sms()) ? (work + 255) / 256 : 8 * num_sms());
    if (blocks < 1) blocks = 1;
    if (nq % 16 == 0 && (uintptr_t)Q % 16 == 0)
        validate16_kernel<<<blocks, 256, 0, s>>>(reinterpret_cast<const uint4 *>(Q), Z, nq / 16, nz,
                                                 qmax, status);
    else
        validate_kernel<<<blocks, 256, 0, s>>>(Q, Z, nq, nz, qmax, status);
    return cudaGetLastError();
}

cudaError_t launch_residual(const float *W, const float *S, const uint8_t *Q, const int32_t *Z,
                            ResidualView rv, int p, int g, cudaStream_t s) {
    size_t n = (size_t)p * rv.d;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 8 * num_sms()) blocks = 8 * num_sms();
    if (blocks < 1) blocks = 1;
    const bool eight = g % 8 == 0 && (uintptr_t)Q % 8 == 0 && rv.d_pad % 8 == 0;
    if (eight && !rv.r)
        residual8_kernel<false><<<blocks, 256, 0, s>>>(W, S, Q, Z, rv, p, g);
    else if (eight && (uintptr_t)W % 16 == 0 && (uintptr_t)rv.r % 16 == 0)
        residual8_kernel<true><<<blocks, 256, 0, s>>>(W, S, Q, Z, rv, p, g);
    else
        residual_kernel<<<blocks, 256, 0, s>>>(W, S, Q, Z, rv, p, g);
    return cudaGetLastError();
}

cudaError_t launch_init_rows(int *active, int *iters, int *accepted, int *ridge, int *rstat,
                             int p, cudaStream_t s) {
    init_rows_kernel<<<(p + 255) / 256, 256, 0, s>>>(active, iters, accepted, ridge, rstat, p);
    return cudaGetLastError();
}

// A wait that nothing completes: one thread polls a fresh mbarrier (count 1,
// no arrival), gives up after `polls` polls and records ST_TIMEOUT, as every
// kernel of the library does when one of its bounded waits runs out.
__global__ void wait_timeout_kernel(int *status, uint32_t polls) {
    __shared__ uint64_t bar;
    if (threadIdx.x != 0) return;
    const uint32_t b = tc::smem_u32(&bar);
    tc::mbar_init(b, 1);
    tc::fence_barrier_init();
    bool done = false;
    for (uint32_t i = 0; i < polls && !done; ++i) done = tc::mbar_try_wait(b, 0);
    if (!done) atomicOr(status, ST_TIMEOUT);
}

cudaError_t launch_wait_timeout(int *status, uint32_t polls, cudaStream_t s) {
    wait_timeout_kernel<<<1, 32, 0, s>>>(status, polls);
    return cudaGetLastError();
}

}  // namespace jarq
