// Write-back of a refined layer: negative-scale canonicalisation (App. E
// "Representing Negative Scales", Eq. canonicalization), the returned
// weights cast to a weight dtype (Sec. 3.1 Eq. quantized_group; App. E
// "Early stopping"), and b-bit code packing.  The entry points act on device
// memory, allocate nothing and validate the codes first.
#include "jarq_internal.cuh"

namespace jarq {
namespace {

// Every kernel below does nothing when the validation before it (same call)
// has set the call's status word.

// if s < 0, s' = -s, z' = qmax - z, q' = qmax - q.  A warp looks at 32 (row,
// group) scales at once and takes the negative ones in turn, so that a layer
// with few of them costs little more than reading its scales; VEC: four codes
// a lane (g a multiple of 4, Q 4-byte aligned).
template <bool VEC>
__global__ void canonicalize_kernel(float *__restrict__ S, uint8_t *__restrict__ Q,
                                    int32_t *__restrict__ Z, long long n, int d, int g, int qmax,
                                    const int *__restrict__ status) {
    if (*status) return;
    const int G = d / g, lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long b = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; b < n; b += nw * 32) {
        const long long i = b + lane;
        const float s = i < n ? S[i] : 0.f;
        const bool neg = s < 0.f;
        if (neg) {
            S[i] = -s;
            Z[i] = qmax - Z[i];
        }
        unsigned m = __ballot_sync(0xffffffffu, neg);
        while (m) {                                   // warp-uniform
            const long long k = b + (__ffs(m) - 1);
            m &= m - 1;
            uint8_t *q = Q + (size_t)(k / G) * d + (size_t)(k % G) * g;
            if (VEC) {
                // qmax - q byte by byte: 0 <= q <= qmax, no borrow
                for (int c = 4 * lane; c < g; c += 128) {
                    uint32_t *w = reinterpret_cast<uint32_t *>(q + c);
                    *w = 0x01010101u * (uint32_t)qmax - *w;
                }
            } else {
                for (int c = lane; c < g; c += 32) q[c] = (uint8_t)(qmax - q[c]);
            }
        }
    }
}

// what = s (q - z) rounded once to the output type.  The product of a float32
// and an integer of at most 9 bits is p + e with p rounded to float32 and e its
// exact error; for the 16-bit types p is first rounded to odd (its last bit
// set, toward zero, when e is not zero), which the second rounding then takes
// to the nearest value of the exact product (float32 has more than two bits
// beyond either type).
template <int DT>
__device__ __forceinline__ float weight(float s, int c) {
    const float cf = (float)c;
    float p = __fmul_rn(s, cf);
    if (DT != JARQ_F32) {
        const float e = __fmaf_rn(s, cf, -p);
        if (e != 0.f && isfinite(p)) {
            uint32_t u = __float_as_uint(p);
            if ((e < 0.f) != (p < 0.f)) --u;          // |p| above the product
            p = __uint_as_float(u | 1u);
        }
    }
    return p;
}

template <int DT>
__global__ void dequantize_kernel(const float *__restrict__ S, const uint8_t *__restrict__ Q,
                                  const int32_t *__restrict__ Z, void *__restrict__ out, int p,
                                  int d, int g, const int *__restrict__ status) {
    if (*status) return;
    const int G = d / g;
    const size_t n = (size_t)p * d;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t j = idx / d;
        const int grp = (int)(idx - j * d) / g;
        const float w = weight<DT>(S[j * G + grp], (int)Q[idx] - Z[j * G + grp]);
        if (DT == JARQ_F32)
            reinterpret_cast<float *>(out)[idx] = w;
        else if (DT == JARQ_F16)
            reinterpret_cast<__half *>(out)[idx] = __float2half_rn(w);
        else
            reinterpret_cast<__nv_bfloat16 *>(out)[idx] = __float2bfloat16_rn(w);
    }
}

// The same, 16 codes of one group per thread (g a multiple of 16, Q and the
// output 16-byte aligned): one 16-byte load, two or four 16-byte stores.
template <int DT>
__global__ void dequantize16_kernel(const float *__restrict__ S, const uint4 *__restrict__ Q16,
                                    const int32_t *__restrict__ Z, uint4 *__restrict__ out,
                                    size_t n16, int g16, const int *__restrict__ status) {
    if (*status) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t grp = i / g16;             // (row, group): groups tile the rows
        const float s = S[grp];
        const int z = Z[grp];
        const uint4 q = Q16[i];
        const uint32_t q4[4] = {q.x, q.y, q.z, q.w};
        uint32_t w[DT == JARQ_F32 ? 16 : 8];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float v = weight<DT>(s, (int)((q4[k / 4] >> (8 * (k % 4))) & 0xFFu) - z);
            if (DT == JARQ_F32) {
                w[k] = __float_as_uint(v);
            } else {
                const uint32_t h = DT == JARQ_F16
                                       ? (uint32_t)__half_as_ushort(__float2half_rn(v))
                                       : (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v));
                w[k / 2] = k % 2 ? w[k / 2] | (h << 16) : h;
            }
        }
        constexpr int kN = DT == JARQ_F32 ? 4 : 2;
#pragma unroll
        for (int k = 0; k < kN; ++k) out[i * kN + k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    }
}

// One thread per 32-bit output word: the codes whose bits [k b, k b + b)
// overlap bits [32 w, 32 w + 32) of the row's stream.
__global__ void pack_codes_kernel(const uint8_t *__restrict__ Q, uint32_t *__restrict__ out, int p,
                                  int d, int bits, int nw, const int *__restrict__ status) {
    if (*status) return;
    const size_t n = (size_t)p * nw;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t j = idx / nw;
        const int w = (int)(idx - j * nw);
        const long long lo = 32LL * w, hi = lo + 32;
        const int k0 = (int)(lo / bits), k1 = (int)min((long long)d, (hi + bits - 1) / bits);
        uint64_t v = 0;
        for (int k = k0; k < k1; ++k) {
            const long long pos = (long long)k * bits - lo;   // may be negative for k0
            const uint64_t q = Q[j * d + k];
            v |= pos >= 0 ? (q << pos) : (q >> (-pos));
        }
        out[idx] = (uint32_t)v;
    }
}

// The same for rows of a multiple of 32 codes (their streams then have no
// padding and follow one another): 32 codes per thread, two 16-byte loads, BITS
// whole words out.
template <int BITS>
__global__ void pack32_kernel(const uint4 *__restrict__ Q16, uint32_t *__restrict__ out, size_t n32,
                              const int *__restrict__ status) {
    if (*status) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n32;
         i += (size_t)gridDim.x * blockDim.x) {
        const uint4 a = Q16[2 * i], b = Q16[2 * i + 1];
        const uint32_t q4[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        uint32_t w[BITS] = {};
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const uint32_t q = (q4[k / 4] >> (8 * (k % 4))) & 0xFFu;
            const int pos = k * BITS, at = pos / 32, sh = pos % 32;
            w[at] |= q << sh;
            if (sh + BITS > 32) w[at + 1] |= q >> (32 - sh);
        }
#pragma unroll
        for (int k = 0; k < BITS; ++k) out[i * BITS + k] = w[k];
    }
}

int grid_for(size_t n) {
    size_t b = (n + 255) / 256;
    const size_t cap = (size_t)32 * num_sms();
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

// Validate codes (and zero points when Z is given); then `launch(stream,
// status)` a kernel that does nothing when the status word is set.  One
// synchronisation for both: waiting for the verdict before the launch cost
// about 15 us a call.  The word is this call's alone: another call's verdict
// must not stop this kernel halfway, nor its start let this one run on bad codes.
template <class F>
jarq_status checked_run(const uint8_t *Q, const int32_t *Z, int p, int d, int G, int qmax,
                        cudaStream_t st, F launch) {
    StatusWord status(st);
    if (!status.ptr()) return JARQ_ERR_CUDA;
    int host = 0;
    cudaError_t e = status.clear();
    if (e == cudaSuccess) e = launch_validate(Q, Z, p, d, Z ? G : 0, qmax, status.ptr(), st);
    if (e == cudaSuccess) e = launch(st, status.ptr());
    if (e == cudaSuccess) e = status.read(&host);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return JARQ_ERR_CUDA;
    }
    count_launches(2);
    return host ? JARQ_ERR_ARG : JARQ_OK;
}

template <int DT>
cudaError_t launch_dequantize(const float *S, const uint8_t *Q, const int32_t *Z, void *out, int p,
                              int d, int g, const int *status, cudaStream_t st) {
    const size_t n = (size_t)p * d;
    if (g % 16 == 0 && (((uintptr_t)Q | (uintptr_t)out) & 15) == 0)
        dequantize16_kernel<DT><<<grid_for(n / 16), 256, 0, st>>>(
            S, reinterpret_cast<const uint4 *>(Q), Z, reinterpret_cast<uint4 *>(out), n / 16, g / 16,
            status);
    else
        dequantize_kernel<DT><<<grid_for(n), 256, 0, st>>>(S, Q, Z, out, p, d, g, status);
    return cudaGetLastError();
}

template <int BITS>
cudaError_t launch_pack(const uint8_t *Q, uint32_t *out, int p, int d, int bits, const int *status,
                        cudaStream_t st) {
    if constexpr (BITS <= 8) {
        if (bits != BITS) return launch_pack<BITS + 1>(Q, out, p, d, bits, status, st);
        const size_t n = (size_t)p * d;
        if (d % 32 == 0 && ((uintptr_t)Q & 15) == 0) {
            pack32_kernel<BITS><<<grid_for(n / 32), 256, 0, st>>>(reinterpret_cast<const uint4 *>(Q), out,
                                                                  n / 32, status);
        } else {
            const int nw = (int)(((long long)d * bits + 31) / 32);
            pack_codes_kernel<<<grid_for((size_t)p * nw), 256, 0, st>>>(Q, out, p, d, bits, nw, status);
        }
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

}  // namespace

bool on_device(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (at.type == cudaMemoryTypeManaged) return true;
    if (at.type != cudaMemoryTypeDevice) return false;
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return at.device == cur;
}

}  // namespace jarq

using namespace jarq;

extern "C" {

jarq_status jarq_canonicalize(float *S, uint8_t *Q, int32_t *Z, int dout, int din, int group_size,
                              int bits, void *stream) {
    if (dout < 0 || din <= 0 || group_size <= 0 || din % group_size || bits < 1 || bits > 8)
        return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    if (!S || !Q || !Z || !on_device(S) || !on_device(Q) || !on_device(Z)) return JARQ_ERR_ARG;
    const int G = din / group_size, qmax = (1 << bits) - 1;
    return checked_run(Q, Z, dout, din, G, qmax, (cudaStream_t)stream, [&](cudaStream_t st, const int *status) {
        const long long n = (long long)dout * G;
        if (group_size % 4 == 0 && ((uintptr_t)Q & 3) == 0)
            canonicalize_kernel<true><<<grid_for((size_t)n), 256, 0, st>>>(S, Q, Z, n, din, group_size,
                                                                           qmax, status);
        else
            canonicalize_kernel<false><<<grid_for((size_t)n), 256, 0, st>>>(S, Q, Z, n, din, group_size,
                                                                            qmax, status);
        return cudaGetLastError();
    });
}

jarq_status jarq_dequantize(const float *S, const uint8_t *Q, const int32_t *Z, int dout, int din,
                            int group_size, int bits, jarq_dtype dtype, void *W_out,
                            void *stream) {
    if (dout < 0 || din <= 0 || group_size <= 0 || din % group_size || bits < 1 || bits > 8 ||
        (dtype != JARQ_F32 && dtype != JARQ_F16 && dtype != JARQ_BF16))
        return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    if (!S || !Q || !Z || !W_out || !on_device(S) || !on_device(Q) || !on_device(Z) ||
        !on_device(W_out))
        return JARQ_ERR_ARG;
    const int G = din / group_size, qmax = (1 << bits) - 1;
    return checked_run(Q, Z, dout, din, G, qmax, (cudaStream_t)stream, [&](cudaStream_t st, const int *status) {
        if (dtype == JARQ_F32)
            return launch_dequantize<JARQ_F32>(S, Q, Z, W_out, dout, din, group_size, status, st);
        if (dtype == JARQ_F16)
            return launch_dequantize<JARQ_F16>(S, Q, Z, W_out, dout, din, group_size, status, st);
        return launch_dequantize<JARQ_BF16>(S, Q, Z, W_out, dout, din, group_size, status, st);
    });
}

jarq_status jarq_pack_codes(const uint8_t *Q, int dout, int din, int bits, uint32_t *packed,
                            void *stream) {
    if (dout < 0 || din <= 0 || bits < 1 || bits > 8) return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    if (!Q || !packed || !on_device(Q) || !on_device(packed)) return JARQ_ERR_ARG;
    return checked_run(Q, nullptr, dout, din, 0, (1 << bits) - 1, (cudaStream_t)stream,
                       [&](cudaStream_t st, const int *status) {
                           return launch_pack<1>(Q, packed, dout, din, bits, status, st);
                       });
}

}  // extern "C"
