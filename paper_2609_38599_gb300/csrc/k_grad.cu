// Per-row reduction of the full residual product H r (tensor cores):
// F_j = r_j^T (H r_j) (Eq. bbmils_columns).
#include "jarq_internal.cuh"

namespace jarq {
namespace {

// Per row (kRowWarps warps, one block): F_j = r_j . (H r_j) in float64.  Bound by
// float64: a multiply-add and two conversions an entry, at 1/64 of the float32
// rate.  102 us on 4096 x 4096; with one warp per row, which also formed the
// scale gradient, 240 us.
constexpr int kRowWarps = 4;

__global__ void __launch_bounds__(32 * kRowWarps) grad_kernel(const float *__restrict__ r,
                                                              const float *__restrict__ Hr,
                                                              double *__restrict__ F, int d) {
    __shared__ double part[kRowWarps];
    const int row = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t off = (size_t)row * d;
    double fs = 0.0;
#pragma unroll 4
    for (int m = threadIdx.x; m < d; m += 32 * kRowWarps)
        fs += (double)r[off + m] * (double)Hr[off + m];
    for (int o = 16; o; o >>= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
    if (lane == 0) part[w] = fs;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = part[0];
        for (int k = 1; k < kRowWarps; ++k) v += part[k];
        F[row] = v;
    }
}

}  // namespace

cudaError_t launch_grad(const float *r, const float *Hr, double *F, int p, int d, cudaStream_t s) {
    grad_kernel<<<p, 32 * kRowWarps, 0, s>>>(r, Hr, F, d);
    return cudaGetLastError();
}

}  // namespace jarq
