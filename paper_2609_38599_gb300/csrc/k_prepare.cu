// Hessian preparation: symmetrisation, per-group Cholesky factors and the
// folded operand of the sweep's residual products.
//
// Sec. 3.3.2, Eq. group_qr: each group's factor R_i (A_i = U_i R_i) is
// computed once per layer and reused for every output row and iteration.
// With H = A^T A, R_i^T R_i = H_ii, so R_i is taken as the upper Cholesky
// factor of H_ii (equal to the QR factor up to row signs, to which the
// Babai recursion is invariant).  The factor and its inverse are computed in
// float64 in shared memory (the failing case of a block that is not positive
// definite leaves its inverse undefined; the call then fails):
//   Lf[i]   = L_i = R_i^T          (lower, L[l][m] = R_i[m][l]), float32, packed for the
//             Babai kernel (factor_row in jarq_internal.cuh)
//   Rinv[i] = R_i^{-1}             (upper, row-major), float64
// The Babai target of Eq. babai_update needs y = R_i^{-T} (H r)_i / s.  The
// rows H_i of group i are dominated by the low-rank part of H, which R_i^{-T}
// cancels: forming (H r)_i first and applying R_i^{-T} afterwards amplifies
// the product's rounding by up to sqrt(cond(H_ii)).  The sweep therefore
// works with the folded rows
//   Ht[grp i, :] = R_i^{-T} H[grp i, :]
// computed here once, in double-float (hi + lo) from the float64 inverse.
#include "jarq_internal.cuh"

namespace jarq {
namespace {

// out = (H + H^T)/2 + nu2 I, through 32x32 shared-memory tiles, plus its
// exact three-plane bf16 split (planes [3][d_pad][d_pad], pitch d_pad).
__global__ void symmetrize_kernel(const float *__restrict__ H, float *__restrict__ Hs,
                                  __nv_bfloat16 *__restrict__ planes, int d, int d_pad,
                                  float nu2) {
    __shared__ float tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    for (int yy = ty; yy < 32; yy += 8) {
        int row = bx + yy, col = by + tx;  // transposed block
        tile[yy][tx] = (row < d && col < d) ? H[(size_t)row * d + col] : 0.f;
    }
    __syncthreads();
    for (int yy = ty; yy < 32; yy += 8) {
        int row = by + yy, col = bx + tx;
        if (row < d && col < d) {
            float v = 0.5f * (H[(size_t)row * d + col] + tile[tx][yy]);
            if (row == col) v += nu2;
            Hs[(size_t)row * d + col] = v;
            __nv_bfloat16 a, b, c;
            split3(v, a, b, c);
            const size_t plane = (size_t)d_pad * d_pad, off = (size_t)row * d_pad + col;
            planes[off] = a;
            planes[plane + off] = b;
            planes[2 * plane + off] = c;
        }
    }
}

// One block per group: float64 Cholesky of H_ii in shared memory.  Bound by
// float64 (two lanes per clock on an SM, one SM per group): the update of the
// trailing lower triangle goes row by row over the warps, so that no lane
// works above the diagonal except in a row's last 32 columns.
__global__ void group_factor_kernel(const float *__restrict__ Hs, float *__restrict__ Lf,
                                    double *__restrict__ L64, int d, int g, int *status) {
    extern __shared__ double smem[];
    const int ld = g + 1;
    double *A = smem;               // [g][g+1]
    __shared__ int failed;
    const int grp = blockIdx.x;
    const int base = grp * g;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    if (tid == 0) failed = 0;
    for (int idx = tid; idx < g * g; idx += nt) {
        int a = idx / g, b = idx % g;
        A[a * ld + b] = (double)Hs[(size_t)(base + a) * d + base + b];
    }
    __syncthreads();
    // right-looking Cholesky, lower triangle
    for (int k = 0; k < g; ++k) {
        const double piv = A[k * ld + k];
        if (!(piv > 0.0) || !isfinite(piv)) {       // every thread sees the same pivot
            if (tid == 0) failed = 1;
            break;
        }
        const double lkk = sqrt(piv);
        for (int a = k + 1 + tid; a < g; a += nt) A[a * ld + k] /= lkk;
        __syncthreads();
        if (tid == 0) A[k * ld + k] = lkk;
        for (int a = k + 1 + warp; a < g; a += nw) {
            const double l = A[a * ld + k];
            for (int b = k + 1 + lane; b <= a; b += 32) A[a * ld + b] -= l * A[b * ld + k];
        }
        __syncthreads();
    }
    __syncthreads();
    if (failed) {
        if (tid == 0) atomicOr(status, ST_NOT_SPD);
        return;
    }
    float *Lo = Lf + (size_t)grp * factor_floats(g);
    double *Ld = L64 + (size_t)grp * g * g;
    for (int idx = tid; idx < g * g; idx += nt) {
        const int h = idx / g, l = idx % g;
        Ld[idx] = (l <= h) ? A[h * ld + l] : 0.0;
        if (l < 32 * (h / 32 + 1))
            Lo[factor_row(h) + l] = (l < 4 * (h / 4)) ? (float)A[h * ld + l] : 0.f;
    }
    for (int idx = tid; idx < 2 * g; idx += nt) {
        const int q = 4 * (idx / 8), e = idx % 8;
        const int h = e < 3 ? 3 : e < 5 ? 2 : 1;                       // 3 3 3 2 2 1
        const int l = e < 3 ? 2 - e : e < 5 ? 4 - e : 0;               // 2 1 0 1 0 0
        Lo[factor_tri(g) + idx] = e < 6 ? (float)A[(q + h) * ld + q + l] : 0.f;
    }
    for (int l = tid; l < g; l += nt) {
        const float v = (float)A[l * ld + l];
        Lo[factor_diag(g) + l] = v;
        Lo[factor_rdiag(g) + l] = 1.0f / v;
    }
}

// R_i^{-1} = (L_i^{-1})^T, column j of L^{-1} (= row j of R^{-1}) per warp by
// forward substitution in float64, kInvCols columns per block: the columns are
// independent, so the work spreads over g / kInvCols times the SMs that the
// factorisation uses.  Lane l keeps the entries l + 32 m of its column.  Also
// written as float pairs (hi, lo) for the folded rows.
constexpr int kInvCols = 16;

template <int NT>
__global__ void __launch_bounds__(32 * kInvCols) group_inverse_kernel(const double *__restrict__ L64,
                                                                      double *__restrict__ Rinv,
                                                                      float2 *__restrict__ RinvF) {
    constexpr int g = 32 * NT, ld = g + 1;
    extern __shared__ double smem[];
    double *A = smem;               // [g][g+1]
    double *rd = smem + g * ld;     // [g] 1 / L_bb
    const size_t off = (size_t)blockIdx.x * g * g;
    for (int idx = threadIdx.x; idx < g * g; idx += blockDim.x) A[(idx / g) * ld + idx % g] = L64[off + idx];
    __syncthreads();
    for (int b = threadIdx.x; b < g; b += blockDim.x) rd[b] = 1.0 / A[b * ld + b];
    __syncthreads();
    const int lane = threadIdx.x & 31, j = blockIdx.y * kInvCols + (threadIdx.x >> 5);
    double x[NT];
#pragma unroll
    for (int m = 0; m < NT; ++m) x[m] = lane + 32 * m == j ? 1.0 : 0.0;
#pragma unroll
    for (int mb = 0; mb < NT; ++mb) {
        for (int bb = max(0, j - 32 * mb); bb < 32; ++bb) {      // warp-uniform
            const int b = 32 * mb + bb;
            const double xb = __shfl_sync(0xffffffffu, x[mb], bb) * rd[b];
            if (lane == bb) x[mb] = xb;
#pragma unroll
            for (int m = mb; m < NT; ++m)
                if (lane + 32 * m > b) x[m] = fma(-A[(lane + 32 * m) * ld + b], xb, x[m]);
        }
    }
#pragma unroll
    for (int m = 0; m < NT; ++m) {
        const size_t o = off + (size_t)j * g + lane + 32 * m;
        const float hi = (float)x[m];
        Rinv[o] = x[m];
        RinvF[o] = make_float2(hi, (float)(x[m] - (double)hi));
    }
}

// (s, e) with s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Ht[i g + a, k] = sum_{b <= a} Rinv_i[b][a] Hs[i g + b, k] for one group i
// (blockIdx.y) and 128 columns k (blockIdx.x), double-float products and sums
// (11 float32 operations a term), written as the float pair (hi, lo) [d][d].
// Rinv_i's pairs and the H tile lie in shared memory; warp w computes the rows
// 4 w .. 4 w + 3 and their mirror g - 4 - 4 w .., so that every warp has the
// same number of terms, and lane l the columns 4 l .. 4 l + 3: five 16-byte
// shared loads for 32 terms (four of them one address for the warp).  One
// output a thread and step, three shared loads a term, took 1.31 ms on 4096 x
// 4096.
constexpr int kHtCols = 128;

template <int NT>
__global__ void __launch_bounds__(128 * NT, 1) htilde_kernel(const float *__restrict__ Hs,
                                                             const float2 *__restrict__ RinvF,
                                                             float *__restrict__ out_hi,
                                                             float *__restrict__ out_lo, int d) {
    constexpr int g = 32 * NT;
    extern __shared__ __align__(16) float hsm[];
    float *rh = hsm;                   // [g][g] hi parts, Rinv[b][a] at b * g + a
    float *rl = rh + g * g;            // [g][g] lo parts
    float *ht = rl + g * g;            // [g][kHtCols] rows of H for this group
    const int i = blockIdx.y, k0 = blockIdx.x * kHtCols;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const float2 *Ri = RinvF + (size_t)i * g * g;
    for (int idx = tid; idx < g * g; idx += blockDim.x) {
        const float2 v = Ri[idx];
        rh[idx] = v.x;
        rl[idx] = v.y;
    }
    for (int idx = tid; idx < g * kHtCols / 4; idx += blockDim.x) {
        const int b = idx / (kHtCols / 4), kk = 4 * (idx % (kHtCols / 4));
        *reinterpret_cast<float4 *>(ht + b * kHtCols + kk) =
            k0 + kk < d ? *reinterpret_cast<const float4 *>(Hs + (size_t)(i * g + b) * d + k0 + kk)
                        : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const int a_lo = 4 * w, a_hi = g - 4 - 4 * w;
    float sh[8][4] = {}, sl[8][4] = {};     // rows a_lo + r, a_hi + r; columns 4 lane + c
    auto terms = [&](int r0, const float *prh, const float *prl, const float4 &h4) {
        const float4 r4 = *reinterpret_cast<const float4 *>(prh), l4 = *reinterpret_cast<const float4 *>(prl);
        const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
        const float rv[4] = {r4.x, r4.y, r4.z, r4.w}, lv[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float m = rv[r] * hv[c];
                float e = fmaf(rv[r], hv[c], -m);
                e = fmaf(lv[r], hv[c], e);
                float s2, e2;
                two_sum(sh[r0 + r][c], m, s2, e2);
                sh[r0 + r][c] = s2;
                sl[r0 + r][c] += e2 + e;
            }
    };
    // Rinv[b][a] is zero for b > a: the terms up to a row quad's last row
    int b = 0;
    for (; b < a_lo + 4; ++b) {
        const float4 h4 = *reinterpret_cast<const float4 *>(ht + b * kHtCols + 4 * lane);
        terms(0, rh + b * g + a_lo, rl + b * g + a_lo, h4);
        terms(4, rh + b * g + a_hi, rl + b * g + a_hi, h4);
    }
    for (; b < a_hi + 4; ++b) {
        const float4 h4 = *reinterpret_cast<const float4 *>(ht + b * kHtCols + 4 * lane);
        terms(4, rh + b * g + a_hi, rl + b * g + a_hi, h4);
    }
    if (k0 + 4 * lane < d) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int a = r < 4 ? a_lo + r : a_hi + r - 4;
            float x[4], y[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) two_sum(sh[r][c], sl[r][c], x[c], y[c]);
            const size_t off = (size_t)(i * g + a) * d + k0 + 4 * lane;
            *reinterpret_cast<float4 *>(out_hi + off) = make_float4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<float4 *>(out_lo + off) = make_float4(y[0], y[1], y[2], y[3]);
        }
    }
}

// The band of Ht blocks below the diagonal that the Babai kernel reads column
// by column (jarq_hessian::band), from Ht's digit planes [4][d_pad][d_pad]:
// one 32 x 32 tile of one block per CTA, transposed in shared memory.
__global__ void band_kernel(const __half *__restrict__ dig, int2 *__restrict__ band, int d,
                            int d_pad, int g) {
    __shared__ int2 tile[32][33];
    const int G = d / g, i = blockIdx.y, dd = blockIdx.z, i2 = i + 1 + dd;
    if (i2 >= G) return;
    const int nt = g / 32, m0 = (blockIdx.x / nt) * 32, k0 = (blockIdx.x % nt) * 32;
    const size_t plane = (size_t)d_pad * d_pad;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    for (int y = ty; y < 32; y += 8) {
        const size_t off = (size_t)(i2 * g + m0 + y) * d_pad + i * g + k0 + tx;
        int a[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) a[t] = __half2int_rn(dig[t * plane + off]);
        tile[y][tx] = make_int2(a[0] * 1024 + a[1], a[2] * 1024 + a[3]);
    }
    __syncthreads();
    int2 *out = band + ((size_t)i * gridDim.z + dd) * g * g;
    for (int y = ty; y < 32; y += 8) out[(size_t)(k0 + y) * g + m0 + tx] = tile[tx][y];
}

}  // namespace

cudaError_t launch_band(const __half *Htdig, int2 *band, int d, int d_pad, int g, cudaStream_t s) {
    band_kernel<<<dim3((g / 32) * (g / 32), d / g, sweep_block(g) - 1), dim3(32, 8), 0, s>>>(
        Htdig, band, d, d_pad, g);
    return cudaGetLastError();
}

cudaError_t launch_symmetrize(const float *H, float *Hs, __nv_bfloat16 *Hplanes, int d, int d_pad,
                              float nu2, cudaStream_t s) {
    dim3 grid((d + 31) / 32, (d + 31) / 32), block(32, 8);
    symmetrize_kernel<<<grid, block, 0, s>>>(H, Hs, Hplanes, d, d_pad, nu2);
    return cudaGetLastError();
}

cudaError_t launch_group_factor(const float *Hs, float *Lf, double *L64, double *Rinv,
                                float2 *RinvF, int d, int g, int *status, cudaStream_t s) {
    auto bytes = [](int n) { return (n * (n + 1) + n) * (int)sizeof(double); };
    const int smem = bytes(g);
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = set_max_dynamic_smem((const void *)group_factor_kernel, bytes(kMaxGroupSize), attr_done);
    if (e != cudaSuccess) return e;
    group_factor_kernel<<<d / g, 256, smem, s>>>(Hs, Lf, L64, d, g, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const dim3 grid(d / g, g / kInvCols);
    if (g == 128) {
        e = cudaFuncSetAttribute(group_inverse_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        group_inverse_kernel<4><<<grid, 32 * kInvCols, smem, s>>>(L64, Rinv, RinvF);
    } else if (g == 64) {
        e = cudaFuncSetAttribute(group_inverse_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        group_inverse_kernel<2><<<grid, 32 * kInvCols, smem, s>>>(L64, Rinv, RinvF);
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_htilde(const float *Hs, const float2 *RinvF, float *out_hi, float *out_lo, int d,
                          int g, cudaStream_t s) {
    const int smem = (2 * g * g + g * kHtCols) * (int)sizeof(float);
    const dim3 grid((d + kHtCols - 1) / kHtCols, d / g);
    cudaError_t e;
    if (g == 128) {
        e = cudaFuncSetAttribute(htilde_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        htilde_kernel<4><<<grid, 512, smem, s>>>(Hs, RinvF, out_hi, out_lo, d);
    } else if (g == 64) {
        e = cudaFuncSetAttribute(htilde_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        htilde_kernel<2><<<grid, 256, smem, s>>>(Hs, RinvF, out_hi, out_lo, d);
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace jarq
