// Residual products (H r) on the tensor cores (tcgen05 + TMA), split precision.
//
// The residual r = w - D_s (q - z) (Eq. quantized_group) and the symmetric
// Hessian H are both split exactly into three bf16 planes,
// x = x1 + x2 + x3 (truncation splits of the float32 value), and
//     H r ~= sum over the eight products r_a H_b but r_3 H_3
// (a, b = 1..3; the dropped product is below float32 resolution),
// accumulated in float32.  Tensor-core accumulation truncates, so its error
// grows with the number of products summed into one accumulator; the kernel
// therefore (a) keeps the leading product r_1 H_1 and the seven small products
// in separate TMEM accumulators, and (b) drains both into float32 registers
// (round to nearest) every 64 columns of K, restarting the TMEM sums at zero.
// Two accumulator pairs alternate so the MMAs of one 64-wide K period overlap
// the drain of the previous one.  Used for the objective (Eq. bbmils_columns).
//
// One CTA computes a 128-row x 128-column output tile:
//   warp 0      TMA producer: 3 A planes + 3 B planes per 64-wide K chunk
//   warp 1      TMEM allocation and the single-thread MMA issuer
//   warps 2..9  drain (TMEM -> register sums) and store (float32); warp w
//               reads TMEM lanes 32 (w % 4) .. + 31 and half (w - 2) / 4 of
//               the tile's columns
// Operands are K-major: A = r planes [3][p_pad][d_pad], B = H planes
// [3][d_pad][d_pad] (H symmetric, so row n of H is column n), both loaded
// with 128-byte swizzle.
#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kTile = 128 * 64 * 2;   // bytes of one 128 x 64 bf16 tile of A or B
constexpr int kStage = 6 * kTile;
constexpr int kStages = 2;
constexpr int kSmem = 1024 + kStages * kStage + 256;
constexpr uint32_t kIdesc = tc::idesc_bf16_f32(128, 128);
constexpr int kProducts = 8;
constexpr int kGroupRows = 8;         // row tiles per band of the tile order
// (A plane, B plane) of each product, smallest first; the last, (0, 0), is
// the leading one.
__host__ __device__ constexpr int prod_a(int k) {
    constexpr int t[8] = {2, 1, 2, 1, 0, 1, 0, 0};
    return t[k];
}
__host__ __device__ constexpr int prod_b(int k) {
    constexpr int t[8] = {1, 2, 0, 1, 2, 0, 1, 0};
    return t[k];
}

struct HrArgs {
    float *out;            // [p][d]
    int p, d;
    int p_pad, d_pad;      // rows between the planes of A and of B
    int *status;
};

// kStalled: for the self-test, the issuer stops after one chunk.
template <bool kStalled>
__global__ void __launch_bounds__(320, 1)
    tc_hr_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                 HrArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(smem + kStages * kStage);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * kStages + 5);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tile order: grouped so that consecutive CTAs share column tiles within
    // a band of kGroupRows row tiles (L2 reuse of both operands)
    const int lin = blockIdx.y * gridDim.x + blockIdx.x;
    const int per_band = kGroupRows * gridDim.y;
    const int band = lin / per_band, in_band = lin % per_band;
    const int rows_in_band = min(kGroupRows, (int)gridDim.x - band * kGroupRows);
    const int j0 = (band * kGroupRows + in_band % rows_in_band) * 128;
    const int n0 = (in_band / rows_in_band) * 128;
    const int nk = a.d_pad / 64;      // 64-wide K chunks, a drain period each

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kStages + s); };
    auto afull = [&](int b) { return tc::smem_u32(bars + 2 * kStages + b); };
    auto aempty = [&](int b) { return tc::smem_u32(bars + 2 * kStages + 2 + b); };
    const uint32_t closing = tc::smem_u32(bars + 2 * kStages + 4);
    auto tileA = [&](int s, int t) { return tc::smem_u32(smem + s * kStage + t * kTile); };
    auto tileB = [&](int s, int t) { return tc::smem_u32(smem + s * kStage + (3 + t) * kTile); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(full(s), 1);
            tc::mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(afull(b), 1);
            tc::mbar_init(aempty(b), 8);   // one arrival per drain warp
        }
        tc::mbar_init(closing, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);   // [buffer][leading, small] x 128 columns
        tc::tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        tc::prefetch_tmap(&mapA);
        tc::prefetch_tmap(&mapB);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---------------- producer
        int issued = 0;
        for (int c = 0; c < nk; ++c) {
            const int s = c % kStages;
            const uint32_t ph = (c / kStages) & 1;
            if (!tc::mbar_wait<kPolls>(empty(s), ph ^ 1) || *abort_flag) {
                *abort_flag = 1;
                break;
            }
            tc::mbar_expect_tx(full(s), kStage);
#pragma unroll
            for (int t = 0; t < 3; ++t) tc::tma_load_2d(tileA(s, t), &mapA, full(s), c * 64, j0 + t * a.p_pad);
#pragma unroll
            for (int t = 0; t < 3; ++t) tc::tma_load_2d(tileB(s, t), &mapB, full(s), c * 64, n0 + t * a.d_pad);
            issued = c + 1;
        }
        // do not leave before the copies have landed
        for (int c = issued > kStages ? issued - kStages : 0; c < issued && !*abort_flag; ++c)
            if (!tc::mbar_wait<kPolls>(full(c % kStages), (c / kStages) & 1)) *abort_flag = 1;
        if (*abort_flag) tc::abandon_ring(full(0), kStages, issued, true);
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        for (int c = 0; c < (kStalled ? 1 : nk) && !*abort_flag; ++c) {
            const int b = c & 1, s = c % kStages;
            if (!tc::mbar_wait<kPolls>(aempty(b), ((c >> 1) & 1) ^ 1)) {
                *abort_flag = 1;
                break;
            }
            const uint32_t acc_big = tmem + b * 256, acc_small = acc_big + 128;
            if (!tc::mbar_wait<kPolls>(full(s), (c / kStages) & 1) || *abort_flag) {
                *abort_flag = 1;
                break;
            }
            tc::tc_fence_after();
#pragma unroll
            for (int sub = 0; sub < 4; ++sub) {
#pragma unroll
                for (int pr = 0; pr < kProducts; ++pr) {
                    const uint64_t ad = tc::sdesc_sw128(tileA(s, prod_a(pr))) + 2 * sub;
                    const uint64_t bd = tc::sdesc_sw128(tileB(s, prod_b(pr))) + 2 * sub;
                    if (pr == kProducts - 1)
                        tc::mma_bf16(acc_big, ad, bd, kIdesc, sub != 0);
                    else
                        tc::mma_bf16(acc_small, ad, bd, kIdesc, sub != 0 || pr != 0);
                }
            }
            tc::mma_commit(empty(s));
            tc::mma_commit(afull(b));
        }
        if (!tc::mma_done<kPolls>(closing, true)) *abort_flag = 1;
    } else if (warp >= 2) {
        // ---------------- drain + store (decisions warp-uniform: tcgen05.ld is .aligned)
        constexpr int HB = 64;                     // columns per drain warp
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int row = j0 + 32 * q + lane;
        float acc[HB];
#pragma unroll
        for (int c = 0; c < HB; ++c) acc[c] = 0.f;
        bool ok = true;
        for (int c = 0; c < nk; ++c) {
            const int b = c & 1;
            bool w = tc::mbar_wait<kPolls>(afull(b), (c >> 1) & 1);
            w = __shfl_sync(0xffffffffu, w && !*abort_flag, 0);
            tc::tc_fence_after();
            if (!w) {
                ok = false;
                *abort_flag = 1;
                break;
            }
            const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + b * 256 + half * HB;
#pragma unroll
            for (int cc = 0; cc < HB; cc += 16) {
                uint32_t vb[16], vs[16];
                tc::tmem_ld16(base + cc, vb);
                tc::tmem_ld16(base + 128 + cc, vs);
                tc::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    acc[cc + e] += __uint_as_float(vb[e]) + __uint_as_float(vs[e]);
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(aempty(b));
        }
        float *orow = a.out + (size_t)row * a.d;
        if (ok && row < a.p) {
#pragma unroll
            for (int e = 0; e < HB; e += 4) {
                const int col = n0 + half * HB + e;
                if (col + 3 < a.d) {
                    *reinterpret_cast<float4 *>(orow + col) =
                        make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
                } else {
                    for (int u = 0; u < 4; ++u)
                        if (col + u < a.d) orow[col + u] = acc[e + u];
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicOr(a.status, ST_TIMEOUT);
}

}  // namespace

// Full product H r for all rows: out[p][d].
cudaError_t launch_tc_hr_full(const CUtensorMap &mapA, const CUtensorMap &mapB, float *out, int p,
                              int p_pad, int d, int d_pad, int *status, cudaStream_t s,
                              bool stalled) {
    HrArgs a{out, p, d, p_pad, d_pad, status};
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t e = set_max_dynamic_smem((const void *)kernel, kSmem, done);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, dim3(p_pad / 128, d_pad / 128), dim3(320), (size_t)kSmem, s, false, mapA, mapB, a);
    };
    static std::atomic<unsigned long long> done[2];
    return stalled ? run(tc_hr_kernel<true>, done[1]) : run(tc_hr_kernel<false>, done[0]);
}

}  // namespace jarq
