// Calibration Hessian accumulation H += scale * X^T X from fp16 activations
// on the tensor cores.  The H-form uses H = A^T A for the augmented design
// A = [X~; nu I] of Eq. strict_target, i.e. H = X~^T X~ + nu^2 I (App.
// "Propagation-Corrected Targets and QEP" writes it out); this entry point
// forms the X~^T X~ part (nu^2 I is added when the Hessian is prepared).  The
// paper forms its products from FP16 activations in FP32 (App. "Metrics");
// here every fp16 x fp16 product is exact and the sums are float32.
//
// X is read as it is produced, token-major [n][d], with no transpose: a TMA
// box of 64 tokens x 64 features lands as 64 rows of 128 bytes (128-byte
// swizzle), which is the MN-major operand layout of tcgen05.mma (MN =
// features, contiguous; K = tokens, 128 bytes apart; 8-token atoms 1024
// bytes apart; 64-feature atoms one box, 8 KiB, apart).
//
// A pair of CTAs (cta_group::2) computes 256 x 256 tiles (rows r0.., columns
// c0..) of the upper triangle of X^T X over all n tokens, every npairs-th tile of
// an order in which the tiles that run at one time lie in blocks of 12 x 12 tiles
// (they share their panels of X in L2).  In each CTA:
//   warp 0      TMA producer, 5-stage ring of 64-token chunks: the features of
//               its own 128 rows and of its half of the columns (on a diagonal
//               tile these are the same), onto the even CTA's barriers
//   warp 1      TMEM allocation; in the even CTA the MMA issuer: one
//               M256 x N256 x K16 MMA per 16 tokens
//   warps 2..9  drain: every 512 tokens the TMEM accumulator (restarted at
//               zero, two of them alternate) is added into float32
//               registers.  At the end of a tile each warp adds its 32 x 128
//               part to H, 32 x 32 at a time through its own shared memory, as
//               H[row][col] and as H[col][row], in float4; the MMAs of the next
//               tile run meanwhile.
// Each unordered pair {i, j} belongs to exactly one tile element with
// col >= row, so every element of H is written exactly once.
//
// What bounds it: for many tokens the MMAs (d = 11008, 32768 tokens: 2.54 ms; 2.43
// ms without the additions to H; the same flops at the 1.75 PFLOP/s that a long
// run sustains take 2.3 ms), for few the additions to H (d = 4096, 2048 tokens: 58
// us; 30 us without them).  One CTA per 128 x 256 tile, its ring reused to stage
// the whole tile, took 2.87 ms and 72 us: 192 bytes of shared memory were written
// and read per cycle of the MMAs, now 128.  Measured and not kept: tiles in
// columns over the whole matrix (2.98 ms), a ring of 4 stages (3.05 ms) or 6 (2.69
// ms), sixteen drain warps (62 us), H prefetched into L2 ahead of the additions
// (62 us, 2.73 ms).
#include <math.h>

#include <algorithm>

#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kBox = 64 * 64 * 2;          // one TMA box: 64 tokens x 64 features, fp16
constexpr int kTileA = 2 * kBox;           // 128 row features
constexpr int kTileB = 2 * kBox;           // 128 of the 256 column features
constexpr int kStage = kTileA + kTileB;
constexpr int kStages = 5;
constexpr int kBars = 2 * kStages + 5;     // full, empty, afull[2], aempty[2], closing
constexpr int kDrainWarps = 8;
constexpr int kTld = 33;                   // row pitch (floats) of a staged 32 x 32 part
constexpr int kPart = 32 * kTld * 4;
constexpr int kSmem = 1024 + kStages * kStage + kDrainWarps * kPart + 8 * kBars + 16;
constexpr int kChunksPerDrain = 8;         // 512 tokens per tensor-core sum
constexpr int kThreads = 32 * (2 + kDrainWarps);
constexpr int kBand = 12;                  // tiles per side of a block of the tile order
static_assert(kSmem <= 227 * 1024, "ring and staged parts must fit an SM's shared memory");

// fp16 x fp16 -> f32, M = 256, N = 256, both operands MN-major.
constexpr uint32_t kIdesc = tc::idesc_f16_f32(256, 256) | (1u << 15) | (1u << 16);

// Descriptor of an MN-major operand written by TMA with 128-byte swizzle:
// 64 contiguous MN elements per 128-byte row, K rows 128 bytes apart,
// 8-row atoms SBO = 1024 bytes apart along K, 64-element MN atoms
// LBO = 8192 bytes (one box) apart along MN.
__device__ __forceinline__ uint64_t sdesc_mn_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(kBox >> 4) << 16;           // leading byte offset: next 64 features
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: next 8 tokens
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

struct SyrkArgs {
    float *H;
    int *status;     // the call's own word
    float scale;
    int d, n;
    int nt;          // tiles per side
    int ntiles;      // nt (nt + 1) / 2
};

// Position t of the tile order, advanced to ever larger t: blocks of kBand x
// kBand tiles on and above the diagonal, column of blocks by column of blocks.
struct TileOrder {
    int nt, bi = 0, bj = 0, base = 0;
    __device__ explicit TileOrder(int n) : nt(n) {}
    __device__ void at(int t, int &ri, int &cj) {
        int nr, nc, cnt;
        for (;;) {
            nr = min(kBand, nt - bi * kBand);
            nc = min(kBand, nt - bj * kBand);
            cnt = bi == bj ? nc * (nc + 1) / 2 : nr * nc;
            if (t < base + cnt) break;
            base += cnt;
            if (bi == bj) {
                bi = 0;
                ++bj;
            } else {
                ++bi;
            }
        }
        int k = t - base, c = 0;
        if (bi == bj) {
            while (k > c) k -= ++c;              // column c holds c + 1 tiles
        } else {
            c = k / nr;
            k %= nr;
        }
        ri = bi * kBand + k;
        cj = bj * kBand + c;
    }
};

// kStalled: for the self-test, the issuer stops after one accumulator.
template <bool kStalled>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    tc_syrk_kernel(const __grid_constant__ CUtensorMap mapX, SyrkArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float *parts = (float *)(smem + kStages * kStage);
    uint64_t *bars = (uint64_t *)(smem + kStages * kStage + kDrainWarps * kPart);
    uint32_t *tmem_slot = (uint32_t *)(bars + kBars);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)tc::cluster_rank();
    const int pair = blockIdx.x / 2, npairs = gridDim.x / 2;
    const int nchunks = (a.n + 63) / 64;
    const int nper = (nchunks + kChunksPerDrain - 1) / kChunksPerDrain;

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kStages + s); };
    auto afull = [&](int b) { return tc::smem_u32(bars + 2 * kStages + b); };
    auto aempty = [&](int b) { return tc::smem_u32(bars + 2 * kStages + 2 + b); };
    const uint32_t closing = tc::smem_u32(bars + 2 * kStages + 4);
    auto tileA = [&](int s) { return tc::smem_u32(smem + s * kStage); };
    auto tileB = [&](int s) { return tc::smem_u32(smem + s * kStage + kTileA); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(full(s), 1);      // the even CTA's: bytes of both CTAs
            tc::mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(afull(b), 1);
            tc::mbar_init(aempty(b), 2 * kDrainWarps);   // the even CTA's: both drains
        }
        tc::mbar_init(closing, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc_pair(tc::smem_u32(tmem_slot), 512);
        tc::tmem_relinquish_pair();
    }
    if (warp == 0 && lane == 0) tc::prefetch_tmap(&mapX);
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- producer
        bool ok = true;
        const uint32_t full0 = tc::map_rank(full(0), 0);
        TileOrder order(a.nt);
        int s = 0, ph = 1, filled = 0;
        for (int it = pair; it < a.ntiles && ok; it += npairs) {
            int ri, cj;
            order.at(it, ri, cj);
            const int ra = ri * 256 + 128 * rank, cb = cj * 256 + 128 * rank;
            for (int c = 0; c < nchunks; ++c) {
                ok = tc::mbar_wait<kPolls>(empty(s), ph);
                if (!ok) break;
                if (tc::elect_one()) {
                    if (rank == 0) tc::mbar_expect_tx(full(s), 2 * (ri == cj ? kTileB : kStage));
                    const uint32_t bar = full0 + 8 * s;
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        if (ri != cj) tc::tma_load_2d_pair(tileA(s) + m * kBox, &mapX, bar, ra + 64 * m, c * 64);
                        tc::tma_load_2d_pair(tileB(s) + m * kBox, &mapX, bar, cb + 64 * m, c * 64);
                    }
                }
                __syncwarp();
                ++filled;
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
        // do not leave before the MMAs have consumed the stages filled here:
        // no copy or commit is in flight afterwards
        for (int n = max(0, filled - kStages); n < filled && ok; ++n)
            ok = tc::mbar_wait<kPolls>(empty(n % kStages), (n / kStages) & 1);
        if (!ok) {
            *abort_flag = 1;
            tc::abandon_ring(full(0), kStages, filled, rank == 0);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer of the pair: an accumulator per 512 tokens
        if (rank == 0) {
            bool ok = true;
            TileOrder order(a.nt);
            const uint64_t a0 = sdesc_mn_sw128(tileA(0)), b0 = sdesc_mn_sw128(tileB(0));
            int s = 0, ph = 0, pc = 0;
            for (int it = pair; it < a.ntiles && ok; it += npairs) {
                if (kStalled && pc > 0) break;
                int ri, cj;
                order.at(it, ri, cj);
                const uint64_t ad0 = ri == cj ? b0 : a0;
                for (int c0 = 0; c0 < nchunks && ok && !(kStalled && pc > 0); c0 += kChunksPerDrain, ++pc) {
                    const int b = pc & 1, c1 = min(nchunks, c0 + kChunksPerDrain);
                    ok = tc::mbar_wait<kPolls>(aempty(b), ((pc >> 1) & 1) ^ 1);
                    for (int c = c0; c < c1 && ok; ++c) {
                        ok = tc::mbar_wait<kPolls>(full(s), ph);
                        if (!ok) break;
                        tc::tc_fence_after();
                        if (tc::elect_one()) {
                            const uint64_t o = (uint64_t)(s * (kStage >> 4));
                            // 16 tokens = two 8-token atoms = 2048 bytes along K
#pragma unroll
                            for (int sub = 0; sub < 4; ++sub)
                                tc::mma_f16_pair(tmem + b * 256, ad0 + o + 128 * sub, b0 + o + 128 * sub, kIdesc,
                                                 c > c0 || sub > 0);
                            tc::mma_commit_pair(empty(s));
                            if (c + 1 == c1) tc::mma_commit_pair(afull(b));
                        }
                        __syncwarp();
                        if (++s == kStages) {
                            s = 0;
                            ph ^= 1;
                        }
                    }
                }
            }
            if (!tc::mma_done_pair<kPolls>(closing, tc::elect_one()) || !ok) *abort_flag = 1;
        }
    } else {
        // ---------------- drain: TMEM -> float32 registers -> H
        const int q = warp & 3, half = (warp - 2) >> 2;   // lane quarter, 128-column half
        const uint32_t released = tc::map_rank(aempty(0), 0);
        float *T = parts + (warp - 2) * (kPart / 4);
        bool ok = true;
        TileOrder order(a.nt);
        int pc = 0;
        for (int it = pair; it < a.ntiles && ok; it += npairs) {
            float acc[128];
#pragma unroll
            for (int e = 0; e < 128; ++e) acc[e] = 0.f;
            int ri, cj;
            order.at(it, ri, cj);
            const int row0 = ri * 256 + 128 * rank + 32 * q, colh = cj * 256 + half * 128;
            for (int per = 0; per < nper; ++per, ++pc) {
                const int b = pc & 1;
                ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(afull(b), (pc >> 1) & 1));
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + b * 256 + half * 128;
#pragma unroll
                for (int cc = 0; cc < 128; cc += 16) {
                    uint32_t v[16];
                    tc::tmem_ld16(base + cc, v);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[cc + e] += __uint_as_float(v[e]);
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_cluster(released + 8 * b);
            }
            if (!ok) break;
            const int u = lane >> 3, v4 = 4 * (lane & 7);
#pragma unroll
            for (int cc = 0; cc < 128; cc += 32) {
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 32; ++e) T[lane * kTld + e] = acc[cc + e];
                __syncwarp();
                const int col0 = colh + cc;
                // the 32 x 32 part lies above, on or below the diagonal as a whole
                if (row0 >= a.d || col0 >= a.d || col0 < row0) continue;
                const bool diag = col0 == row0;
                if (diag) {
                    // H[j][i] takes the element of H[i][j], i < j, as well
#pragma unroll 1
                    for (int j = lane + 1; j < 32; ++j) T[j * kTld + lane] = T[lane * kTld + j];
                    __syncwarp();
                }
                // H[row0 + 4 k + u][col0 + v4 ..] and H[col0 + 4 k + u][row0 + v4 ..]
                float *hp = a.H + (size_t)(row0 + u) * a.d + col0 + v4;
                float *hm = a.H + (size_t)(col0 + u) * a.d + row0 + v4;
                const size_t step = (size_t)4 * a.d;
                // rows 4 k + u of the two parts that exist: 4 k below these
                const int np = col0 + v4 < a.d ? a.d - row0 - u : 0;
                const int nm = row0 + v4 < a.d && !diag ? a.d - col0 - u : 0;
                const float *tp = T + u * kTld + v4, *tm = T + v4 * kTld + u;
#pragma unroll 1
                for (int k0 = 0; k0 < 32; k0 += 16) {        // 16 rows of each part
                    float4 h[4], m[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k0 + 4 * k < np) h[k] = *reinterpret_cast<const float4 *>(hp + k * step);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k0 + 4 * k < nm) m[k] = *reinterpret_cast<const float4 *>(hm + k * step);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k0 + 4 * k < np) {
                            const float *t = tp + 4 * k * kTld;
                            h[k].x = fmaf(a.scale, t[0], h[k].x);
                            h[k].y = fmaf(a.scale, t[1], h[k].y);
                            h[k].z = fmaf(a.scale, t[2], h[k].z);
                            h[k].w = fmaf(a.scale, t[3], h[k].w);
                            *reinterpret_cast<float4 *>(hp + k * step) = h[k];
                        }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k0 + 4 * k < nm) {
                            const float *t = tm + 4 * k;
                            m[k].x = fmaf(a.scale, t[0], m[k].x);
                            m[k].y = fmaf(a.scale, t[kTld], m[k].y);
                            m[k].z = fmaf(a.scale, t[2 * kTld], m[k].z);
                            m[k].w = fmaf(a.scale, t[3 * kTld], m[k].w);
                            *reinterpret_cast<float4 *>(hm + k * step) = m[k];
                        }
                    hp += 4 * step;
                    hm += 4 * step;
                    tp += 16 * kTld;
                    tm += 16;
                }
            }
        }
        if (!ok) *abort_flag = 1;
    }
    // neither CTA leaves while the other may still read its shared memory,
    // signal its barriers or hold TMEM of the pair
    tc::tc_fence_before();
    __syncwarp();
    __syncthreads();
    tc::cluster_sync();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc_pair(tmem, 512);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicOr(a.status, ST_TIMEOUT);
}

}  // namespace

cudaError_t launch_tc_syrk(const CUtensorMap &mapX, float *H, int *status, float scale, int d, int n,
                           cudaStream_t s, bool stalled) {
    const int nt = (d + 255) / 256, ntiles = nt * (nt + 1) / 2;
    const SyrkArgs args{H, status, scale, d, n, nt, ntiles};
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t e = set_max_dynamic_smem((const void *)kernel, kSmem, done);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, dim3(2 * std::min(ntiles, num_sms() / 2)), dim3(kThreads), (size_t)kSmem, s, false,
                        mapX, args);
    };
    static std::atomic<unsigned long long> done[2];
    return stalled ? run(tc_syrk_kernel<true>, done[1]) : run(tc_syrk_kernel<false>, done[0]);
}

}  // namespace jarq

using namespace jarq;

extern "C" jarq_status jarq_accumulate_hessian(const void *X, int n, int d, float scale, float *H,
                                               void *stream) {
    if (n < 0 || d < 8 || d % 8 || d > 65536 || !isfinite(scale)) return JARQ_ERR_ARG;
    if (!H || !on_device(H) || ((uintptr_t)H & 15)) return JARQ_ERR_ARG;
    if (n == 0) return JARQ_OK;
    if (!X || !on_device(X) || ((uintptr_t)X & 15)) return JARQ_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    CUtensorMap map;
    if (make_tmap_f16(&map, X, (uint64_t)n, (uint64_t)d, 64) != cudaSuccess) {
        (void)cudaGetLastError();
        return JARQ_ERR_ARG;
    }
    StatusWord status(st);
    if (!status.ptr()) return JARQ_ERR_CUDA;
    int host = 0;
    cudaError_t e = status.clear();
    if (e == cudaSuccess) {
        ProfScope ps("syrk", st);
        e = launch_tc_syrk(map, H, status.ptr(), scale, d, n, st);
        ps.done();
        count_launches(1);
    }
    if (e == cudaSuccess) e = status.read(&host);
    prof_collect();
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return JARQ_ERR_CUDA;
    }
    return host ? JARQ_ERR_TIMEOUT : JARQ_OK;
}
