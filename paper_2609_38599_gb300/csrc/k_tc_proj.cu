// Target projection P = W H on the tensor cores, exact to double-float
// accuracy, and the quantities derived from it.  For the main target the
// reduced target is R W, so the right-hand side of Eq.
// scale_normal_equations is rhs_j[i] = c_i^T P_j[grp i] with P_j = H w_j
// (App. G "Computational Complexity", the target-projection shortcut), and
// the objective is F_j = w_j^T H w_j - 2 s^T rhs_j + s^T Gram_j s.
//
// Both operands are written in integer digits so that every tensor-core
// partial sum is exact:
//   W[j, k] = 2^(ew(j,h) - 7) sum_{t<4} a_t 2^(-8t),  k in group h, one exponent
//             per (row, group) with max |W[j, grp h]| <= 2^ew;
//   H[k, m] = 2^(E(h,n) - 7) sum_{u<6} b_u 2^(-8u),   the block exponent of
//             block (h, n), n = the group of m,
// with |a_t|, |b_u| <= 128 (exact in bf16).  Four digits hold every float32 W
// entry within 2^7 of its group maximum exactly, six every H entry within
// 2^24 of its block maximum.  For each group h of K the eighteen digit
// products with t + u <= 5 (six MMAs per K step) accumulate in six TMEM
// "levels" l = t + u; a level sums at most 4 x 128 products of 14-bit
// integers per output, an exact integer below 2^23.  The epilogue combines the levels in
// double-float (pairs of float32), applies 2^(ew + E - 14) and adds the
// group's contribution to a double-float accumulator.  The dropped products
// (t + u >= 6) are below 2^-48 of the block scales.
//
// The target projection runs on CTA pairs (cta_group::2): 256 rows x 64
// columns per pair, each CTA loading its 128 rows of the four W planes and
// three of the six H planes, 32 of K at a time (five stages of 44 KB).  An MMA
// takes its B rows half from each CTA, so the planes are split {0, 1, 4 | 2, 3,
// 5}: W digit t meets planes 0..3 in one N = 256 MMA (levels t .. t + 3) and,
// for t < 2, planes 4, 5 in one N = 128 MMA (levels t + 4, t + 5).  The
// products that land on level 6 are not read.
//   warp 0       TMA producer of its CTA's tiles, onto the even CTA's barriers
//   warp 1       TMEM allocation; in the even CTA the MMA issuer
//   warps 2..17  drain: warp w reads TMEM lanes 32 (w % 4) and 16 columns
// The levels (7 x 64 TMEM columns) are single-buffered and handed back in two
// steps: levels 4, 5 first, which is all that the N = 128 MMAs of the next
// group's first tiles need, then levels 0..3.
//
// What bounds it: the MMAs.  20 x 64 columns per K step (two of them for level
// 6) at 4096 x 4096 x 4096 in 1.58 ms are 1.74 PFLOP/s issued, at 4096 x 11008
// x 11008 in 10.7 ms 1.85 PFLOP/s, of a measured 1.94 PFLOP/s.  One CTA per
// 128 x 64 tile, with two stages of 112 KB and a drain that combined the
// levels by two-sums (55 operations an output and group, now 21) before it
// released them, took 2.43 and 16.2 ms.
#include "df.cuh"
#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kWDig = 4, kHDig = 6, kLevels = 6;
// For a row digit t the right-hand digit planes u are consecutive 64-row tiles
// and the levels t + u consecutive 64-column blocks, so one MMA covers up to
// four planes (N = 64 per plane).
__host__ __device__ constexpr uint32_t idesc_n(int n) { return tc::idesc_bf16_f32(128, n); }
// Target projection on CTA pairs
constexpr int kPairA = 128 * 32 * 2;   // one W digit plane, 128 rows x 32 K
constexpr int kPairB = 64 * 32 * 2;    // one H digit plane, 64 rows x 32 K
// Folded projection: all digits of 128 rows and 64 columns, 32 of K at a time
constexpr int kFoldStage = kHDig * (kPairA + kPairB);
constexpr int kFoldStages = 3;
constexpr int kFoldSmem = 1024 + kFoldStages * kFoldStage + 256;
constexpr int kPairStage = kWDig * kPairA + 3 * kPairB;
constexpr int kPairStages = 5;
constexpr int kPairSmem = 1024 + kPairStages * kPairStage + 256;
constexpr int kPairDrain = 16;
constexpr int kPairThreads = 32 * (2 + kPairDrain);
constexpr int kGroupPairs = 4;         // tile pairs per band of the tile order

struct ProjArgs {
    float *Phi, *Plo;    // [p][d] double-float result
    const int *wexp;     // [p][G] row-group exponents of W
    const int *hexp;     // [G][G] block exponents of H ([G] in the diagonal form)
    int *status;
    int p, d, g, G, w_plane, h_plane;   // rows between digit planes in the two maps
};

// (s, e) with s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Levels 0..3 and w = L_4 + L_5 2^-8 of two columns: sum_l L_l 2^(-8 l) as (v, r).
// L_0 is an integer, and every partial sum of the first l levels a multiple of
// 2^(-8 l) (or of a larger power, rounded): an integer multiple of the last place
// of the next term (|L_l| <= 2^23), so that three operations give each sum's
// rounding error exactly (Fast2Sum).
__device__ __forceinline__ void sum_levels(tc::F2 l0, tc::F2 l1, tc::F2 l2, tc::F2 l3, tc::F2 w, tc::F2 &v,
                                           tc::F2 &r) {
    v = l0;
    auto add_level = [&](tc::F2 x, float f) {
        const tc::F2 v2 = tc::f2_fma(x, tc::f2(f), v);
        const tc::F2 e = tc::f2_fma(x, tc::f2(f), tc::f2_sub(v, v2));
        v = v2;
        return e;
    };
    r = add_level(l1, 0x1p-8f);
    r = tc::f2_add(r, add_level(l2, 0x1p-16f));
    r = tc::f2_add(r, add_level(l3, 0x1p-24f));
    r = tc::f2_fma(w, tc::f2(0x1p-32f), r);
}

// Folded projection (launch_ptilde): persistent CTAs over 128 x 64 tiles, the K
// block of the tile's own column group only, and of that the rows of R_i^{-1}
// (upper triangular) that reach the tile's columns.
//   warp 0       TMA producer (three stages of 32 of K, 72 KB each)
//   warp 1       TMEM allocation and MMA issue
//   warps 2..17  drain: warp w reads TMEM lanes 32 (w % 4) and 16 of the tile's
//                64 columns
// What bounds it: memory (the digit planes and the result, 20 bytes an entry)
// and, tile by tile, the MMAs and the drain one after the other: six levels of 64
// columns leave no room for a second accumulator.  4096 x 4096, g = 128: 108 us,
// 175 with the digits of P before it; 465 us on 4096 x 11008, 582 on 14336 x 4096.
// A single stage of 64 of K, all rows of R_i^{-1} and a drain of eight warps that
// combined the levels by two-sums took 325, 920 and 1100 us.
// kStalled: for the self-test, the issuer does nothing.
template <bool kStalled>
__global__ void __launch_bounds__(kPairThreads, 1)
    tc_fold_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapH,
                   ProjArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    constexpr int kStages = kFoldStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(smem + kStages * kFoldStage);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * kStages + 3);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tile it: row tile it / nct, column tile it % nct (in one group: g is a
    // multiple of 64); K chunks of 32 up to the tile's last column
    const int nct = a.d / 64, nitems = ((a.p + 127) / 128) * nct;
    auto chunks_of = [&](int it) { return ((it % nct) * 64 % a.g + 64) / 32; };

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kStages + s); };
    const uint32_t afull = tc::smem_u32(bars + 2 * kStages);
    const uint32_t aempty = tc::smem_u32(bars + 2 * kStages + 1);
    const uint32_t closing = tc::smem_u32(bars + 2 * kStages + 2);
    auto tileA = [&](int s, int t) { return tc::smem_u32(smem + s * kFoldStage + t * kPairA); };
    auto tileB = [&](int s, int u) {
        return tc::smem_u32(smem + s * kFoldStage + kHDig * kPairA + u * kPairB);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(full(s), 1);
            tc::mbar_init(empty(s), 1);
        }
        tc::mbar_init(afull, 1);
        tc::mbar_init(aempty, kPairDrain);
        tc::mbar_init(closing, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
        tc::tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        tc::prefetch_tmap(&mapW);
        tc::prefetch_tmap(&mapH);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- producer
        bool ok = true;
        int s = 0, ph = 1, filled = 0;
        for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
            const int j0 = it / nct * 128, n0 = it % nct * 64, k0 = n0 / a.g * a.g, nc = chunks_of(it);
            for (int c = 0; c < nc; ++c) {
                ok = tc::mbar_wait<kPolls>(empty(s), ph);
                if (!ok) break;
                if (tc::elect_one()) {
                    tc::mbar_expect_tx(full(s), kFoldStage);
                    // the right-hand side holds only the g columns of each group's block
#pragma unroll
                    for (int t = 0; t < kHDig; ++t) {
                        tc::tma_load_2d(tileA(s, t), &mapW, full(s), k0 + c * 32, t * a.w_plane + j0);
                        tc::tma_load_2d(tileB(s, t), &mapH, full(s), c * 32, t * a.h_plane + n0);
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
        // do not leave before the MMAs have consumed the stages filled here
        for (int n = max(0, filled - kStages); n < filled && ok; ++n)
            ok = tc::mbar_wait<kPolls>(empty(n % kStages), (n / kStages) & 1);
        if (!ok) {
            *abort_flag = 1;
            tc::abandon_ring(full(0), kStages, filled, true);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        const uint64_t ad0 = tc::sdesc_sw64(tileA(0, 0)), bd0 = tc::sdesc_sw64(tileB(0, 0));
        bool ok = true;
        int s = 0, ph = 0, n = 0;
        for (int it = blockIdx.x; it < (kStalled ? 0 : nitems) && ok; it += gridDim.x, ++n) {
            const int nc = chunks_of(it);
            for (int c = 0; c < nc; ++c) {
                ok = tc::mbar_wait<kPolls>(full(s), ph);
                if (c == 0) ok = tc::mbar_wait<kPolls>(aempty, (n & 1) ^ 1) && ok;
                if (!ok) break;
                tc::tc_fence_after();
                if (tc::elect_one()) {
                    const uint64_t o = (uint64_t)(s * (kFoldStage >> 4));
#pragma unroll
                    for (int k = 0; k < 4; k += 2)
#pragma unroll
                        for (int t = 0; t < kHDig; ++t)
                            // the products of row digit t with digits u < kLevels - t,
                            // in runs of at most four planes; t = 0 opens every level
#pragma unroll
                            for (int u0 = 0; u0 < kLevels - t; u0 += 4)
                                tc::mma_bf16(tmem + (t + u0) * 64, ad0 + o + t * (kPairA >> 4) + k,
                                             bd0 + o + u0 * (kPairB >> 4) + k,
                                             idesc_n(64 * min(4, kLevels - t - u0)), (c | k | t) != 0);
                    tc::mma_commit(empty(s));
                    if (c + 1 == nc) tc::mma_commit(afull);
                }
                __syncwarp();
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
        if (!tc::mma_done<kPolls>(closing, tc::elect_one()) || !ok) *abort_flag = 1;
    } else {
        // ---------------- drain: levels -> double-float
        const int q = warp & 3, cq = (warp - 2) >> 2;    // lane quarter, 16-column quarter
        const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + cq * 16;
        bool ok = true;
        int n = 0;
        for (int it = blockIdx.x; it < nitems; it += gridDim.x, ++n) {
            const int row = it / nct * 128 + 32 * q + lane, n0 = it % nct * 64, hb = n0 / a.g;
            const int ex = a.wexp[(size_t)min(row, a.p - 1) * a.G + hb] + a.hexp[hb] - 14;
            const tc::F2 scale = tc::f2(ldexpf(1.0f, ex));
            ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(afull, n & 1));
            if (!ok) break;
            tc::tc_fence_after();
            tc::F2 w[8];     // L_4 + L_5 2^-8
            {
                uint32_t x4[16], x5[16];
                tc::tmem_ld16(base + 4 * 64, x4);
                tc::tmem_ld16(base + 5 * 64, x5);
                tc::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    w[e] = tc::f2_fma(tc::f2(__uint_as_float(x5[2 * e]), __uint_as_float(x5[2 * e + 1])),
                                      tc::f2(0x1p-8f),
                                      tc::f2(__uint_as_float(x4[2 * e]), __uint_as_float(x4[2 * e + 1])));
            }
            const size_t o = (size_t)row * a.d + n0 + cq * 16;
#pragma unroll
            for (int cc = 0; cc < 16; cc += 8) {
                uint32_t x[4][8];
#pragma unroll
                for (int l = 0; l < 4; ++l) tc::tmem_ld8(base + l * 64 + cc, x[l]);
                tc::tmem_wait_ld();
                if (cc == 8) {
                    // every level is in registers: hand the columns back
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(aempty);
                }
                float xh[8], xl[8];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    auto lv = [&](int l) {
                        return tc::f2(__uint_as_float(x[l][e]), __uint_as_float(x[l][e + 1]));
                    };
                    tc::F2 v, r;
                    sum_levels(lv(0), lv(1), lv(2), lv(3), w[(cc + e) / 2], v, r);
                    // (v + r) 2^ex, normalised
                    float v0, v1, r0, r1;
                    tc::f2_get(tc::f2_mul(v, scale), v0, v1);
                    tc::f2_get(tc::f2_mul(r, scale), r0, r1);
                    two_sum(v0, r0, xh[e], xl[e]);
                    two_sum(v1, r1, xh[e + 1], xl[e + 1]);
                }
                if (row < a.p)
#pragma unroll
                    for (int e = 0; e < 8; e += 4) {
                        *reinterpret_cast<float4 *>(a.Phi + o + cc + e) =
                            make_float4(xh[e], xh[e + 1], xh[e + 2], xh[e + 3]);
                        *reinterpret_cast<float4 *>(a.Plo + o + cc + e) =
                            make_float4(xl[e], xl[e + 1], xl[e + 2], xl[e + 3]);
                    }
            }
        }
        if (!ok) *abort_flag = 1;
    }
    tc::tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicOr(a.status, ST_TIMEOUT);
}

// kStalled: for the self-test, the issuer stops after one group.
template <bool kStalled>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    tc_proj_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapH,
                   ProjArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(smem + kPairStages * kPairStage);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * kPairStages + 4);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)tc::cluster_rank();
    // tiles in bands: kGroupPairs pairs of row tiles sweep all column tiles
    const int npairs = gridDim.x / 2;
    const int lin = blockIdx.y * npairs + blockIdx.x / 2;
    const int band = lin / (kGroupPairs * gridDim.y), in_band = lin % (kGroupPairs * gridDim.y);
    const int in_rows = min(kGroupPairs, npairs - band * kGroupPairs);
    const int j0 = (band * kGroupPairs + in_band % in_rows) * 256 + 128 * rank;
    const int n0 = (in_band / in_rows) * 64;
    const int nsub = a.g / 32;              // 32-wide K chunks per group
    const int nchunks = a.G * nsub;

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kPairStages + s); };
    const uint32_t afull = tc::smem_u32(bars + 2 * kPairStages);
    const uint32_t afree = tc::smem_u32(bars + 2 * kPairStages + 1);   // [2]: levels 4, 5; 0..3
    const uint32_t closing = tc::smem_u32(bars + 2 * kPairStages + 3);
    auto tileA = [&](int s, int t) { return tc::smem_u32(smem + s * kPairStage + t * kPairA); };
    auto tileB = [&](int s, int u) {
        return tc::smem_u32(smem + s * kPairStage + kWDig * kPairA + u * kPairB);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPairStages; ++s) {
            tc::mbar_init(full(s), 1);      // the even CTA's: bytes of both CTAs
            tc::mbar_init(empty(s), 1);
        }
        tc::mbar_init(afull, 1);
        tc::mbar_init(afree, 2 * kPairDrain);       // the even CTA's: both drains
        tc::mbar_init(afree + 8, 2 * kPairDrain);
        tc::mbar_init(closing, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc_pair(tc::smem_u32(tmem_slot), 512);
        tc::tmem_relinquish_pair();
    }
    if (warp == 0 && lane == 0) {
        tc::prefetch_tmap(&mapW);
        tc::prefetch_tmap(&mapH);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- producer
        bool ok = true;
        const uint32_t full0 = tc::map_rank(full(0), 0);
        int s = 0, ph = 1, c = 0;
        for (; c < nchunks; ++c) {
            ok = tc::mbar_wait<kPolls>(empty(s), ph);
            if (!ok) break;
            if (tc::elect_one()) {
                if (rank == 0) tc::mbar_expect_tx(full(s), 2 * kPairStage);
                const uint32_t bar = full0 + 8 * s;
#pragma unroll
                for (int t = 0; t < kWDig; ++t)
                    tc::tma_load_2d_pair(tileA(s, t), &mapW, bar, c * 32, t * a.w_plane + j0);
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const int plane = u < 2 ? 2 * rank + u : 4 + rank;
                    tc::tma_load_2d_pair(tileB(s, u), &mapH, bar, c * 32, plane * a.h_plane + n0);
                }
            }
            __syncwarp();
            if (++s == kPairStages) {
                s = 0;
                ph ^= 1;
            }
        }
        // do not leave before the MMAs have consumed the stages filled here:
        // no copy or commit is in flight afterwards
        for (int n = max(0, nchunks - kPairStages); n < nchunks && ok; ++n)
            ok = tc::mbar_wait<kPolls>(empty(n % kPairStages), (n / kPairStages) & 1);
        if (!ok) {
            *abort_flag = 1;
            tc::abandon_ring(full(0), kPairStages, c, rank == 0);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer of the pair
        if (rank == 0) {
            constexpr uint32_t id256 = tc::idesc_bf16_f32(256, 256), id128 = tc::idesc_bf16_f32(256, 128);
            const uint64_t ad0 = tc::sdesc_sw64(tileA(0, 0)), bd0 = tc::sdesc_sw64(tileB(0, 0));
            constexpr uint64_t kPl = kPairA >> 4, kHi = (2 * kPairB) >> 4;   // next W plane; planes 4, 5
            bool ok = true;
            int s = 0, ph = 0;
            const int ngroups = kStalled ? 1 : a.G;
            for (int sg = 0; sg < ngroups && ok; ++sg) {
                for (int c = 0; c < nsub; ++c) {
                    ok = tc::mbar_wait<kPolls>(full(s), ph);
                    if (c == 0) ok = tc::mbar_wait<kPolls>(afree, (sg & 1) ^ 1) && ok;
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint64_t ad = ad0 + (uint64_t)(s * (kPairStage >> 4));
                    const uint64_t bd = bd0 + (uint64_t)(s * (kPairStage >> 4));
                    if (tc::elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; k += 2) {
                            // planes 4, 5: levels 4, 5 (opened by the first) and 5, 6
                            tc::mma_f16_pair(tmem + 4 * 64, ad + k, bd + kHi + k, id128, (c | k) != 0);
                            tc::mma_f16_pair(tmem + 5 * 64, ad + kPl + k, bd + kHi + k, id128, 1);
                        }
                    }
                    __syncwarp();
                    if (c == 0) {
                        ok = tc::mbar_wait<kPolls>(afree + 8, (sg & 1) ^ 1);
                        if (!ok) break;
                        tc::tc_fence_after();
                    }
                    if (tc::elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; k += 2)
#pragma unroll
                            for (int t = 0; t < kWDig; ++t)     // planes 0..3: levels t .. t + 3
                                tc::mma_f16_pair(tmem + t * 64, ad + t * kPl + k, bd + k, id256,
                                                 t > 0 || (c | k) != 0);
                        tc::mma_commit_pair(empty(s));
                        if (c + 1 == nsub) tc::mma_commit_pair(afull);
                    }
                    __syncwarp();
                    if (++s == kPairStages) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            if (!tc::mma_done_pair<kPolls>(closing, tc::elect_one()) || !ok) *abort_flag = 1;
        }
    } else {
        // ---------------- drain: levels -> double-float per group -> accumulator
        const int q = warp & 3, cq = (warp - 2) >> 2;    // lane quarter, 16-column quarter
        const int hb = n0 / a.g;
        const int row = j0 + 32 * q + lane;
        tc::F2 hi[8], lo[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) hi[e] = lo[e] = tc::f2(0.f);
        bool ok = true;
        const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + cq * 16;
        const uint32_t freed = tc::map_rank(afree, 0);
        // exponents of the next group, loaded one group ahead
        const int *wrow = a.wexp + (size_t)min(row, a.p - 1) * a.G;
        int e_next = wrow[0] + a.hexp[hb];
        const tc::F2 c8 = tc::f2(0x1p-8f);
        for (int sg = 0; sg < a.G; ++sg) {
            const int ex = e_next - 14;
            if (sg + 1 < a.G) e_next = wrow[sg + 1] + a.hexp[(sg + 1) * a.G + hb];
            // 2^ex, from its bits while it is a normal number
            const tc::F2 scale = tc::f2((unsigned)(ex + 126) <= 252u ? __int_as_float((ex + 127) << 23)
                                                                     : ldexpf(1.0f, ex));
            ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(afull, sg & 1));
            if (!ok) break;
            tc::tc_fence_after();
            tc::F2 w[8];     // L_4 + L_5 2^-8
            {
                uint32_t x4[16], x5[16];
                tc::tmem_ld16(base + 4 * 64, x4);
                tc::tmem_ld16(base + 5 * 64, x5);
                tc::tmem_wait_ld();
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_cluster(freed);
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    w[e] = tc::f2_fma(tc::f2(__uint_as_float(x5[2 * e]), __uint_as_float(x5[2 * e + 1])), c8,
                                      tc::f2(__uint_as_float(x4[2 * e]), __uint_as_float(x4[2 * e + 1])));
            }
#pragma unroll
            for (int cc = 0; cc < 16; cc += 8) {
                uint32_t x0[8], x1[8], x2[8], x3[8];
                tc::tmem_ld8(base + 0 * 64 + cc, x0);
                tc::tmem_ld8(base + 1 * 64 + cc, x1);
                tc::tmem_ld8(base + 2 * 64 + cc, x2);
                tc::tmem_ld8(base + 3 * 64 + cc, x3);
                tc::tmem_wait_ld();
                if (cc == 8) {
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_cluster(freed + 8);
                }
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    auto pair = [&](const uint32_t (&x)[8]) {
                        return tc::f2(__uint_as_float(x[e]), __uint_as_float(x[e + 1]));
                    };
                    tc::F2 v, r;
                    sum_levels(pair(x0), pair(x1), pair(x2), pair(x3), w[(cc + e) / 2], v, r);
                    // (v + r) 2^ex (exact products) added to the accumulator
                    tc::F2 &H = hi[(cc + e) / 2], &L = lo[(cc + e) / 2];
                    const tc::F2 sm = tc::f2_fma(v, scale, H);
                    const tc::F2 nb = tc::f2_sub(H, sm);
                    const tc::F2 er = tc::f2_add(tc::f2_sub(H, tc::f2_add(sm, nb)), tc::f2_fma(v, scale, nb));
                    H = sm;
                    L = tc::f2_add(L, tc::f2_fma(r, scale, er));
                }
            }
        }
        if (!ok) *abort_flag = 1;
        if (ok && row < a.p) {
            const size_t o = (size_t)row * a.d + n0 + cq * 16;
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                float x[4], y[4];
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    float h2[2], l2[2];
                    tc::f2_get(hi[(e + k) / 2], h2[0], h2[1]);
                    tc::f2_get(lo[(e + k) / 2], l2[0], l2[1]);
                    two_sum(h2[0], l2[0], x[k], y[k]);
                    two_sum(h2[1], l2[1], x[k + 1], y[k + 1]);
                }
                *reinterpret_cast<float4 *>(a.Phi + o + e) = make_float4(x[0], x[1], x[2], x[3]);
                *reinterpret_cast<float4 *>(a.Plo + o + e) = make_float4(y[0], y[1], y[2], y[3]);
            }
        }
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

// NT consecutive floats / bf16 of one lane.
template <int NT>
__device__ __forceinline__ void load_nt(const float *p, float (&v)[NT]) {
    if constexpr (NT == 4) {
        const float4 a = *reinterpret_cast<const float4 *>(p);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    } else {
        const float2 a = *reinterpret_cast<const float2 *>(p);
        v[0] = a.x; v[1] = a.y;
    }
}
template <int NT>
__device__ __forceinline__ void store_nt(__nv_bfloat16 *p, const float (&v)[NT]) {
    __align__(8) __nv_bfloat16 q[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) q[k] = __float2bfloat16_rn(v[k]);
    if constexpr (NT == 4)
        *reinterpret_cast<uint2 *>(p) = *reinterpret_cast<const uint2 *>(q);
    else
        *reinterpret_cast<uint32_t *>(p) = *reinterpret_cast<const uint32_t *>(q);
}

// Digits of W per (row, group): x = W 2^(7 - ew) in [-128, 128] with
// max |W[j, grp h]| <= 2^ew; a_0 = rint(x), a_t = rint(256 * remainder).
// One warp per (row, group), lane owns NT = g/32 consecutive entries, loaded as
// one vector if W is 16-byte aligned (`vec`).
template <int NT>
__global__ void slice_rows_kernel(const float *__restrict__ W, __nv_bfloat16 *__restrict__ planes,
                                  int *__restrict__ wexp, int p, int d, int d_pad, int p_pad, bool vec) {
    constexpr int g = 32 * NT;
    const int G = d / g;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= (long long)p * G) return;
    const int j = (int)(warp / G), h = (int)(warp % G);
    float x[NT];
    const float *src = W + (size_t)j * d + (size_t)h * g + NT * lane;
    if (vec) {
        load_nt<NT>(src, x);
    } else {
#pragma unroll
        for (int k = 0; k < NT; ++k) x[k] = src[k];
    }
    float mx = 0.f;
#pragma unroll
    for (int k = 0; k < NT; ++k) mx = fmaxf(mx, fabsf(x[k]));
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = 0;
    if (mx > 0.f) frexpf(mx, &e);
    if (lane == 0) wexp[(size_t)j * G + h] = e;
    const size_t plane = (size_t)p_pad * d_pad;
    const size_t off = (size_t)j * d_pad + (size_t)h * g + NT * lane;
#pragma unroll
    for (int k = 0; k < NT; ++k) x[k] = ldexpf(x[k], 7 - e);
#pragma unroll
    for (int t = 0; t < kWDig; ++t) {
        float dg[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            dg[k] = rintf(x[k]);
            x[k] = (x[k] - dg[k]) * 256.f;
        }
        store_nt<NT>(planes + t * plane + off, dg);
    }
}

// Exact product c * (ph + pl) added to the double-float (sh, sl): c is a small
// integer, so c * ph splits exactly by one fma.
__device__ __forceinline__ void df_axpy(float c, float ph, float pl, float &sh, float &sl) {
    const float m = c * ph;
    const float me = fmaf(c, ph, -m);
    float s2, e2;
    two_sum(sh, m, s2, e2);
    sh = s2;
    sl += e2 + fmaf(c, pl, me);
}

__device__ __forceinline__ void df_warp_sum(float &sh, float &sl) {
    for (int o = 16; o; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, sh, o);
        const float ol = __shfl_xor_sync(0xffffffffu, sl, o);
        float s2, e2;
        two_sum(sh, oh, s2, e2);
        sh = s2;
        sl += e2 + ol;
    }
}

// rhs_j[i] = sum_{l in grp i} (q_l - z_i) P_j[l], one warp per row, lane owns
// NT = g/32 consecutive entries of every group; NB groups are loaded and reduced
// together.  What bounds it: memory (9 bytes an entry), at the loads that a row's
// warp keeps in flight.  4096 x 4096: 37 us for g = 128 (NB = 8; 39 with 4), 47 us
// for g = 64 (NB = 2; 52 and 57 with 4 and 8); 14336 x 4096 97 us, 4096 x 11008 86
// us.  One group at a time: 42, 68, 102 and 98 us.
constexpr int kRhsThreads = 64;

template <int NT, int NB>
__global__ void __launch_bounds__(kRhsThreads) rhs_kernel(const uint8_t *__restrict__ Q,
                                                          const int32_t *__restrict__ Z,
                                                          const float *__restrict__ Phi,
                                                          const float *__restrict__ Plo,
                                                          const int *__restrict__ active,
                                                          double *__restrict__ rhs, int p, int d) {
    constexpr int g = 32 * NT;
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    const int G = d / g;
    const int j = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= p || (active && !active[j])) return;   // warp-uniform
    const size_t off = (size_t)j * d + NT * lane;
    const int32_t *zj = Z + (size_t)j * G;
#pragma unroll 1
    for (int i = 0; i < G; i += NB) {
        float ph[NB][NT], pl[NB][NT];
        uint32_t q[NB];
        int z[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int iu = min(i + u, G - 1);       // past the end: the last group again, not stored
            const size_t o = off + (size_t)iu * g;
            if constexpr (NT == 4) {
                const float4 a4 = __ldg(reinterpret_cast<const float4 *>(Phi + o));
                const float4 b4 = __ldg(reinterpret_cast<const float4 *>(Plo + o));
                q[u] = __ldg(reinterpret_cast<const uint32_t *>(Q + o));
                ph[u][0] = a4.x; ph[u][1] = a4.y; ph[u][2] = a4.z; ph[u][3] = a4.w;
                pl[u][0] = b4.x; pl[u][1] = b4.y; pl[u][2] = b4.z; pl[u][3] = b4.w;
            } else {
                const float2 a2 = __ldg(reinterpret_cast<const float2 *>(Phi + o));
                const float2 b2 = __ldg(reinterpret_cast<const float2 *>(Plo + o));
                q[u] = __ldg(reinterpret_cast<const uint16_t *>(Q + o));
                ph[u][0] = a2.x; ph[u][1] = a2.y;
                pl[u][0] = b2.x; pl[u][1] = b2.y;
            }
            z[u] = __ldg(zj + iu);
        }
        float sh[NB], sl[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            sh[u] = sl[u] = 0.f;
            const float zf = (float)z[u];
#pragma unroll
            for (int t = 0; t < NT; ++t)
                df_axpy((float)((q[u] >> (8 * t)) & 0xFFu) - zf, ph[u][t], pl[u][t], sh[u], sl[u]);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) df_warp_sum(sh[u], sl[u]);
        // every lane holds the sums: lane u stores group i + u
        float h = sh[0], l = sl[0];
#pragma unroll
        for (int u = 1; u < NB; ++u) {
            h = lane == u ? sh[u] : h;
            l = lane == u ? sl[u] : l;
        }
        if (lane < NB && i + lane < G) rhs[(size_t)j * G + i + lane] = (double)h + (double)l;
    }
}

// wHw_j = sum_k W[j,k] P[j,k] with P = Phi + Plo, double-float per lane, four
// warps (one block) per row.  Bound by memory (12 bytes an entry): 41 us on
// 4096 x 4096, 95 us on 4096 x 11008; with one warp per row 51 and 116 us.
constexpr int kWhwWarps = 4;

__global__ void __launch_bounds__(32 * kWhwWarps) whw_kernel(const float *__restrict__ W,
                                                             const float *__restrict__ Phi,
                                                             const float *__restrict__ Plo,
                                                             double *__restrict__ out, int d) {
    __shared__ float ph_s[kWhwWarps], pl_s[kWhwWarps];
    const int j = blockIdx.x, lane = threadIdx.x & 31;
    const size_t off = (size_t)j * d;
    float sh = 0.f, sl = 0.f;
#pragma unroll 8
    for (int k = threadIdx.x; k < d; k += 32 * kWhwWarps) {
        const float w = W[off + k], ph = Phi[off + k], pl = Plo[off + k];
        const float m = w * ph;
        const float me = fmaf(w, ph, -m);
        float s2, e2;
        two_sum(sh, m, s2, e2);
        sh = s2;
        sl += e2 + fmaf(w, pl, me);
    }
    df_warp_sum(sh, sl);
    if (lane == 0) {
        ph_s[threadIdx.x >> 5] = sh;
        pl_s[threadIdx.x >> 5] = sl;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < kWhwWarps; ++w) v += (double)ph_s[w] + (double)pl_s[w];
        out[j] = v;
    }
}

// Propagation-corrected target (App. "Propagation-Corrected Targets and
// QEP", Eqs. mu-target, w-corr).  With H = X~^T X~ + nu^2 I and K = X~^T X,
// the projection of the corrected weights needs no inverse of H:
//   H w_corr = A^T y(mu) = mu H w + (1 - mu) (K w + nu^2 w),
// and the target energy that replaces w^T H w in the objective is
//   ||y(mu)||^2 = (1-mu)^2 w^T XX w + 2 mu (1-mu) w^T K w
//                 + mu^2 (w^T H w - nu^2 w^T w) + nu^2 w^T w.
// On entry P = Phi + Plo holds H w, PK = Khi + Klo holds K w (rows of the
// target projection with K in place of H), wHw[j] = w^T H w and
// wXXw[j] = w^T XX w; on exit P holds H w_corr and wHw[j] ||y_j(mu)||^2.
// Four warps (one block) per row, float64 arithmetic: seven operations an entry,
// which bound the kernel (1/64 of the float32 rate); the conversions in and the
// split out are integer operations.  429 us on 4096 x 4096; with conversions (eight
// more operations on the float64 pipe) and one warp per row 599 us.
__global__ void __launch_bounds__(32 * kWhwWarps)
    mu_combine_kernel(float *__restrict__ Phi, float *__restrict__ Plo, const float *__restrict__ Khi,
                      const float *__restrict__ Klo, const float *__restrict__ W,
                      const double *__restrict__ wXXw, double *__restrict__ wHw, int d, double mu, double nu2) {
    __shared__ double part[2][kWhwWarps];
    const int j = blockIdx.x, lane = threadIdx.x & 31;
    const size_t off = (size_t)j * d;
    double wKw = 0.0, ww = 0.0;
#pragma unroll 2
    for (int k = threadIdx.x; k < d; k += 32 * kWhwWarps) {
        const double P = widen(Phi[off + k]) + widen(Plo[off + k]);
        const double PK = widen(Khi[off + k]) + widen(Klo[off + k]);
        const double w = widen(W[off + k]);
        const double r = mu * P + (1.0 - mu) * fma(nu2, w, PK);
        const DF v = split_double(r);
        Phi[off + k] = v.h;
        Plo[off + k] = v.l;
        wKw = fma(w, PK, wKw);
        ww = fma(w, w, ww);
    }
    for (int o = 16; o; o >>= 1) {
        wKw += __shfl_xor_sync(0xffffffffu, wKw, o);
        ww += __shfl_xor_sync(0xffffffffu, ww, o);
    }
    if (lane == 0) {
        part[0][threadIdx.x >> 5] = wKw;
        part[1][threadIdx.x >> 5] = ww;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        wKw = ww = 0.0;
        for (int w = 0; w < kWhwWarps; ++w) {
            wKw += part[0][w];
            ww += part[1][w];
        }
        const double a = 1.0 - mu;
        wHw[j] = a * a * wXXw[j] + 2.0 * mu * a * wKw + mu * mu * (wHw[j] - nu2 * ww) + nu2 * ww;
    }
}

// Digits of the double-float P for the folded projection: per (row, group)
// the exponent e with max |P| < 2^e, and six balanced base-256 digits of
// P 2^(7-e) (|digit| <= 128, exact in bf16), taken from the float pair
// (xh, xl) = (Phi, Plo) 2^(7-e) with exact float operations: the digit is
// rint(xh), and the remainder (xh - digit) + xl is renormalised by an exact
// two-sum before the next digit.  Six digits hold P to 2^-48 of its group
// maximum (the pair itself carries about 48 bits).
template <int NT>
__global__ void slice_df_rows_kernel(const float *__restrict__ Phi, const float *__restrict__ Plo,
                                     __nv_bfloat16 *__restrict__ planes, int *__restrict__ pexp,
                                     int p, int d, int d_pad, int p_pad) {
    constexpr int g = 32 * NT;
    const int G = d / g;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= (long long)p * G) return;
    const int j = (int)(warp / G), h = (int)(warp % G);
    const size_t src = (size_t)j * d + (size_t)h * g + NT * lane;
    float xh[NT], xl[NT];
    load_nt<NT>(Phi + src, xh);
    load_nt<NT>(Plo + src, xl);
    float mx = 0.f;
#pragma unroll
    for (int k = 0; k < NT; ++k) mx = fmaxf(mx, fabsf(xh[k]));
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = 0;
    if (mx > 0.f) frexpf(mx, &e);
    if (lane == 0) pexp[(size_t)j * G + h] = e;
    const size_t plane = (size_t)p_pad * d_pad;
    const size_t off = (size_t)j * d_pad + (size_t)h * g + NT * lane;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        xh[k] = ldexpf(xh[k], 7 - e);
        xl[k] = ldexpf(xl[k], 7 - e);
    }
#pragma unroll
    for (int t = 0; t < kHDig; ++t) {
        float dg[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            dg[k] = rintf(xh[k]);
            float s2, e2;
            two_sum(xh[k] - dg[k], xl[k], s2, e2);
            xh[k] = s2 * 256.f;
            xl[k] = e2 * 256.f;
        }
        store_nt<NT>(planes + t * plane + off, dg);
    }
}

// Digits of the group inverses for the folded projection (once per prepared
// Hessian): plane u, row i g + a, column b holds digit u of R_i^{-1}[b][a]
// (zero below the diagonal), so that the 64 x 64 tiles of the projection
// kernel read the transposed block; exponent E_i with max |R_i^{-1}| < 2^E_i,
// six balanced base-256 digits of R_i^{-1} 2^(7-E_i) in float64.  Bound by float64
// (some thirty operations an entry): four blocks a group, each of which finds
// the maximum for itself, and no arithmetic for the zeros.  32 groups of 128:
// 51 us; one block a group took 152 us.
constexpr int kRinvParts = 4;

__global__ void slice_rinv_kernel(const double *__restrict__ Rinv, __nv_bfloat16 *__restrict__ rdig,
                                  int *__restrict__ rexp, int d, int g) {
    __shared__ double red[32];
    const int i = blockIdx.x;
    const double *Ri = Rinv + (size_t)i * g * g;
    double mx = 0.0;
    for (int idx = threadIdx.x; idx < g * g; idx += blockDim.x) mx = fmax(mx, fabs(Ri[idx]));
    for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x < 32) {
        mx = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (threadIdx.x == 0) red[0] = mx;
    }
    __syncthreads();
    mx = red[0];
    int E = 0;
    if (mx > 0.0) frexp(mx, &E);
    if (threadIdx.x == 0 && blockIdx.y == 0) rexp[i] = E;
    const size_t plane = (size_t)d * g;
    for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < g * g; idx += gridDim.y * blockDim.x) {
        const int a = idx / g, b = idx % g;
        const size_t off = ((size_t)i * g + a) * g + b;
        if (b > a) {
#pragma unroll
            for (int u = 0; u < kHDig; ++u) rdig[u * plane + off] = __float2bfloat16_rn(0.f);
            continue;
        }
        double x = ldexp(Ri[(size_t)b * g + a], 7 - E);
#pragma unroll
        for (int u = 0; u < kHDig; ++u) {
            const double dg = rint(x);
            rdig[u * plane + off] = __float2bfloat16_rn((float)dg);
            x = (x - dg) * 256.0;
        }
    }
}

}  // namespace

cudaError_t launch_slice_rinv(const double *Rinv, __nv_bfloat16 *rdig, int *rexp, int d, int g,
                              cudaStream_t s) {
    slice_rinv_kernel<<<dim3(d / g, kRinvParts), 256, 0, s>>>(Rinv, rdig, rexp, d, g);
    return cudaGetLastError();
}

// Pt = the folded projection, Pt[j, i g + a] = sum_{b <= a} R_i^{-1}[b][a] P[j, i g + b]:
// the six digit planes of P (into the row-digit workspace) and the
// block-diagonal product with the digits of R_i^{-1} on the tensor cores.
cudaError_t launch_ptilde(const CUtensorMap &mapPd, const CUtensorMap &mapR, const float *Phi,
                          const float *Plo, __nv_bfloat16 *pdig, int *pexp, const int *rexp,
                          float *out_hi, float *out_lo, int p, int p_pad, int d, int d_pad, int g,
                          int *status, cudaStream_t s, bool stalled) {
    const long long warps = (long long)p * (d / g);
    const unsigned blocks = (unsigned)((warps * 32 + 255) / 256);
    if (g == 128)
        slice_df_rows_kernel<4><<<blocks, 256, 0, s>>>(Phi, Plo, pdig, pexp, p, d, d_pad, p_pad);
    else
        slice_df_rows_kernel<2><<<blocks, 256, 0, s>>>(Phi, Plo, pdig, pexp, p, d, d_pad, p_pad);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ProjArgs a{out_hi, out_lo, pexp, rexp, status, p, d, g, d / g, p_pad, d};
    // persistent: one CTA per SM over the (p_pad / 128) x (d / 64) tiles
    (void)d_pad;
    const int items = ((p + 127) / 128) * (d / 64);
    const int ctas = items < num_sms() ? items : num_sms();
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t r = set_max_dynamic_smem((const void *)kernel, kFoldSmem, done);
        if (r != cudaSuccess) return r;
        return launch_k(kernel, dim3(ctas), dim3(kPairThreads), (size_t)kFoldSmem, s, false, mapPd, mapR, a);
    };
    static std::atomic<unsigned long long> done[2];
    return stalled ? run(tc_fold_kernel<true>, done[1]) : run(tc_fold_kernel<false>, done[0]);
}

cudaError_t launch_slice_rows(const float *W, __nv_bfloat16 *planes, int *wexp, int p, int d,
                              int d_pad, int p_pad, int g, cudaStream_t s) {
    const long long warps = (long long)p * (d / g);
    const unsigned blocks = (unsigned)((warps * 32 + 255) / 256);
    const bool vec = ((uintptr_t)W & 15) == 0;
    if (g == 128)
        slice_rows_kernel<4><<<blocks, 256, 0, s>>>(W, planes, wexp, p, d, d_pad, p_pad, vec);
    else
        slice_rows_kernel<2><<<blocks, 256, 0, s>>>(W, planes, wexp, p, d, d_pad, p_pad, vec);
    return cudaGetLastError();
}

cudaError_t launch_tc_proj(const CUtensorMap &mapW, const CUtensorMap &mapH, float *Phi,
                           float *Plo, const int *wexp, const int *hexp, int p, int p_pad, int d,
                           int d_pad, int g, int *status, cudaStream_t s, bool stalled) {
    ProjArgs a{Phi, Plo, wexp, hexp, status, p, d, g, d / g, p_pad, d_pad};
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t e = set_max_dynamic_smem((const void *)kernel, kPairSmem, done);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, dim3((p + 255) / 256 * 2, d / 64), dim3(kPairThreads), (size_t)kPairSmem, s, false,
                        mapW, mapH, a);
    };
    static std::atomic<unsigned long long> done[2];
    return stalled ? run(tc_proj_kernel<true>, done[1]) : run(tc_proj_kernel<false>, done[0]);
}

cudaError_t launch_whw(const float *W, const float *Phi, const float *Plo, double *out, int p,
                       int d, cudaStream_t s) {
    whw_kernel<<<p, 32 * kWhwWarps, 0, s>>>(W, Phi, Plo, out, d);
    return cudaGetLastError();
}

cudaError_t launch_mu_combine(float *Phi, float *Plo, const float *Khi, const float *Klo,
                              const float *W, const double *wXXw, double *wHw, int p, int d,
                              double mu, double nu2, cudaStream_t s) {
    mu_combine_kernel<<<p, 32 * kWhwWarps, 0, s>>>(Phi, Plo, Khi, Klo, W, wXXw, wHw, d, mu, nu2);
    return cudaGetLastError();
}

cudaError_t launch_rhs(const uint8_t *Q, const int32_t *Z, const float *Phi, const float *Plo,
                       const int *active, double *rhs, int p, int d, int g, cudaStream_t s,
                       bool pdl) {
    const unsigned blocks = (unsigned)(((long long)p * 32 + kRhsThreads - 1) / kRhsThreads);
    if (g == 128)
        return launch_k(rhs_kernel<4, 8>, dim3(blocks), dim3(kRhsThreads), 0, s, pdl, Q, Z, Phi, Plo, active, rhs,
                        p, d);
    if (g == 64)
        return launch_k(rhs_kernel<2, 2>, dim3(blocks), dim3(kRhsThreads), 0, s, pdl, Q, Z, Phi, Plo, active, rhs,
                        p, d);
    return cudaErrorInvalidValue;
}

}  // namespace jarq
