// Babai targets of one Gauss-Seidel phase on the tensor cores, exact to
// double-float accuracy (Sec. 3.3.2, Eqs. conditional_residual and
// babai_update).
//
// The target of group i is y = R_i^{-T} (H r)_i / s_i with r = w - D_s c.
// With the folded rows Ht_i = R_i^{-T} H[grp i, :] and Pt = R^{-T}-folded
// target projection (Pt_i = R_i^{-T} (H w)_i),
//     s_i y = Pt_i - sum_h s_h Ht_ih c_h,
// where c = q - z are the current codes (new for groups before i, previous
// for the rest).  This kernel forms T_i = sum_h s_h Ht_ih c_h; the Babai
// kernel subtracts it from Pt_i.  The codes are exact in fp16, and Ht is
// held in four fp16 digit planes base 2^10 per g x g block (block exponent
// E_ih, |digit| <= 512), so for each group h of K the four digit products
//     D_t[j, m] = sum_{k in grp h} c_j[k] a_t[m, k]
// are integers below 128 * 255 * 512 < 2^24, exact in the tensor-core
// accumulators.  Per group h the epilogue combines the digits in
// double-float, multiplies by s_jh 2^(E_ih - 9) and adds to a double-float
// accumulator, so T_i carries about 40 significant bits: the subtraction
// Pt_i - T_i, where the low-rank parts of H cancel, loses none of the
// precision float32 would.
//
// A pair of CTAs (cta_group::2): 256 rows x 64 columns of the block's groups
// over the groups of one K split.  Per 64-wide K chunk each CTA loads the
// codes of its own 128 rows and two of the four digit planes, so that an M256
// x N256 MMA (four planes of 64 columns) reads half of its B from each CTA.
//   warp 0       TMA producer of its CTA's tiles, onto the even CTA's barriers
//   warp 1       TMEM allocation; in the even CTA the single-thread MMA issuer
//   warps 2..17  drain: warp w reads TMEM lanes 32 (w % 4) and 16 columns
// Four 64-column accumulators per group h, double-buffered (512 columns).
// The drain does 14 float32 operations per output and group (two outputs per
// instruction), hence sixteen drain warps.
//
// What bounds it, per group and CTA (4096 rows, g = 128): the MMAs take 1024
// cycles, the drain's arithmetic 896 at the full float32 rate, the tile loads
// and operand reads 128 KB of shared-memory traffic.  Two accumulators keep MMA
// and drain of consecutive groups overlapped, but a group's MMAs start only when
// all 32 drain warps have read the accumulator two groups back.  Per launch of
// two groups (256 columns, CUDA events): 32.8 us at K = 4096, 72 us at K = 11008;
// with 17 operations in the drain (the integer part of D_1 split off by adding a
// constant, the product's error formed apart) 36.7 and 82 us.  One CTA per tile
// took 58.9 us at K = 4096 (192 KB of shared-memory traffic per group, and an
// issuing thread that needed 800 cycles per group beside the drain's
// arithmetic).  Measured and not kept, at 17 operations: all digit sums read and
// the accumulator released before any arithmetic (39.1 us: the four warps of a
// scheduler drift apart by a whole group), a block barrier among the drain warps
// per group (39.1 us), one polling lane per warp (37.3 us).
#include <cmath>

#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kTileA = 128 * 64 * 2;   // codes: 128 rows x 64 K, fp16
constexpr int kTileB = 64 * 64 * 2;    // one digit plane: 64 rows of Ht x 64 K
constexpr int kStage = kTileA + 2 * kTileB;
constexpr int kStages = 5;
constexpr int kSRow = 129;             // pitch (floats) of a group's scales: 128 rows, conflict-free
// stages, barriers, and per group of the K split the scales and an exponent
constexpr int smem_bytes(int groups) {
    return 1024 + kStages * kStage + 256 + groups * (kSRow + 1) * 4;
}
// one MMA covers the four digit planes: they are consecutive 64-row tiles
// in the two CTAs' shared memory, and their accumulators consecutive
// 64-column blocks
constexpr uint32_t kIdesc = tc::idesc_f16_f32(256, 256);
constexpr int kDrainWarps = 16;
constexpr int kThreads = 32 * (2 + kDrainWarps);

struct TargetArgs {
    float *out_hi, *out_lo;   // [nsplit][p_pad][nb g]
    const float *S;           // [p][G]
    const int *expoT;         // [G][G] block exponents of Ht
    const int *active;        // optional: rows still refined
    int *status;
    int p, p_pad, d_pad, g, G, seg_per_split;
    int i0, nb;               // groups i0 .. i0 + nb - 1 of this launch
    int prev0;                // groups prev0 .. i0 - 1: the previous grid rewrites their codes
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// kStalled: for the self-test, the issuer stops after one group.
template <bool kStalled>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    tc_target_kernel(const __grid_constant__ CUtensorMap mapC, const __grid_constant__ CUtensorMap mapT,
                     TargetArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(smem + kStages * kStage);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * kStages + 5);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    float *sS = (float *)(smem + kStages * kStage + 256);    // [seg_per_split][kSRow]
    int *sE = (int *)(sS + a.seg_per_split * kSRow);         // [seg_per_split]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = tc::cluster_rank();
    const int j0 = blockIdx.x * 128, jp = j0 - 128 * (int)rank;   // rows of this CTA, of the pair
    const int m0 = a.i0 * a.g + blockIdx.y * 64;         // first row of Ht (output column)
    const int h0 = blockIdx.z * a.seg_per_split;
    const int h1 = min(a.G, h0 + a.seg_per_split);
    const int nkc = a.g / 64;

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kStages + s); };
    auto afull = [&](int b) { return tc::smem_u32(bars + 2 * kStages + b); };
    auto aempty = [&](int b) { return tc::smem_u32(bars + 2 * kStages + 2 + b); };
    const uint32_t closing = tc::smem_u32(bars + 2 * kStages + 4);
    auto tileA = [&](int s) { return tc::smem_u32(smem + s * kStage); };
    auto tileB = [&](int s, int t) { return tc::smem_u32(smem + s * kStage + kTileA + t * kTileB); };

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
    if (warp == 0 && lane == 0) {
        tc::prefetch_tmap(&mapC);
        tc::prefetch_tmap(&mapT);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // The previous grid (the Babai steps of the previous block) rewrites only
    // that block's codes, and reads the phase partials this grid writes.
    // Without the early stop (no active flags to read) each role therefore
    // waits for it only where it must: the producer before the code tile of
    // a chunk of that block, the drain before writing the partials.  The
    // Ht digit tiles, the other code tiles and the scales do not change
    // during the sweep, so the products of the other groups can run while
    // the previous grid finishes.  With the early stop every thread waits
    // here, before reading the flags; so it does in the first block, whose
    // previous grid is the scale solve that writes the scales.
    const bool early = !a.active && a.i0 > 0;
    if (!early) tc::pdl_wait();
    // The next grid (this block's Babai steps) is released at once: before its
    // own wait it reads nothing that this grid or the previous one writes.
    tc::pdl_launch_dependents();
    // a pair of tiles none of whose rows is still active (early stop, App. E)
    // does no work: the Babai step reads the partials of active rows only.
    // Flags are optional in the later branch too: without the early stop the
    // first block has none, nor has the multi-code probe's group 0, and reading
    // them without the null check is a memory fault.
    const bool live = early ? jp < a.p
                            : __syncthreads_or(threadIdx.x < 256 && jp + (int)threadIdx.x < a.p &&
                                               (!a.active || a.active[jp + threadIdx.x] != 0));
    const int nseg = live ? max(0, h1 - h0) : 0;
    const int nchunks = nseg * nkc;

    // The three roles run as whole warps with one elected lane for the TMA and
    // tcgen05 instructions: the control flow stays uniform and the issuing
    // warps need few issue slots beside the drain's arithmetic.
    if (warp == 0) {
        // ---------------- producer
        bool waited = !early, ok = true;
        const uint32_t full0 = tc::map_rank(full(0), 0);
        int s = 0, ph = 1, c = 0;
        for (; c < nchunks; ++c) {
            ok = tc::mbar_wait<kPolls>(empty(s), ph);
            if (!ok) break;
            const int kx = h0 * a.g + c * 64;
            if (!waited && kx >= a.prev0 * a.g && kx < a.i0 * a.g) {
                tc::pdl_wait();   // the codes of the previous block
                waited = true;
            }
            if (tc::elect_one()) {
                if (rank == 0) tc::mbar_expect_tx(full(s), 2 * kStage);
                const uint32_t bar = full0 + 8 * s;
                tc::tma_load_2d_pair(tileA(s), &mapC, bar, kx, j0);
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    tc::tma_load_2d_pair(tileB(s, t), &mapT, bar, kx, (2 * (int)rank + t) * a.d_pad + m0);
            }
            __syncwarp();
            if (++s == kStages) {
                s = 0;
                ph ^= 1;
            }
        }
        // do not leave before the MMAs have consumed the stages filled here:
        // no copy or commit is in flight afterwards
        for (int e = 0; e < min(nchunks, kStages) && ok; ++e) {
            // the slots in order from the oldest: s, s + 1, ...
            const int n = nchunks - min(nchunks, kStages) + e;
            ok = tc::mbar_wait<kPolls>(empty(n % kStages), (n / kStages) & 1);
        }
        if (!ok) {
            *abort_flag = 1;
            tc::abandon_ring(full(0), kStages, c, rank == 0);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer of the pair: one unit per group h
        if (rank == 0) {
            const uint64_t ad0 = tc::sdesc_sw128(tileA(0)), bd0 = tc::sdesc_sw128(tileB(0, 0));
            int s = 0, ph = 0;
            bool ok = true;
            const int nunits = kStalled ? min(nseg, 1) : nseg;
            for (int u = 0; u < nunits && ok; ++u) {
                const int b = u & 1;
                // the unit's stages first (they are usually there already),
                // then its accumulator: nothing but the MMAs' issue lies
                // between the drain's release and the next products
                int s1 = s + 1, ph1 = ph;
                if (s1 == kStages) {
                    s1 = 0;
                    ph1 ^= 1;
                }
                ok = tc::mbar_wait<kPolls>(full(s), ph);
                if (nkc == 2) ok = tc::mbar_wait<kPolls>(full(s1), ph1) && ok;
                ok = tc::mbar_wait<kPolls>(aempty(b), ((u >> 1) & 1) ^ 1) && ok;
                if (!ok) break;
                tc::tc_fence_after();
                if (tc::elect_one()) {
                    const uint64_t o = (uint64_t)(s * (kStage >> 4));
#pragma unroll
                    for (int sub = 0; sub < 4; ++sub)
                        tc::mma_f16_pair(tmem + b * 256, ad0 + o + 2 * sub, bd0 + o + 2 * sub, kIdesc, sub != 0);
                    tc::mma_commit_pair(empty(s));
                    if (nkc == 2) {
                        const uint64_t o1 = (uint64_t)(s1 * (kStage >> 4));
#pragma unroll
                        for (int sub = 0; sub < 4; ++sub)
                            tc::mma_f16_pair(tmem + b * 256, ad0 + o1 + 2 * sub, bd0 + o1 + 2 * sub, kIdesc, 1);
                        tc::mma_commit_pair(empty(s1));
                    }
                    tc::mma_commit_pair(afull(b));
                }
                __syncwarp();
                s = s1;
                ph = ph1;
                if (nkc == 2 && ++s == kStages) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (!tc::mma_done_pair<kPolls>(closing, tc::elect_one()) || !ok) *abort_flag = 1;
        }
    } else {
        // ---------------- drain: digits -> double-float x s_h 2^(E - 9) -> accumulator
        const int q = warp & 3, cq = (warp - 2) >> 2;    // lane quarter, 16-column quarter
        const int rl = 32 * q + lane, row = j0 + rl;
        // the scales of this tile's rows and the block exponents of this
        // split's groups, once (neither changes during a sweep)
        const int t = threadIdx.x - 64;
        for (int u = lane; u < nseg; u += 32) {
            constexpr int kR = 128 / kDrainWarps;    // rows of this warp, all loads in flight
            float sv[kR];
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                const int jr = j0 + (t >> 5) + r * kDrainWarps;
                sv[r] = jr < a.p ? a.S[(size_t)jr * a.G + h0 + u] : 0.f;
            }
#pragma unroll
            for (int r = 0; r < kR; ++r) sS[u * kSRow + (t >> 5) + r * kDrainWarps] = sv[r];
        }
        for (int u = t; u < nseg; u += 32 * kDrainWarps)
            sE[u] = a.expoT[(size_t)(m0 / a.g) * a.G + h0 + u] - 9;
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kDrainWarps) : "memory");
        tc::F2 hi[8], lo[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) hi[e] = lo[e] = tc::f2(0.f);
        bool ok = true;
        const tc::F2 c10 = tc::f2(0x1p-10f), c20 = tc::f2(0x1p-20f);
        const uint32_t released = tc::map_rank(aempty(0), 0);
        for (int u = 0; u < nseg; ++u) {
            const int b = u & 1;
            const float sv = sS[u * kSRow + rl];
            const int e2 = sE[u];
            // s 2^(E - 9): one exact product unless 2^(E - 9) is not normal
            const float sc = (unsigned)(e2 + 126) <= 252u ? sv * __int_as_float((e2 + 127) << 23)
                                                          : ldexpf(sv, e2);
            const tc::F2 scale = tc::f2(sc), nscale = tc::f2(-sc);
            ok = tc::mbar_wait<kPolls>(afull(b), (u >> 1) & 1);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            tc::tc_fence_after();
            const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + b * 256 + cq * 16;
#pragma unroll
            for (int cc = 0; cc < 16; cc += 8) {
                uint32_t v0[8], v1[8], v2[8], v3[8];
                tc::tmem_ld8(base + 0 * 64 + cc, v0);
                tc::tmem_ld8(base + 1 * 64 + cc, v1);
                tc::tmem_ld8(base + 2 * 64 + cc, v2);
                tc::tmem_ld8(base + 3 * 64 + cc, v3);
                tc::tmem_wait_ld();
                if (cc == 8) {
                    // every digit sum of this group is in registers
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_cluster(released + 8 * b);
                }
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    // D_0 + D_1 2^-10 exactly as (vh, vl): vh is the rounded
                    // sum, D_0 - vh is exact (both are multiples of 2^-10, and
                    // D_1 2^-10, where it is the larger, is below 2^14), and so
                    // is what the rounding left out.  The D_2, D_3 terms are
                    // below 2^-20 of the sum and enter the low part.
                    auto pair = [&](const uint32_t (&v)[8]) {
                        return tc::f2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
                    };
                    const tc::F2 d0 = pair(v0), d1 = pair(v1);
                    const tc::F2 vh = tc::f2_fma(d1, c10, d0);
                    const tc::F2 vl = tc::f2_fma(tc::f2_fma(pair(v3), c10, pair(v2)), c20,
                                                 tc::f2_fma(d1, c10, tc::f2_sub(d0, vh)));
                    // (vh + vl) * scale, added to the accumulator: a two-sum of
                    // the rounded product (a sum formed by a multiply-add would
                    // carry bits below both terms, and the differences would
                    // not be exact; the product is negated for that reason)
                    // whose last difference takes the product unrounded and so
                    // its rounding error as well
                    tc::F2 &H = hi[(cc + e) / 2], &L = lo[(cc + e) / 2];
                    const tc::F2 sm = tc::f2_sub(H, tc::f2_mul(vh, nscale));
                    const tc::F2 nb = tc::f2_sub(H, sm);        // - (sm - H)
                    const tc::F2 er = tc::f2_add(tc::f2_sub(H, tc::f2_add(sm, nb)), tc::f2_fma(vh, scale, nb));
                    H = sm;
                    L = tc::f2_add(L, tc::f2_fma(vl, scale, er));
                }
            }
        }
        if (!ok) *abort_flag = 1;
        // the previous grid reads the partials this drain overwrites
        if (early) tc::pdl_wait();
        if (ok && row < a.p) {
            const size_t ncol = (size_t)a.nb * a.g;
            const size_t o = ((size_t)blockIdx.z * a.p_pad + row) * ncol + blockIdx.y * 64 + cq * 16;
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
                *reinterpret_cast<float4 *>(a.out_hi + o + e) = make_float4(x[0], x[1], x[2], x[3]);
                *reinterpret_cast<float4 *>(a.out_lo + o + e) = make_float4(y[0], y[1], y[2], y[3]);
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

}  // namespace

// Split of the K range (groups) over CTAs so that a launch of nb groups covers
// the SMs.
int target_splits(int p_pad, int g, int G, int nb) {
    const int pairs = ((p_pad / 128 + 1) / 2) * (nb * g / 64);
    int n = num_sms() / 2 / pairs;
    if (n < 1) n = 1;
    if (n > kMaxSplit) n = kMaxSplit;
    if (n > G) n = G;
    return n;
}

cudaError_t launch_tc_target(const CUtensorMap &mapC, const CUtensorMap &mapT, float *out_hi,
                             float *out_lo, const float *S, const int *expoT, const int *active,
                             int p, int p_pad, int d_pad, int g, int G, int i0, int nb,
                             int nb_prev, int nsplit, int qmax, int *status, cudaStream_t s,
                             bool pdl, bool stalled) {
    static_assert(smem_bytes(kMaxGroups) <= 227 * 1024, "stages and scales must fit an SM's shared memory");
    const int per = (G + nsplit - 1) / nsplit;
    const int tiles = (p + 255) / 256 * 2;   // pairs of row tiles
    // the digit sums stay exact: 128 * 255 * 512 < 2^24
    if (qmax < 1 || qmax > 255 || g > 128) return cudaErrorInvalidValue;
    if (nb < 1 || i0 + nb > G || nsplit < 1) return cudaErrorInvalidValue;
    TargetArgs a{out_hi, out_lo, S, expoT, active, status, p, p_pad, d_pad, g, G, per,
                 i0, nb, i0 - nb_prev};
    dim3 grid(tiles, nb * g / 64, nsplit);
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t e = set_max_dynamic_smem((const void *)kernel, smem_bytes(kMaxGroups), done);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, grid, dim3(kThreads), (size_t)smem_bytes(per), s, pdl, mapC, mapT, a);
    };
    static std::atomic<unsigned long long> done[2];
    return stalled ? run(tc_target_kernel<true>, done[1]) : run(tc_target_kernel<false>, done[0]);
}

}  // namespace jarq
