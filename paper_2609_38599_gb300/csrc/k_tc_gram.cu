// Gram matrices of the joint scale fit on the tensor cores, exact for the
// digit representation of H.
//
// Sec. 3.3.1, Eq. scale_design: Gram_j[i,h] = (A_i c_i)^T (A_h c_h)
// = c_i^T H_ih c_h with integer codes c = q - z.  Each g x g block H_ih is
// written as 2^(E_ih - 9) * sum_t a_t 2^(-10 t), t = 0..3, with integer
// digits |a_t| <= 512 (exact in fp16) and E_ih the block's exponent
// (max |H_ih| <= 2^E_ih), which represents every entry to within
// 2^(E_ih - 40).  The codes are fp16 as well (|c| <= 255), so
//     D_t[j, m] = sum_{k in grp h} c_j[k] a_t[k, m]
// is an integer below 128 * 255 * 512 < 2^24: every tensor-core partial sum
// is exact whatever the accumulator's rounding.  The epilogue forms the
// integer dots G_t = sum_{m in grp i} c_j[m] D_t[j, m] and
//     Gram_j[i,h] = 2^(E_ih - 9) (G_0 + G_1 2^-10 + G_2 2^-20 + G_3 2^-30)
// in float64.  Only h <= i is computed; the block is mirrored.  The pair of
// groups {i, G-1-i} of a row tile holds G + 1 blocks.  Work items are 256 rows
// and one of `nparts` contiguous ranges of a group pair's blocks, about four
// blocks; each pair of CTAs stays on its SMs and takes every npairs-th item, the
// row tiles of one range first (they share its digit tiles of H in L2).
//
// The CTAs of a pair (cta_group::2) share each MMA as in the sweep's product
// (k_tc_target.cu): each loads the codes of its own 128 rows and two of the four
// digit planes.  One unit of work is (h, column half of group i): 4 accumulators
// of 64 columns (one per digit plane), double-buffered in 512 TMEM columns.
//   warp 0       TMA producer of its CTA's tiles, onto the even CTA's barriers
//   warp 1       TMEM allocation; in the even CTA the MMA issuer
//   warps 2..17  epilogue: warp w reads TMEM lanes 32 (w % 4) .. and 16 of the
//                64 columns of a unit; at the end of a block it leaves its
//                partial dots in shared memory
//   warps 18, 19 add the four partial dots of each row and write the entry of
//                the block: in one of the epilogue warps the conversion and the
//                stores (about 1000 cycles) would hold back the next unit's
//                accumulator, which goes back to the issuer when all of them
//                have read it
//
// What bounds it, per unit and CTA (clock64 in a copy, 4-bit codes): about 2000
// cycles, of which the MMAs are 1024 and the epilogue 900 to 1000 issue slots per
// scheduler (64 digit sums a thread: an add, an integer multiply-add at half
// rate); the rest is the hand-over between them (a ready barrier costs about
// 150 cycles, the four TMEM loads 200 to 400).  Without the dots a launch on
// 4096 x 4096, g = 128 takes 188 us, without the epilogue 162 us, in full 217
// us; 1424 us on 4096 x 11008.  Codes of up to three bits: 200 us, and 409 us with
// groups of 64 (218 and 450 us with the integer dots).  One CTA per tile with
// eight epilogue warps took 325 and 2150 us; the block's sum in one of the
// epilogue warps 231 us, by shared-memory atomics 252 us.
#include <type_traits>

#include "df.cuh"
#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kTileA = 128 * 64 * 2;   // 128 code rows x 64 K (fp16)
constexpr int kTileB = 64 * 64 * 2;    // 64 H rows x 64 K, one digit plane (fp16)
constexpr int kStage = kTileA + 2 * kTileB;
constexpr int kStages = 5;
constexpr int kDrainWarps = 16, kWriteWarps = 2;
constexpr int kThreads = 32 * (2 + kDrainWarps + kWriteWarps);
constexpr int kSlots = 4;              // blocks whose partial dots wait to be written
constexpr int kPartBytes = kSlots * 4 * 2 * 128 * 8;   // int64 partial dots
constexpr int kMaxTiles = 4096;        // row tile pairs whose activity is looked up
constexpr int kSmem = 1024 + kStages * kStage + kPartBytes + 256 + kMaxTiles;
// one MMA covers the four digit planes: they are consecutive 64-row tiles
// in the two CTAs' shared memory, and their accumulators consecutive
// 64-column blocks
constexpr uint32_t kIdesc = tc::idesc_f16_f32(256, 256);

struct GramArgs {
    const uint8_t *Q;
    const int32_t *Z;
    const int *expo;     // [G][G] block exponents E_ih
    const int *active;   // optional: rows whose Gram matrix is needed
    float2 *gram;        // [p][G][G] as float pairs (hi, lo) of the float64 value
    int *status;
    int p, d, g, G, d_pad;
    int nparts;          // block ranges per (row tile pair, group pair)
    int tiles, nitems;   // row tile pairs; tiles x group pairs x nparts
};

// Units of a CTA pair: the blocks (i_lo, h <= i_lo), then (i_hi, h <= i_hi), each
// as its column halves in turn.
struct GramUnit {
    int i_lo, i_hi, nhalf;
    int gi, h, half;
    __device__ __forceinline__ void start(int blk) {
        const bool first = blk <= i_lo;
        gi = first ? i_lo : i_hi;
        h = first ? blk : blk - i_lo - 1;
        half = 0;
    }
    __device__ __forceinline__ void next() {
        if (++half < nhalf) return;
        half = 0;
        if (++h <= gi) return;
        h = 0;
        gi = i_hi;
    }
};

// How an epilogue warp forms its dots, by the width of the codes:
//   up to 3 bits  |c| <= 7, |D_t| <= 128 * 7 * 512, so float32 sums of four
//                 products are exact integers (< 2^24); a conversion and an
//                 integer addition per four products instead of a multiply-add
//                 at half rate for each
//   4 bits        |c| <= 15, |D_t| < 2^20: integer products, every partial dot of
//                 32 terms fits in 32 bits.  Float32 would hold one product, and
//                 a conversion for each takes 328 us where this takes 217 us.
//   wider         |D_t| < 2^24 converted by cvt, 64-bit integer dots
enum { kWideDots = -1, kIntDots = 0 };    // or the number of terms of a float32 sum

// kStalled: for the self-test, the issuer stops after one unit.
template <int kMode, bool kStalled>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    tc_gram_kernel(const __grid_constant__ CUtensorMap mapC, const __grid_constant__ CUtensorMap mapS,
                   GramArgs a) {
    constexpr uint32_t kPolls = tc::wait_polls(kStalled);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    long long *part = (long long *)(smem + kStages * kStage);   // [kSlots][4 warps][2][128]
    uint64_t *bars = (uint64_t *)(smem + kStages * kStage + kPartBytes);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * kStages + 5 + 2 * kSlots);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)tc::cluster_rank();
    uint8_t *live = smem + kStages * kStage + kPartBytes + 256;   // [tiles]
    const int G = a.G, g = a.g;
    const int nkc = g / 64;                // K chunks per unit (and column halves of a group)
    const int npairs = gridDim.x / 2, ngp = (G + 1) / 2;
    // a row tile pair none of whose rows is active is skipped; both CTAs read
    // the same flags
    const bool flags = a.active && a.tiles <= kMaxTiles;
    // item -> first row of the tile pair, first unit and number of units
    // [nblk z / nparts, nblk (z + 1) / nparts) of the group pair's blocks; 0
    // units for a tile without active rows
    auto item = [&](int it, int &jp, GramUnit &un) {
        const int tile = it % a.tiles, gp = (it / a.tiles) % ngp, z = it / (a.tiles * ngp);
        jp = tile * 256;
        un.i_lo = gp;
        un.i_hi = G - 1 - gp;
        un.nhalf = nkc;
        if (flags && !live[tile]) return 0;
        const int nblk = un.i_lo == un.i_hi ? un.i_lo + 1 : G + 1;
        const int blk0 = nblk * z / a.nparts;
        un.start(blk0);
        return (nblk * (z + 1) / a.nparts - blk0) * nkc;
    };

    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kStages + s); };
    auto afull = [&](int b) { return tc::smem_u32(bars + 2 * kStages + b); };
    auto aempty = [&](int b) { return tc::smem_u32(bars + 2 * kStages + 2 + b); };
    auto sfull = [&](int s) { return tc::smem_u32(bars + 2 * kStages + 4 + s); };
    auto sfree = [&](int s) { return tc::smem_u32(bars + 2 * kStages + 4 + kSlots + s); };
    const uint32_t closing = tc::smem_u32(bars + 2 * kStages + 4 + 2 * kSlots);
    auto tileA = [&](int s) { return tc::smem_u32(smem + s * kStage); };
    auto tileB = [&](int s, int t) { return tc::smem_u32(smem + s * kStage + kTileA + t * kTileB); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            tc::mbar_init(sfull(s), kDrainWarps);
            tc::mbar_init(sfree(s), kWriteWarps);
        }
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
        tc::prefetch_tmap(&mapS);
    }
    // launched programmatically the previous grid may still run: all that it
    // writes (codes, flags) is read, and the next grid released, after it
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    if (flags)
        for (int t = warp; t < a.tiles; t += kThreads / 32) {
            int mine = 0;
            for (int r = lane; r < 256; r += 32)
                if (t * 256 + r < a.p) mine |= a.active[t * 256 + r];
            mine = __any_sync(0xffffffffu, mine);
            if (lane == 0) live[t] = (uint8_t)mine;
        }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- producer: per chunk, codes of group h and two digit planes
        bool ok = true;
        const uint32_t full0 = tc::map_rank(full(0), 0);
        GramUnit un;
        int s = 0, ph = 1, nchunks = 0, jp;
        for (int it = blockIdx.x / 2; it < a.nitems && ok; it += npairs) {
            const int nunits = item(it, jp, un);
            for (int u = 0; u < nunits && ok; ++u, un.next()) {
                for (int kc = 0; kc < nkc; ++kc) {
                    ok = tc::mbar_wait<kPolls>(empty(s), ph);
                    if (!ok) break;
                    if (tc::elect_one()) {
                        if (rank == 0) tc::mbar_expect_tx(full(s), 2 * kStage);
                        const uint32_t bar = full0 + 8 * s;
                        const int kx = un.h * g + kc * 64;
                        tc::tma_load_2d_pair(tileA(s), &mapC, bar, kx, jp + 128 * rank);
#pragma unroll
                        for (int t = 0; t < 2; ++t)
                            tc::tma_load_2d_pair(tileB(s, t), &mapS, bar, kx,
                                                 (2 * rank + t) * a.d_pad + un.gi * g + un.half * 64);
                    }
                    __syncwarp();
                    ++nchunks;
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
        }
        // do not leave before the MMAs have consumed the stages filled here:
        // no copy or commit is in flight afterwards
        for (int n = max(0, nchunks - kStages); n < nchunks && ok; ++n)
            ok = tc::mbar_wait<kPolls>(empty(n % kStages), (n / kStages) & 1);
        if (!ok) {
            *abort_flag = 1;
            tc::abandon_ring(full(0), kStages, nchunks, rank == 0);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer of the pair
        if (rank == 0) {
            const uint64_t ad0 = tc::sdesc_sw128(tileA(0)), bd0 = tc::sdesc_sw128(tileB(0, 0));
            int s = 0, ph = 0;
            bool ok = true;
            GramUnit un;
            int jp, total = 0;
            for (int it = blockIdx.x / 2; it < a.nitems; it += npairs) total += item(it, jp, un);
            if (kStalled) total = min(total, 1);
            for (int u = 0; u < total && ok; ++u) {
                const int b = u & 1;
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
    } else if (warp < 2 + kDrainWarps) {
        // ---------------- epilogue: exact integer dots with the codes of group i
        const int q = warp & 3, cq = (warp - 2) >> 2;   // lane quarter, 16-column quarter
        const int rl = 32 * q + lane;           // row within the tile
        const uint32_t released = tc::map_rank(aempty(0), 0);
        GramUnit un;
        int z = 0, jp, ug = 0, nb = 0;          // ug, nb: units, blocks of this pair so far
        uint32_t q4[2][4] = {};                 // this warp's codes of group i, both halves
        bool ok = true;
        typedef typename std::conditional<kMode == kWideDots, long long, int>::type acc_t;
        acc_t acc[4] = {0, 0, 0, 0};
        for (int it = blockIdx.x / 2; it < a.nitems && ok; it += npairs) {
            const int nunits = item(it, jp, un);
            const int rc = min(jp + 128 * rank + rl, a.p - 1);
            int cur_g = -1;
            for (int u = 0; u < nunits; ++u, ++ug, un.next()) {
                if (un.gi != cur_g) {
                    cur_g = un.gi;
                    z = a.Z[(size_t)rc * G + cur_g];
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
                        if (hf < nkc) {
                            const uint4 v = *reinterpret_cast<const uint4 *>(
                                a.Q + (size_t)rc * a.d + cur_g * g + hf * 64 + cq * 16);
                            q4[hf][0] = v.x; q4[hf][1] = v.y; q4[hf][2] = v.z; q4[hf][3] = v.w;
                        }
                }
                // c = q - z, as integers or as float pairs (the bits of 2^23 + q
                // are 0x4B000000 + q; both differences are exact)
                int c[16];
                tc::F2 cf[8];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const uint32_t w = un.half ? q4[1][e >> 2] : q4[0][e >> 2];
                    c[e] = kMode > 0 ? (int)__byte_perm(w, 0x4B000000u, 0x7440 | (e & 3))
                                               : (int)__byte_perm(w, 0, 0x4440 | (e & 3)) - z;
                }
                if (kMode > 0) {
                    const tc::F2 off = tc::f2(-8388608.0f - (float)z);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        cf[e] = tc::f2_add(tc::f2(__int_as_float(c[2 * e]), __int_as_float(c[2 * e + 1])), off);
                }
                const int b = ug & 1;
                ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(afull(b), (ug >> 1) & 1));
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + b * 256 + cq * 16;
                auto release = [&]() {
                    // every digit sum of this unit is in registers
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_cluster(released + 8 * b);
                };
                if constexpr (kMode == kWideDots) {
#pragma unroll
                    for (int t = 0; t < 4; t += 2) {
                        uint32_t v[2][16];
                        tc::tmem_ld16(base + t * 64, v[0]);
                        tc::tmem_ld16(base + (t + 1) * 64, v[1]);
                        tc::tmem_wait_ld();
                        if (t == 2) release();
#pragma unroll
                        for (int k = 0; k < 2; ++k)
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                acc[t + k] += (long long)c[e] * __float2int_rn(__uint_as_float(v[k][e]));
                    }
                } else if constexpr (kMode > 0) {
                    uint32_t v[4][16];
#pragma unroll
                    for (int t = 0; t < 4; ++t) tc::tmem_ld16(base + t * 64, v[t]);
                    tc::tmem_wait_ld();
                    release();
                    // |c D| <= 7 * 7 * 128 * 512: sums of four are below 2^24
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        auto dg = [&](int e) {
                            return tc::f2(__uint_as_float(v[t][2 * e]), __uint_as_float(v[t][2 * e + 1]));
                        };
#pragma unroll
                        for (int h = 0; h < 8; h += kMode) {
                            tc::F2 sum = tc::f2_fma(cf[h], dg(h), tc::f2(0.f));
#pragma unroll
                            for (int e = h + 1; e < h + kMode; ++e) sum = tc::f2_fma(cf[e], dg(e), sum);
                            float x0, x1;
                            tc::f2_get(sum, x0, x1);
                            acc[t] += __float2int_rn(x0) + __float2int_rn(x1);
                        }
                    }
                } else {
                    uint32_t v[4][16];
#pragma unroll
                    for (int t = 0; t < 4; ++t) tc::tmem_ld16(base + t * 64, v[t]);
                    tc::tmem_wait_ld();
                    release();
                    // D is an integer, |D| < 2^22: the bits of D + 1.5 2^23 are
                    // 0x4B400000 + D; the offset's share is taken off once
                    // (modulo 2^32; the dot itself fits)
                    int cs = 0;
#pragma unroll
                    for (int e = 0; e < 16; ++e) cs += c[e];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        uint32_t p0 = 0, p1 = 0;
#pragma unroll
                        for (int e = 0; e < 16; e += 2) {
                            float x0, x1;
                            tc::f2_get(tc::f2_add(tc::f2(__uint_as_float(v[t][e]), __uint_as_float(v[t][e + 1])),
                                                  tc::f2(12582912.0f)), x0, x1);
                            p0 += (uint32_t)c[e] * __float_as_uint(x0);
                            p1 += (uint32_t)c[e + 1] * __float_as_uint(x1);
                        }
                        acc[t] += (int)(p0 + p1 - 0x4B400000u * (uint32_t)cs);
                    }
                }
                if (un.half == nkc - 1) {
                    // two digits to a 64-bit integer (four for narrow codes:
                    // |acc_t| < 128 * 15 * 2^20 < 2^31 over all columns)
                    const long long hi = (long long)acc[0] * (1 << 10) + acc[1];
                    const long long lo = (long long)acc[2] * (1 << 10) + acc[3];
                    const int slot = nb % kSlots;
                    ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(sfree(slot), ((nb / kSlots) & 1) ^ 1));
                    if (!ok) break;
                    long long *pp = part + (size_t)((slot * 4 + cq) * 2) * 128 + rl;
                    if constexpr (kMode == kWideDots) {
                        pp[0] = hi;
                        pp[128] = lo;
                    } else {
                        pp[0] = hi * (1 << 20) + lo;
                    }
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(sfull(slot));
#pragma unroll
                    for (int t = 0; t < 4; ++t) acc[t] = 0;
                    ++nb;
                }
            }
        }
        if (!ok) *abort_flag = 1;
    } else {
        // ---------------- write the finished blocks, 64 rows a warp
        const int r0 = 64 * (warp - 2 - kDrainWarps) + lane;
        GramUnit un;
        int jp, nb = 0;
        bool ok = true;
        for (int it = blockIdx.x / 2; it < a.nitems && ok; it += npairs) {
            const int nblk = item(it, jp, un) / nkc;
            for (int k = 0; k < nblk; ++k, ++nb) {
                const int E = a.expo[un.gi * G + un.h], slot = nb % kSlots;
                ok = __all_sync(0xffffffffu, tc::mbar_wait<kPolls>(sfull(slot), (nb / kSlots) & 1));
                if (!ok) break;
                const long long *pp = part + (size_t)slot * 4 * 2 * 128;
                float2 v2[2];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const long long *pr = pp + r0 + 32 * r;
                    const long long s0 = (pr[0] + pr[256]) + (pr[512] + pr[768]);
                    double v;
                    if constexpr (kMode == kWideDots) {
                        const long long s1 = (pr[128] + pr[384]) + (pr[640] + pr[896]);
                        v = ldexp((double)s0, E - 19) + ldexp((double)s1, E - 39);
                    } else {
                        // one exact 64-bit integer, converted with a single
                        // rounding (two float64 operations; float64 is a narrow
                        // pipe on this GPU)
                        v = __ll2double_rn(s0) * __longlong_as_double((long long)(E - 39 + 1023) << 52);
                    }
                    // stored once as the float pair the scale solve works on
                    const DF vp = split_double(v);
                    v2[r] = make_float2(vp.h, vp.l);
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(sfree(slot));
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int row = jp + 128 * rank + r0 + 32 * r;
                    if (row < a.p) {
                        float2 *gr = a.gram + (size_t)row * G * G;
                        gr[(size_t)un.gi * G + un.h] = v2[r];
                        gr[(size_t)un.h * G + un.gi] = v2[r];
                    }
                }
                un.half = nkc - 1;      // on to the next block
                un.next();
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

// Per g x g block of H: E = the exponent with max |H_blk| <= 2^E.  With
// `sym` the maximum also runs over the mirrored block (bh, bi), so that the
// exponent map is symmetric for a matrix that is not (the target projection
// reads the exponent of block (k, n) for the digits of entry (n, k)).
__global__ void block_exponent_kernel(const float *__restrict__ Hs, int *__restrict__ expo, int d,
                                      int g, int sym) {
    const int G = d / g, bi = blockIdx.y, bh = blockIdx.x, g4 = g / 4;
    float mx = 0.f;
    auto take = [&](int br, int bc, int idx) {
        const float4 v = *reinterpret_cast<const float4 *>(
            Hs + (size_t)(br * g + idx / g4) * d + bc * g + 4 * (idx % g4));
        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    };
#pragma unroll 4
    for (int idx = threadIdx.x; idx < g * g4; idx += blockDim.x) take(bi, bh, idx);
    if (sym)
#pragma unroll 4
        for (int idx = threadIdx.x; idx < g * g4; idx += blockDim.x) take(bh, bi, idx);
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ float wm[32];
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, wm[w]);
        int e = 0;
        if (m > 0.f) {
            frexpf(m, &e);     // m = f 2^e, f in [0.5, 1): |H| <= 2^e
        }
        expo[bi * G + bh] = e;
    }
}

// The digit kernels take eight consecutive entries of a row per thread (they
// lie in one block: g is a multiple of 64) and store each plane's eight digits
// as 16 bytes.  One entry a thread, a 2-byte store per plane, took 147 us for the
// ten planes of a 4096 x 4096 H.
__device__ __forceinline__ void load8(const float *p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// Digits of every entry of H for the two integer-digit schemes, from the
// block exponent E (max |H_blk| <= 2^E):
//  * dig8 (bf16, six planes, target projection): x = H 2^(7 - E) in
//    [-128, 128], a_0 = rint(x), a_t = rint(256 * remainder);
//  * dig10 (fp16, four planes, Gram): x = H 2^(9 - E) in [-512, 512],
//    a_0 = rint(x), a_t = rint(1024 * remainder).
__global__ void slice_kernel(const float *__restrict__ Hs, const int *__restrict__ expo,
                             __nv_bfloat16 *__restrict__ dig8, __half *__restrict__ dig10, int d,
                             int d_pad, int g) {
    const int G = d / g, d8 = d / 8;
    const size_t n8 = (size_t)d * d8;
    const size_t plane = (size_t)d_pad * d_pad;
    for (size_t i8 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i8 < n8;
         i8 += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(i8 / d8), c = 8 * (int)(i8 % d8);
        const int E = expo[(r / g) * G + c / g];
        const size_t off = (size_t)r * d_pad + c;
        float h[8], x[8];
        load8(Hs + (size_t)r * d + c, h);
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = ldexpf(h[k], 7 - E);
#pragma unroll
        for (int t = 0; t < 6; ++t) {
            __align__(16) __nv_bfloat16 q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dgt = rintf(x[k]);
                q[k] = __float2bfloat16_rn(dgt);
                x[k] = (x[k] - dgt) * 256.f;
            }
            *reinterpret_cast<uint4 *>(dig8 + t * plane + off) = *reinterpret_cast<const uint4 *>(q);
        }
        if (!dig10) continue;
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = ldexpf(h[k], 9 - E);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            __align__(16) __half q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dgt = rintf(x[k]);
                q[k] = __float2half_rn(dgt);
                x[k] = (x[k] - dgt) * 1024.f;
            }
            *reinterpret_cast<uint4 *>(dig10 + t * plane + off) = *reinterpret_cast<const uint4 *>(q);
        }
    }
}

// Digits of a double-float matrix M = hi + lo (not necessarily symmetric) in
// the Gram scheme: x = M 2^(9 - E) in [-512, 512] with E the block exponent,
// four fp16 planes base 2^10.  The low part enters before the remainder is
// scaled, so the digits represent hi + lo to 2^(E - 40).
__global__ void slice10_kernel(const float *__restrict__ hi, const float *__restrict__ lo,
                               const int *__restrict__ expo, __half *__restrict__ dig, int d,
                               int d_pad, int g) {
    const int G = d / g, d8 = d / 8;
    const size_t n8 = (size_t)d * d8;
    const size_t plane = (size_t)d_pad * d_pad;
    for (size_t i8 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i8 < n8;
         i8 += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(i8 / d8), c = 8 * (int)(i8 % d8);
        const int E = expo[(r / g) * G + c / g];
        const size_t off = (size_t)r * d_pad + c;
        float x[8], xl[8];
        load8(hi + (size_t)r * d + c, x);
        load8(lo + (size_t)r * d + c, xl);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            x[k] = ldexpf(x[k], 9 - E);
            xl[k] = ldexpf(xl[k], 9 - E);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            __align__(16) __half q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dgt = rintf(x[k]);
                q[k] = __float2half_rn(dgt);
                x[k] = x[k] - dgt;
                if (t == 0) x[k] += xl[k];
                x[k] *= 1024.f;
            }
            *reinterpret_cast<uint4 *>(dig + t * plane + off) = *reinterpret_cast<const uint4 *>(q);
        }
    }
}

}  // namespace

cudaError_t launch_slice10(const float *hi, const float *lo, int *expo, __half *dig, int d,
                           int d_pad, int g, cudaStream_t s) {
    const int G = d / g;
    block_exponent_kernel<<<dim3(G, G), 256, 0, s>>>(hi, expo, d, g, 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    size_t n = (size_t)d * d / 8;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 16 * num_sms()) blocks = 16 * num_sms();
    slice10_kernel<<<blocks, 256, 0, s>>>(hi, lo, expo, dig, d, d_pad, g);
    return cudaGetLastError();
}

cudaError_t launch_slices(const float *Hs, int *expo, __nv_bfloat16 *dig8, __half *dig10, int d,
                          int d_pad, int g, cudaStream_t s) {
    const int G = d / g;
    block_exponent_kernel<<<dim3(G, G), 256, 0, s>>>(Hs, expo, d, g, 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    size_t n = (size_t)d * d / 8;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 16 * num_sms()) blocks = 16 * num_sms();
    slice_kernel<<<blocks, 256, 0, s>>>(Hs, expo, dig8, dig10, d, d_pad, g);
    return cudaGetLastError();
}

cudaError_t launch_slices8(const float *M, int *expo, __nv_bfloat16 *dig8, int d, int d_pad,
                           int g, cudaStream_t s) {
    const int G = d / g;
    block_exponent_kernel<<<dim3(G, G), 256, 0, s>>>(M, expo, d, g, 1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    size_t n = (size_t)d * d / 8;
    int blocks = (int)((n + 255) / 256);
    if (blocks > 16 * num_sms()) blocks = 16 * num_sms();
    slice_kernel<<<blocks, 256, 0, s>>>(M, expo, dig8, nullptr, d, d_pad, g);
    return cudaGetLastError();
}

cudaError_t launch_tc_gram(const CUtensorMap &mapC, const CUtensorMap &mapS, const uint8_t *Q,
                           const int32_t *Z, const int *expo, const int *active, float2 *gram,
                           int p, int p_pad, int d, int d_pad, int g, int bits, int *status,
                           cudaStream_t s, bool pdl, bool stalled) {
    const int G = d / g;
    // ranges per (row tile pair, group pair): the fewest blocks for the busiest
    // CTA pair, each item costing about a sixth of a block beside its blocks
    // (its rows' codes of the group)
    const int npairs = num_sms() / 2, tiles = (p + 255) / 256, ngp = (G + 1) / 2;
    int nparts = 1;
    double best = 0.0;
    for (int n = 1; n <= G + 1; ++n) {
        const long long rounds = ((long long)tiles * ngp * n + npairs - 1) / npairs;
        const double t = (double)rounds * ((double)(G + 1) / n + 0.17);
        if (n == 1 || t < best - 1e-9) {
            best = t;
            nparts = n;
        }
    }
    const long long items = (long long)tiles * ngp * nparts;
    if (items > 0x7fffffff) return cudaErrorInvalidValue;
    GramArgs a{Q, Z, expo, active, gram, status, p, d, g, G, d_pad, nparts, tiles, (int)items};
    const dim3 grid(2 * (items < npairs ? (int)items : npairs));
    auto run = [&](auto *kernel, std::atomic<unsigned long long> &done) {
        const cudaError_t e = set_max_dynamic_smem((const void *)kernel, kSmem, done);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, grid, dim3(kThreads), (size_t)kSmem, s, pdl, mapC, mapS, a);
    };
    static std::atomic<unsigned long long> done[4];
    if (stalled) return run(tc_gram_kernel<kIntDots, true>, done[3]);
    if (bits <= 3) return run(tc_gram_kernel<4, false>, done[0]);
    if (bits <= 4) return run(tc_gram_kernel<kIntDots, false>, done[1]);
    return run(tc_gram_kernel<kWideDots, false>, done[2]);
}

}  // namespace jarq
