// Bounded Babai proposals and acceptance for the groups of one block of the
// sweep, every active row (Sec. 3.3.2, Eqs. conditional_residual, group_bils,
// group_qr, babai_update; App. E "Small scales").
//
// The sweep runs in blocks of a few groups (sweep_block).  The product
// (k_tc_target.cu) has formed T_i = sum_h s_h R_i^{-T} H_ih c_h for every
// group i of the block from the codes before the block; this kernel takes
// each row through the block's groups in order.  A proposal that is accepted
// for group i changes T_i' of the later groups i' of the block by
// s_i R_i'^{-T} H_i'i Delta, and only 2 to 25 % of the proposals are accepted, 35
// to 70 changed codes each, so the change is added here column by column
// (the integer digits of Ht_i'i, in integers: exactly the digit sums that
// the product would form from the new codes) instead of by a product per
// group.
//
// Per group the recursion is evaluated relative to the row's current codes q.
// The target y = R_i^{-T} (H r)_i / s is formed in double-float as
// (Pt_i - T_i) / s: Pt_i = R_i^{-T} (H w)_i from the folded target projection,
// so that the cancellation of H's low-rank part costs no precision.  Then
//     v = R_i^{-T} [(H r)_i + s H_ii c] / s = y + R_i c,   c = q - z,
// so the pre-round value of Eq. babai_update is
//     z + x_l = q_l + (y_l - sum_{h>l} R_lh Delta_h) / R_ll,
// Delta_h = q^cand_h - q_h.
//
// Sixteen lanes hold one row: lane k owns the quads l = 64 m + 4 k + b of its
// coordinates, and a warp takes two rows at once.  The back substitution scans
// the quads from the last to the first: the owner decides its four coordinates
// one after the other, the four changes are broadcast to the row's lanes by
// shuffles, and every lane updates the running vector u = y - R Delta of the
// coordinates below.
//
// The change of the group objective (Eq. group_bils) is
// dF = s^2 (||R Delta - y||^2 - ||y||^2) = s^2 sum_l (a_l - y_l)(a_l + y_l)
// with a_l = R_ll Delta_l - u_l, exactly zero for an unchanged proposal.  A
// proposal is kept iff it changes a code, dF is finite and dF < 0.
//
// The last warp of a block streams what the rows share through shared
// memory: the groups' packed factors and the digits of the blocks Ht_i'i.
//
// What bounds it: latency and issue slots together.  Each quad is a chain of
// four decisions, four shuffles and the column updates; 4096 rows put 14 row
// warps on an SM, which issue in half of the cycles (a quarter of their stalls
// is the wait for a group's targets).  Measured (CUDA events around a launch, a
// block of 256 columns): 27.6 us for 4096 rows at g = 128, 24.2 us for 1000 rows
// at g = 64, 74.6 us for 14336 rows at g = 128.  Four rows a warp (half the
// warps) took 27.5, 30.3 and 68.9 us, eight rows 35 us on 4096; one launch per
// group with a whole warp per row 18.8 us a group (its scan spent most of its
// issue slots on decisions that 31 of 32 lanes repeat).  The lanes of a warp's
// rows lie side by side, so that a 16-byte shared load of the factor is one
// address for both.
// Gathering the columns of Ht_i'i from global memory instead of shared
// memory, with blocks of four groups, took 157 us per block (4 x 27 us for
// the groups alone): an accepted row waits on L2 for every few columns.
#include <type_traits>

#include "tc_common.cuh"

namespace jarq {
namespace {

constexpr int kFactorSlots = 2;  // group factors in shared memory at once
constexpr int kMaxWarps = 15;    // row warps per block at most (and one loader)

// Blocks Ht_i'i in shared memory at once: those of one group i.
__host__ __device__ constexpr int pair_slots(int g) { return sweep_block(g) - 1; }

struct BabaiArgs {
    float *t_hi, *t_lo;          // [nsplit][p_pad][nb g] split-K partials of T
    const float *pt_hi, *pt_lo;  // [p][d] folded target projection Pt
    int nsplit;
    const float *Lf;             // [G][factor_floats(g)]
    const int2 *band;            // digits of Ht_{i'i} (jarq_hessian::band)
    const int *expoT;            // [G][G] block exponents of Ht
    const float *S;
    uint8_t *Q;
    const int32_t *Z;
    ResidualView rv;
    const int *active;
    int *accepted;
    int *status;
    int p, i0, nb, qmax;
    float eps;
};

// T_i' += s Ht_i'i Delta for one row: `list` holds the n changed coordinates
// (Delta * 256 + coordinate), `blk` the digits of Ht_i'i column by column;
// the warp's lane owns MV = g/32 consecutive outputs.  The digit sums are
// integers: 20-bit halves times |Delta| <= qmax summed over at most g terms
// fit in 32 bits for qmax <= 15 and are summed in 64 bits otherwise (WIDE).
template <int MV, bool WIDE>
__device__ __forceinline__ void add_changes(const int2 *blk, const int *list, int n, float s,
                                            int E, float *th, float *tl) {
    constexpr int g = 32 * MV;
    typedef typename std::conditional<WIDE, long long, int>::type acc_t;
    const int lane = threadIdx.x & 31;
    float told[MV], lold[MV];
#pragma unroll
    for (int m = 0; m < MV; ++m) {
        told[m] = th[MV * lane + m];
        lold[m] = tl[MV * lane + m];
    }
    acc_t ah[MV], al[MV];
#pragma unroll
    for (int m = 0; m < MV; ++m) ah[m] = al[m] = 0;
    const int2 *col = blk + MV * lane;
#pragma unroll 4
    for (int e = 0; e < n; ++e) {
        const int ent = list[e], dq = ent >> 8;
        const int4 *c4 = reinterpret_cast<const int4 *>(col + (ent & 0xFF) * g);
#pragma unroll
        for (int m = 0; m < MV; m += 2) {
            const int4 v = c4[m / 2];
            ah[m] += (acc_t)dq * v.x;
            al[m] += (acc_t)dq * v.y;
            ah[m + 1] += (acc_t)dq * v.z;
            al[m + 1] += (acc_t)dq * v.w;
        }
    }
    const float scale = ldexpf(s, E - 9);
#pragma unroll
    for (int m = 0; m < MV; ++m) {
        // the digit sum in units of 2^-30, as a float pair
        const long long v = (long long)ah[m] * (1 << 20) + (long long)al[m];
        const float fh = __ll2float_rn(v);
        const float fl = __ll2float_rn(v - __float2ll_rn(fh));
        const float vh = fh * 0x1p-30f, vl = fl * 0x1p-30f;
        const float ph = vh * scale;
        const float pe = fmaf(vh, scale, -ph);
        const float t = told[m];
        const float sm = __fadd_rn(t, ph);
        const float bb = __fsub_rn(sm, t);
        const float er = __fadd_rn(__fsub_rn(t, __fsub_rn(sm, bb)), __fsub_rn(ph, bb));
        th[MV * lane + m] = sm;
        tl[MV * lane + m] = lold[m] + (er + fmaf(vl, scale, pe));
    }
}

// Byte b of a word as a float (exact).
__device__ __forceinline__ float byte_float(uint32_t w, int b) {
    return __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 | b)), 8388608.0f);
}

// NM: quads per lane
template <int NM, bool WIDE>
__global__ void __launch_bounds__(32 * (kMaxWarps + 1), 1) babai_kernel(BabaiArgs a) {
    constexpr int g = 64 * NM;
    constexpr int kFactor = factor_floats(g), kPairs = pair_slots(g);
    extern __shared__ __align__(128) float smem[];
    __shared__ uint64_t bars[2 * (kFactorSlots + kPairs)];
    __shared__ int abort_flag;
    volatile int *abort_f = &abort_flag;
    int2 *pairs = reinterpret_cast<int2 *>(smem + kFactorSlots * kFactor);   // [kPairs][g][g]
    const int d = a.rv.d, G = d / g;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = (blockDim.x >> 5) - 1;
    auto full = [&](int s) { return tc::smem_u32(bars + s); };
    auto empty = [&](int s) { return tc::smem_u32(bars + kFactorSlots + s); };
    auto pfull = [&](int s) { return tc::smem_u32(bars + 2 * kFactorSlots + s); };
    auto pempty = [&](int s) { return tc::smem_u32(bars + 2 * kFactorSlots + kPairs + s); };
    if (threadIdx.x == 0) {
        for (int s = 0; s < kFactorSlots; ++s) {
            tc::mbar_init(full(s), 1);
            tc::mbar_init(empty(s), nwarps);
        }
        for (int s = 0; s < kPairs; ++s) {
            tc::mbar_init(pfull(s), 1);
            tc::mbar_init(pempty(s), nwarps);
        }
        *abort_f = 0;
        tc::fence_barrier_init();
    }
    __syncthreads();
    if (wid == nwarps) {
        // ---------------- loader.  Nothing it reads depends on the previous
        // kernel: the first copies overlap that kernel's tail.  Group n takes
        // factor slot n % kFactorSlots, its block with group n2 > n pair
        // slot n2 - n - 1.
        if (lane == 0) {
            for (int n = 0; n < a.nb; ++n) {
                const int s = n % kFactorSlots;
                if (!tc::mbar_wait(empty(s), ((n / kFactorSlots) & 1) ^ 1) || *abort_f) {
                    *abort_f = 1;
                    break;
                }
                tc::mbar_expect_tx(full(s), kFactor * sizeof(float));
                tc::bulk_load(tc::smem_u32(smem + s * kFactor),
                              a.Lf + (size_t)(a.i0 + n) * kFactor, kFactor * sizeof(float), full(s));
                for (int t = 0; t < a.nb - 1 - n; ++t) {
                    // slot t held the blocks of the groups 0 .. n - 1
                    if (!tc::mbar_wait(pempty(t), (n & 1) ^ 1) || *abort_f) {
                        *abort_f = 1;
                        break;
                    }
                    tc::mbar_expect_tx(pfull(t), g * g * sizeof(int2));
                    tc::bulk_load(tc::smem_u32(pairs + (size_t)t * g * g),
                                  a.band + ((size_t)(a.i0 + n) * kPairs + t) * g * g,
                                  g * g * sizeof(int2), pfull(t));
                }
            }
            if (*abort_f) atomicOr(a.status, ST_TIMEOUT);
        }
    } else {
        // The block's product (previous kernel) must be complete before its
        // partials are read and before the codes it reads are rewritten.  The
        // next grid is released only after this wait: by then every grid before
        // this one has completed, so the next product may read the codes of the
        // groups outside this block before its own wait.
        // The rows' Pt, which no kernel of the sweep writes, starts for L2 now.
        {
            const float *pt = (lane & 16) ? a.pt_lo : a.pt_hi;
            const int j = (blockIdx.x * nwarps + wid) * 2 + (lane & 1);
            if (j < a.p)
                for (int e = 32 * ((lane >> 1) & 7); e < a.nb * g; e += 256)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(pt + (size_t)j * d + a.i0 * g + e));
        }
        tc::pdl_wait();
        tc::pdl_launch_dependents();
        int *list = reinterpret_cast<int *>(pairs + (size_t)kPairs * g * g) + wid * g;
        const int k = lane >> 1, sub = lane & 1;     // 16 lanes a row
        const int ncol = a.nb * g;
        // rounding to the nearest even integer adds 1.5 * 2^23 (exact for
        // |x| < 2^22; beyond that the clamp gives the same code as rintf); the
        // clamp to [0, qmax] and the difference to the current code are taken
        // in that offset form, where all three are exact
        constexpr float kRound = 12582912.0f;      // 1.5 * 2^23
        const float rmax = kRound + (float)a.qmax;
        bool ok = true;
        for (int n = 0; n < a.nb && ok; ++n) {
            const int i = a.i0 + n, slot = n % kFactorSlots;
            ok = tc::mbar_wait(full(slot), (n / kFactorSlots) & 1);
            for (int t = 0; t < a.nb - 1 - n; ++t) ok = tc::mbar_wait(pfull(t), n & 1) && ok;
            ok = __all_sync(0xffffffffu, ok && *abort_f == 0);
            if (!ok) {
                *abort_f = 1;
                break;
            }
            const float *F = smem + slot * kFactor;
            const float *Ftri = F + factor_tri(g) + 8 * k, *Fdiag = F + factor_diag(g) + 4 * k,
                        *Frd = F + factor_rdiag(g) + 4 * k;
            for (int base = (blockIdx.x * nwarps + wid) * 2; base < a.p;
                 base += gridDim.x * nwarps * 2) {
                const int j = base + sub, jc = min(j, a.p - 1);
                const size_t off = (size_t)jc * d + (size_t)i * g + 4 * k;
                const float s = a.S[(size_t)jc * G + i];
                const int z = a.Z[(size_t)jc * G + i];
                const bool live = j < a.p && a.active[jc] != 0 && fabsf(s) > a.eps;   // false for NaN
                float u[NM][4], y[NM][4], yl[NM][4];
                uint32_t qo[NM], qn[NM];             // current and proposed codes
#pragma unroll
                for (int c = 0; c < NM; ++c)
                    qo[c] = *reinterpret_cast<const uint32_t *>(a.Q + off + 64 * c);
                // s y = Pt_i - sum_sp T_sp, in double-float
#pragma unroll
                for (int c = 0; c < NM; ++c) {
                    const float4 h4 = *reinterpret_cast<const float4 *>(a.pt_hi + off + 64 * c);
                    const float4 l4 = *reinterpret_cast<const float4 *>(a.pt_lo + off + 64 * c);
                    y[c][0] = h4.x; y[c][1] = h4.y; y[c][2] = h4.z; y[c][3] = h4.w;
                    yl[c][0] = l4.x; yl[c][1] = l4.y; yl[c][2] = l4.z; yl[c][3] = l4.w;
                }
                for (int sp = 0; sp < a.nsplit; ++sp) {
                    const size_t o = ((size_t)sp * a.rv.p_pad + jc) * ncol + n * g + 4 * k;
#pragma unroll
                    for (int c = 0; c < NM; ++c) {
                        const float4 h4 = *reinterpret_cast<const float4 *>(a.t_hi + o + 64 * c);
                        const float4 l4 = *reinterpret_cast<const float4 *>(a.t_lo + o + 64 * c);
                        const float th[4] = {h4.x, h4.y, h4.z, h4.w};
                        const float tl[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const float yh = y[c][b];
                            const float sm = yh - th[b];
                            const float bb = sm - yh;
                            const float e = (yh - (sm - bb)) + (-th[b] - bb);
                            y[c][b] = sm;
                            yl[c][b] += e - tl[b];
                        }
                    }
                }
                // y = R^{-T} (H r)_i / s; a row that is skipped keeps its codes
#pragma unroll
                for (int c = 0; c < NM; ++c)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const float v = (y[c][b] + yl[c][b]) / s;
                        y[c][b] = u[c][b] = live ? v : 0.f;
                    }
                if (!__any_sync(0xffffffffu, live)) continue;
#pragma unroll
                for (int c = 0; c < NM; ++c) qn[c] = qo[c];
                // back substitution (Eq. babai_update), quads in descending
                // order: 32 coordinates (eight quads, lanes of one half v of
                // the row) at a time
#pragma unroll
                for (int c = 2 * NM - 1; c >= 0; --c) {
                    const int m = c >> 1;            // the lanes' quad of these coordinates
                    const bool half = (k >> 3) == (c & 1);
                    const float4 rd4 = *reinterpret_cast<const float4 *>(Frd + 64 * m);
                    const float4 ta = *reinterpret_cast<const float4 *>(Ftri + 128 * m);
                    const float4 tb = *reinterpret_cast<const float4 *>(Ftri + 128 * m + 4);
                    float qc[4], qk[4], tn[4];
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        qc[b] = byte_float(qo[m], b);
                        qk[b] = tn[b] = __fadd_rn(qc[b], kRound);
                    }
                    // row h of the factor: vector 2 m2 + v of 32 entries for
                    // this lane's quad m2; with c even the lanes of the upper
                    // half have no entry in the last one (coordinates above
                    // h): they read the lower half's and multiply by zero
                    const bool above = !(c & 1) && k >= 8;
                    const float *Frow = F + factor_row(32 * c) + 4 * k;
                    const int last = 64 * m - (above ? 32 : 0);
#pragma unroll 1
                    for (int kk = 7; kk >= 0; --kk) {
                        const float *Fq = Frow + 4 * kk * 32 * (c + 1);
                        float4 L[4][NM];
#pragma unroll
                        for (int b = 3; b >= 0; --b)
#pragma unroll
                            for (int m2 = 0; m2 <= m; ++m2)
                                L[b][m2] = *reinterpret_cast<const float4 *>(
                                    Fq + b * 32 * (c + 1) + (m2 < m ? 64 * m2 : last));
                        // every lane decides its own quad m; the owner's is
                        // the one that counts
                        float dn[4], t[4];
                        auto decide = [&](float w, float rdl, int b) {
                            const float v = __fadd_rn(fmaf(w, rdl, qc[b]), kRound);
                            t[b] = fmaxf(fminf(v, rmax), kRound);
                            dn[b] = __fsub_rn(t[b], qk[b]);
                        };
                        float w2 = u[m][2], w1 = u[m][1], w0 = u[m][0];
                        decide(u[m][3], rd4.w, 3);
                        w2 = fmaf(-ta.x, dn[3], w2);
                        w1 = fmaf(-ta.y, dn[3], w1);
                        w0 = fmaf(-ta.z, dn[3], w0);
                        decide(w2, rd4.z, 2);
                        w1 = fmaf(-ta.w, dn[2], w1);
                        w0 = fmaf(-tb.x, dn[2], w0);
                        decide(w1, rd4.y, 1);
                        w0 = fmaf(-tb.y, dn[1], w0);
                        decide(w0, rd4.x, 0);
                        const bool mine = half && (k & 7) == kk;
                        u[m][2] = mine ? w2 : u[m][2];
                        u[m][1] = mine ? w1 : u[m][1];
                        u[m][0] = mine ? w0 : u[m][0];
                        const int src = 16 * (c & 1) + 2 * kk + sub;
#pragma unroll
                        for (int b = 3; b >= 0; --b) {
                            tn[b] = mine ? t[b] : tn[b];
                            dn[b] = __shfl_sync(0xffffffffu, dn[b], src);
                        }
#pragma unroll
                        for (int b = 3; b >= 0; --b)
#pragma unroll
                            for (int m2 = m; m2 >= 0; --m2) {
                                const float dl = (m2 == m && above) ? 0.f : dn[b];
                                u[m2][0] = fmaf(-L[b][m2].x, dl, u[m2][0]);
                                u[m2][1] = fmaf(-L[b][m2].y, dl, u[m2][1]);
                                u[m2][2] = fmaf(-L[b][m2].z, dl, u[m2][2]);
                                u[m2][3] = fmaf(-L[b][m2].w, dl, u[m2][3]);
                            }
                    }
                    // the low byte of the offset form is the code
                    const uint32_t qq = __byte_perm(
                        __byte_perm(__float_as_uint(tn[0]), __float_as_uint(tn[1]), 0x0040),
                        __byte_perm(__float_as_uint(tn[2]), __float_as_uint(tn[3]), 0x0040), 0x5410);
                    qn[m] = half ? qq : qn[m];
                }
                // acceptance
                float acc = 0.f;
#pragma unroll
                for (int c = 0; c < NM; ++c) {
                    const float4 dg = *reinterpret_cast<const float4 *>(Fdiag + 64 * c);
                    const float dgv[4] = {dg.x, dg.y, dg.z, dg.w};
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const float dq = byte_float(qn[c], b) - byte_float(qo[c], b);
                        const float av = dgv[b] * dq - u[c][b];
                        acc = fmaf(av - y[c][b], av + y[c][b], acc);
                    }
                }
                for (int o = 16; o >= 2; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                const float dF = s * s * acc;
                const bool keep = live && isfinite(dF) && dF < 0.f;
                unsigned kept = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    __half *cp = a.rv.cplane + (size_t)j * a.rv.d_pad + (size_t)i * g + 4 * k;
#pragma unroll
                    for (int c = 0; c < NM; ++c) {
                        __align__(8) __half hc[4];
#pragma unroll
                        for (int b = 0; b < 4; ++b)
                            hc[b] = __int2half_rn((int)((qn[c] >> (8 * b)) & 0xFFu) - z);
                        *reinterpret_cast<uint32_t *>(a.Q + off + 64 * c) = qn[c];
                        *reinterpret_cast<uint2 *>(cp + 64 * c) = *reinterpret_cast<const uint2 *>(hc);
                    }
                    if (k == 0) atomicAdd(a.accepted + j, 1);   // result unused: no wait
                }
                // the later groups of the block see the new codes
                if (n + 1 == a.nb) continue;
                while (kept) {                            // warp-uniform
                    const int rr = (__ffs(kept) - 1) & 1;
                    kept &= ~(0x55555555u << rr);
                    int cnt = 0;
#pragma unroll
                    for (int c = 0; c < NM; ++c)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const int dq = (int)((qn[c] >> (8 * b)) & 0xFFu) -
                                           (int)((qo[c] >> (8 * b)) & 0xFFu);
                            const bool nz = sub == rr && dq != 0;
                            const unsigned bal = __ballot_sync(0xffffffffu, nz);
                            if (nz)
                                list[cnt + __popc(bal & ((1u << lane) - 1u))] =
                                    dq * 256 + (64 * c + 4 * k + b);
                            cnt += __popc(bal);
                        }
                    __syncwarp();
                    const float sr = __shfl_sync(0xffffffffu, s, rr);
                    const size_t trow = (size_t)(base + rr) * ncol;
                    for (int n2 = n + 1; n2 < a.nb; ++n2)
                        add_changes<2 * NM, WIDE>(pairs + (size_t)(n2 - n - 1) * g * g, list, cnt, sr,
                                              a.expoT[(size_t)(a.i0 + n2) * G + i],
                                              a.t_hi + trow + n2 * g, a.t_lo + trow + n2 * g);
                    __syncwarp();
                }
            }
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(empty(slot));
                for (int t = 0; t < a.nb - 1 - n; ++t) tc::mbar_arrive(pempty(t));
            }
        }
    }
    // a copy that nobody waited for (after a wait gave up) must land before
    // the block ends; every other copy has been waited for above
    __syncthreads();
    if (*abort_f && threadIdx.x == 0) {
        for (int n = 0; n < a.nb; ++n) {
            (void)tc::mbar_wait<tc::kCloseIters>(full(n % kFactorSlots), (n / kFactorSlots) & 1);
            for (int t = 0; t < a.nb - 1 - n; ++t) (void)tc::mbar_wait<tc::kCloseIters>(pfull(t), n & 1);
        }
        atomicOr(a.status, ST_TIMEOUT);
    }
}

template <int NM, bool WIDE>
cudaError_t launch_rows(const BabaiArgs &a, cudaStream_t s) {
    constexpr int g = 64 * NM;
    // row warps spread evenly over the SMs, one block per SM
    const int nsm = num_sms();
    const int rw = (a.p + 1) / 2;
    const int passes = (rw + nsm * kMaxWarps - 1) / (nsm * kMaxWarps);
    const int warps = (rw + nsm * passes - 1) / (nsm * passes);
    const int blocks = (rw + warps * passes - 1) / (warps * passes);
    constexpr int smem = kFactorSlots * factor_floats(g) * 4 + pair_slots(g) * g * g * 8 +
                         kMaxWarps * g * 4;
    static_assert(smem <= 226 * 1024, "factors, pair blocks and lists must fit an SM's shared memory");
    static std::atomic<unsigned long long> attr_done{0};
    const cudaError_t e = set_max_dynamic_smem((const void *)babai_kernel<NM, WIDE>, smem, attr_done);
    if (e != cudaSuccess) return e;
    return launch_pdl(babai_kernel<NM, WIDE>, dim3(blocks), dim3(32 * (warps + 1)), (size_t)smem, s, a);
}

}  // namespace

cudaError_t launch_babai(float *t_hi, float *t_lo, const float *pt_hi, const float *pt_lo, int nsplit,
                         const float *Lf, const int2 *band, const int *expoT, const float *S,
                         uint8_t *Q, const int32_t *Z, ResidualView rv, const int *active,
                         int *accepted, int *status, int p, int g, int i0, int nb, int qmax,
                         float eps, cudaStream_t s) {
    if (p < 1 || nb < 1 || nb > sweep_block(g)) return cudaErrorInvalidValue;
    BabaiArgs a{t_hi, t_lo, pt_hi, pt_lo, nsplit, Lf, band, expoT, S, Q, Z, rv, active, accepted,
                status, p, i0, nb, qmax, eps};
    const bool wide = qmax > 15;
    if (g == 128) return wide ? launch_rows<2, true>(a, s) : launch_rows<2, false>(a, s);
    if (g == 64) return wide ? launch_rows<1, true>(a, s) : launch_rows<1, false>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace jarq
