// Joint scale solve (Sec. 3.3.1; App. E): one warp per output row for up to 32
// groups, one block of four warps per row for more.
//
// For each active row j the kernel
//  1. reads its G x G Gram matrix -- symmetric by construction, since the
//     Gram kernel computes each block once and writes it to both triangles,
//     so the symmetrisation of App. E "Solving for scales" is the identity
//     on it -- and forms, in double-float (the Gram entries arrive as
//     float pairs), the gradient g = rhs - Gram s_old of the current scales
//     (rhs_i = c_i^T P_i from the target projection) and the objective
//     F(s_old) = wHw - s_old^T (rhs + g);
//  2. factors the Gram matrix by Cholesky in float32 (the paper solves this
//     system in FP32).  A pivot at or below rcond * max(max diag, eps), a
//     nonfinite entry or a failed factorisation adds ridge * I and retries
//     once; a second failure marks the row numerical and keeps its state;
//  3. solves the normal equations of Eq. scale_normal_equations for the
//     increment of the scales: Gram s_new = rhs <=> Gram (s_new - s_old) = g,
//     and with the ridge (Gram + lambda I) delta = g - lambda s_old (float32
//     Cholesky, then two refinement steps whose residuals are formed in
//     double-float), and stores s_new rounded to float32;
//  4. evaluates L^{(k)} = F(s_new) = wHw - 2 s_new^T rhs + s_new^T Gram s_new
//     at the stored float32 scales and applies the early stop of Eq.
//     strict_stopping against L^{(k-1)}; with the ridge-acceptance option a
//     ridge-stabilised s_new that would raise F is dropped (App. G Remark
//     ridge-acceptance).
// In evaluation mode it only writes F(s) of the current state, for every
// row.
#include <float.h>

#include "df.cuh"
#include "tc_common.cuh"

namespace jarq {
namespace {

__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

struct SolveArgs {
    const float2 *gram;  // [p][G][G] Gram matrices as float pairs (hi, lo)
    const double *rhs, *wHw;
    float *S;
    double *L_prev;
    double *L_out;       // optional: F(s_old) of every processed row
    int *active, *iters, *ridge, *rstat, *status;
    int p, d, g, k;
    bool eval_only;
    jarq_options o;
};

// ---------------------------------------------------------------------------
// Solve for G > 32 (e.g. 64 groups of the 4096-input layers at g = 64, 86 of the
// 11008-input ones): a block of NT = 64, 96 or 128 threads per row (G rounded
// up), thread t owning row t of the Gram matrix.  The matrix stays in global
// memory (L2) and is read column by column, 16 coalesced loads in flight
// (exactly symmetric, so entry (t, c) is read as (c, t)): once for the gradient
// and the float32 copy, twice for the refinement residuals, once for the
// objective.  The float32 factor lives in shared memory and is formed in panels
// of eight columns: the first warp factors the 8 x 8 diagonal block, every
// thread solves its row of the panel, and 4 x 4 tiles take the rank-8 update of
// the trailing triangle.
// Every dot product with the Gram matrix -- the gradient, the two refinement
// residuals, the objective -- is summed in double-float on the entries' float
// pairs.
//
// What bounds it: the latency of a row's chain (8 to 11 panels, as many steps of
// each triangular solve, four passes over the matrix) against the rows that fit
// an SM (12, 8 or 6 by registers).  4096 rows: 213 us for 64 groups, 427 us for
// 86.  One warp per row, the trailing triangle updated a column at a time, took
// 324 and 800 us; both divide by the pivots and add in the same order, so the
// factor and the ridge decision are those of that kernel bit for bit (with
// products by the pivots' reciprocals: 181 and 367 us, but other last bits).
// ---------------------------------------------------------------------------

constexpr int kPanel = 8;

// Row pitch of the float32 factor: a multiple of 4 that is 4 mod 8, so that 16-
// byte loads of consecutive rows fall into different banks.
__host__ __device__ inline int solve_ld(int G) { return (G + 7) / 8 * 8 + 4; }
__host__ __device__ inline size_t solve_bytes(int G) {
    const int Gp = (G + 7) / 8 * 8;
    return ((size_t)Gp * solve_ld(G) + 7 * Gp) * sizeof(float);
}

// Row t of the Gram matrix times x = xh + xl (xl null: x = xh), in double-float.
// COPY: also the float32 entries on and below the diagonal into A, entry (c, t)
// for t <= c, with `finite` false if any entry is not.
template <bool COPY>
__device__ __forceinline__ DF big_dot(const float2 *gj, int G, int t, const float *xh, const float *xl,
                                      float *A, int ld, bool &finite) {
    DF acc{0.f, 0.f};
    constexpr int kU = 16;
    for (int c0 = 0; c0 < G; c0 += kU) {
        float2 v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            v[u] = c0 + u < G ? __ldg(gj + (size_t)(c0 + u) * G + t) : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int c = c0 + u;
            if (c >= G) break;               // uniform
            df_add_prod(acc, v[u].x, xh[c]);
            acc.l = fmaf(v[u].y, xh[c], acc.l);
            if (xl) acc.l = fmaf(v[u].x, xl[c], acc.l);
            if (COPY) {
                if (t <= c) A[c * ld + t] = v[u].x;
                finite &= (bool)isfinite(v[u].x);
            }
        }
    }
    return acc;
}

// Sum of one DF per thread, the same in every thread.
template <int NT>
__device__ __forceinline__ DF block_sum(DF v, DF *red) {
    v = df_warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    DF s = red[0];
    for (int w = 1; w < NT / 32; ++w) s = df_add(s, red[w]);
    return s;
}

__device__ __forceinline__ void load_row8(const float *p, float (&l)[kPanel]) {
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    l[0] = a.x; l[1] = a.y; l[2] = a.z; l[3] = a.w;
    l[4] = b.x; l[5] = b.y; l[6] = b.z; l[7] = b.w;
}

// In-place lower Cholesky of A (rows and columns beyond G are not touched),
// rd[a] = 1 / L_aa.  False (in every thread) when a pivot is not above `thr` or
// not finite.
template <int NT>
__device__ bool big_cholesky(float *A, int ld, int G, float thr, float *rd, int *flag) {
    const int t = threadIdx.x, lane = t & 31;
    if (t == 0) *flag = 1;
    for (int k0 = 0; k0 < G; k0 += kPanel) {
        const int nk = min(kPanel, G - k0);
        __syncthreads();
        if (t < 32) {
            // lane r < 8: row k0 + r of the diagonal block
            float a[kPanel];
#pragma unroll
            for (int c = 0; c < kPanel; ++c)
                a[c] = (lane < nk && c <= lane) ? A[(k0 + lane) * ld + k0 + c] : 0.f;
            bool good = true;
            float inv = 0.f;
#pragma unroll
            for (int k = 0; k < kPanel; ++k) {
                if (k < nk) {                       // uniform
                    const float piv = __shfl_sync(0xffffffffu, a[k], k);
                    good = good && piv > thr && isfinite(piv);
                    const float l = sqrtf(piv);
                    if (lane == k) {
                        a[k] = l;
                        inv = 1.0f / l;
                    }
                    if (lane > k) a[k] /= l;
#pragma unroll
                    for (int c = k + 1; c < kPanel; ++c) {
                        const float lc = __shfl_sync(0xffffffffu, a[k], c);
                        if (lane >= c) a[c] = fmaf(-a[k], lc, a[c]);
                    }
                }
            }
            if (lane < nk) {
                rd[k0 + lane] = inv;
#pragma unroll
                for (int c = 0; c < kPanel; ++c)
                    if (c <= lane) A[(k0 + lane) * ld + k0 + c] = a[c];
            }
            if (!good && lane == 0) *flag = 0;
        }
        __syncthreads();
        if (!*flag) return false;                   // uniform
        const int k1 = k0 + kPanel;
        // rows below: x L_kk^T = a
        if (t >= k1 && t < G) {
            float x[kPanel];
            float4 *row = reinterpret_cast<float4 *>(A + t * ld + k0);
            const float4 p0 = row[0], p1 = row[1];
            x[0] = p0.x; x[1] = p0.y; x[2] = p0.z; x[3] = p0.w;
            x[4] = p1.x; x[5] = p1.y; x[6] = p1.z; x[7] = p1.w;
#pragma unroll
            for (int c = 0; c < kPanel; ++c) {
                float l[kPanel];
                load_row8(A + (k0 + c) * ld + k0, l);
#pragma unroll
                for (int k = 0; k < c; ++k) x[c] = fmaf(-x[k], l[k], x[c]);
                x[c] /= l[c];
            }
            row[0] = make_float4(x[0], x[1], x[2], x[3]);
            row[1] = make_float4(x[4], x[5], x[6], x[7]);
        }
        __syncthreads();
        // trailing triangle, 4 x 4 tiles (i, j), j <= i
        const int nt = (G - k1 + 3) / 4;
        for (int e = t; e < nt * (nt + 1) / 2; e += NT) {
            int i = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
            if ((i + 1) * (i + 2) / 2 <= e) ++i;
            if (i * (i + 1) / 2 > e) --i;
            const int j = e - i * (i + 1) / 2;
            const float *pa = A + (k1 + 4 * i) * ld + k0, *pb = A + (k1 + 4 * j) * ld + k0;
            float *pc = A + (k1 + 4 * i) * ld + k1 + 4 * j;
            float4 b0[4], b1[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                b0[c] = *reinterpret_cast<const float4 *>(pb + c * ld);
                b1[c] = *reinterpret_cast<const float4 *>(pb + c * ld + 4);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 a0 = *reinterpret_cast<const float4 *>(pa + r * ld);
                const float4 a1 = *reinterpret_cast<const float4 *>(pa + r * ld + 4);
                float4 c4 = *reinterpret_cast<const float4 *>(pc + r * ld);
                float cv[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    cv[c] = fmaf(-a0.x, b0[c].x, cv[c]);
                    cv[c] = fmaf(-a0.y, b0[c].y, cv[c]);
                    cv[c] = fmaf(-a0.z, b0[c].z, cv[c]);
                    cv[c] = fmaf(-a0.w, b0[c].w, cv[c]);
                    cv[c] = fmaf(-a1.x, b1[c].x, cv[c]);
                    cv[c] = fmaf(-a1.y, b1[c].y, cv[c]);
                    cv[c] = fmaf(-a1.z, b1[c].z, cv[c]);
                    cv[c] = fmaf(-a1.w, b1[c].w, cv[c]);
                }
                *reinterpret_cast<float4 *>(pc + r * ld) = make_float4(cv[0], cv[1], cv[2], cv[3]);
            }
        }
    }
    __syncthreads();
    return true;
}

// v <- (L L^T)^{-1} v, thread t holding v_t; x [Gp] is shared scratch.  Per panel
// every thread solves the 8 x 8 block for itself (rows beyond G are zero, their
// reciprocal pivots too) and updates its own entry.
__device__ float big_chol_solve(const float *A, int ld, int G, const float *rd, float *x, float v) {
    const int t = threadIdx.x;
    for (int k0 = 0; k0 < G; k0 += kPanel) {
        if (t >= k0 && t < k0 + kPanel) x[t] = v;
        __syncthreads();
        float s[kPanel], r[kPanel];
        load_row8(x + k0, s);
        load_row8(rd + k0, r);
#pragma unroll
        for (int c = 0; c < kPanel; ++c) {
            float l[kPanel];
            load_row8(A + (k0 + c) * ld + k0, l);
#pragma unroll
            for (int k = 0; k < c; ++k) s[c] = fmaf(-l[k], s[k], s[c]);
            s[c] *= r[c];
            if (t == k0 + c) v = s[c];
        }
        if (t >= k0 + kPanel && t < G) {
            float l[kPanel];
            load_row8(A + t * ld + k0, l);
#pragma unroll
            for (int k = 0; k < kPanel; ++k) v = fmaf(-l[k], s[k], v);
        }
    }
    __syncthreads();        // the last panel's x is written again below
    for (int k0 = (G - 1) / kPanel * kPanel; k0 >= 0; k0 -= kPanel) {
        if (t >= k0 && t < k0 + kPanel) x[t] = v;
        __syncthreads();
        float s[kPanel], r[kPanel];
        load_row8(x + k0, s);
        load_row8(rd + k0, r);
#pragma unroll
        for (int c = kPanel - 1; c >= 0; --c) {
            // x_c is final: take it out of the rows above (columns k < c of row c)
            s[c] *= r[c];
            if (t == k0 + c) v = s[c];
            float l[kPanel];
            load_row8(A + (k0 + c) * ld + k0, l);
#pragma unroll
            for (int k = 0; k < c; ++k) s[k] = fmaf(-l[k], s[c], s[k]);
        }
        if (t < k0) {
#pragma unroll
            for (int k = kPanel - 1; k >= 0; --k) v = fmaf(-A[(k0 + k) * ld + t], s[k], v);
        }
    }
    return v;
}

template <int NT>
__global__ void __launch_bounds__(NT, 768 / NT) scale_solve_kernel(SolveArgs a) {
    extern __shared__ __align__(16) float fsm[];
    __shared__ DF red[NT / 32];
    __shared__ int flag;
    const int G = a.d / a.g, Gp = (G + 7) / 8 * 8, ld = solve_ld(G);
    const int j = blockIdx.x, t = threadIdx.x, tc = min(t, G - 1);
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    if (!a.eval_only && !a.active[j]) return;   // uniform
    const bool own = t < G;
    float *A = fsm;                      // [Gp][ld]
    float *so = A + Gp * ld;             // s_old, later s_new
    float *rd = so + Gp, *x = rd + Gp;   // reciprocal pivots; solve scratch
    float *ih = x + Gp, *il = ih + Gp;   // increment of the scales (double-float)
    const float2 *gj = a.gram + (size_t)j * G * G;
    const float s_old = own ? a.S[(size_t)j * G + t] : 0.f;
    const DF rh = own ? split_double(a.rhs[(size_t)j * G + t]) : DF{0.f, 0.f};
    if (own) so[t] = s_old;
    // the rows that pad the last panel; what stands right of the diagonal, the
    // columns from G on included, is never read into an entry on or below it
    for (int e = G * ld + t; e < Gp * ld; e += NT) A[e] = 0.f;
    if (t >= G && t < Gp) rd[t] = 0.f;
    __syncthreads();
    // gradient g = rhs - Gram s_old and F(s_old) = wHw - s_old^T (rhs + g)
    bool finite = true;
    const DF gs0 = big_dot<true>(gj, G, tc, so, nullptr, A, ld, finite);
    const DF gd = df_add(rh, df_neg(gs0));
    const bool bfin = !own || isfinite(gd.h);
    DF fs{0.f, 0.f};
    if (own) {
        const DF rg = df_add(rh, gd);
        df_add_prod(fs, s_old, rg.h);
        fs.l = fmaf(s_old, rg.l, fs.l);
    }
    const double F_old = a.wHw[j] - df_to_double(block_sum<NT>(fs, red));
    if (a.L_out && t == 0) a.L_out[j] = F_old;
    if (a.eval_only) return;
    if (a.o.fixed_grid) {
        // fixed grid: the scales stay; L^(k) is the objective of the current state
        if (t == 0) {
            bool stop = false;
            if (a.o.early_stop && a.k >= 2) {
                const double dec = a.L_prev[j] - F_old;
                const double den = fmax(fabs(a.L_prev[j]), (double)a.o.eps);
                stop = (dec / den <= (double)a.o.tau_rel) || (fabs(dec) <= (double)a.o.tau_abs);
            }
            a.L_prev[j] = F_old;
            a.iters[j] = a.k;
            if (stop) a.active[j] = 0;
        }
        return;
    }
    // float32 factor (the high part of a pair is the correctly rounded float32
    // of the entry), with the ridge retry
    finite = __syncthreads_and(finite);
    __shared__ float wmax[NT / 32];
    {
        const float m = warp_max(own ? A[t * ld + t] : 0.f);
        if ((t & 31) == 0) wmax[t >> 5] = m;
    }
    __syncthreads();
    float md = wmax[0];
    for (int w = 1; w < NT / 32; ++w) md = fmaxf(md, wmax[w]);
    bool ok = finite && big_cholesky<NT>(A, ld, G, a.o.rcond * fmaxf(md, a.o.eps), rd, &flag);
    int used_ridge = 0;
    if (!ok) {                                  // uniform
        used_ridge = 1;
        __syncthreads();
        if (own)
            for (int c = t; c < G; ++c) A[c * ld + t] = __ldg(gj + (size_t)c * G + t).x + (c == t ? a.o.ridge : 0.f);
        for (int e = G * ld + t; e < Gp * ld; e += NT) A[e] = 0.f;
        __syncthreads();
        ok = big_cholesky<NT>(A, ld, G, 0.f, rd, &flag);
    }
    ok = __syncthreads_and(ok && bfin);
    auto fail = [&]() {
        if (t == 0) {
            a.ridge[j] += used_ridge;
            a.rstat[j] = JARQ_ERR_NUMERICAL;
            a.active[j] = 0;
            atomicOr(a.status, ST_NUMERICAL);
        }
    };
    if (!ok) {
        fail();
        return;
    }
    // (Gram + lambda I) inc = g - lambda s_old, refined twice with
    // double-float residuals
    const float lam = used_ridge ? a.o.ridge : 0.f;
    DF rhs0 = gd;
    df_add_prod(rhs0, -lam, s_old);
    DF inc{0.f, 0.f};
    float y = own ? __fadd_rn(rhs0.h, rhs0.l) : 0.f;
    for (int step = 0; step < 3; ++step) {
        y = big_chol_solve(A, ld, G, rd, x, y);
        if (own) {
            inc = df_add(inc, DF{y, 0.f});
            ih[t] = inc.h;
            il[t] = inc.l;
        }
        if (step == 2) break;
        __syncthreads();
        // res = g - lambda (s_old + inc) - Gram inc
        DF res = rhs0;
        df_add_prod(res, -lam, inc.h);
        res.l = fmaf(-lam, inc.l, res.l);
        bool f2 = true;
        res = df_add(res, df_neg(big_dot<false>(gj, G, tc, ih, il, nullptr, 0, f2)));
        y = own ? __fadd_rn(res.h, res.l) : 0.f;
        __syncthreads();
    }
    if (!__syncthreads_and(!own || (isfinite(inc.h) && isfinite(inc.l)))) {
        fail();
        return;
    }
    // s_new = s_old + inc, rounded once to float32
    float sn = 0.f;
    if (own) {
        const DF s2 = df_add({s_old, 0.f}, inc);
        sn = __fadd_rn(s2.h, s2.l);
        so[t] = sn;
    }
    __syncthreads();
    // L^{(k)} at the stored float32 scales, from the unridged Gram matrix
    bool f2 = true;
    const DF gs = big_dot<false>(gj, G, tc, so, nullptr, nullptr, 0, f2);
    DF t1{0.f, 0.f}, t2{0.f, 0.f};
    if (own) {
        df_add_prod(t1, sn, rh.h);
        t1.l = fmaf(sn, rh.l, t1.l);
        df_add_prod(t2, sn, gs.h);
        t2.l = fmaf(sn, gs.l, t2.l);
    }
    t1 = block_sum<NT>(t1, red);
    t2 = block_sum<NT>(t2, red);
    double L_new = a.wHw[j] - 2.0 * df_to_double(t1) + df_to_double(t2);
    // Remark ridge-acceptance (optional): a ridge-stabilised solve that would
    // raise F_j is dropped and the previous scales stay
    const bool keep_old = used_ridge && a.o.ridge_accept && !(L_new <= F_old);
    if (keep_old) L_new = F_old;
    if (!keep_old && own) a.S[(size_t)j * G + t] = sn;
    if (t == 0) {
        bool stop = false;
        if (a.o.early_stop && a.k >= 2) {
            const double dec = a.L_prev[j] - L_new;
            const double den = fmax(fabs(a.L_prev[j]), (double)a.o.eps);
            stop = (dec / den <= (double)a.o.tau_rel) || (fabs(dec) <= (double)a.o.tau_abs);
        }
        a.L_prev[j] = L_new;
        a.iters[j] = a.k;
        a.ridge[j] += used_ridge;
        if (stop) a.active[j] = 0;
    }
}

// ---------------------------------------------------------------------------
// Register-resident solve for G <= 32 (the g = 128 layers of 4096 inputs).
//
// Same steps, same decisions, no bulk float64: on GB300 float64 runs at
// about 1/64 of the float32 rate, so the dot products of the gradient, the
// refinement residuals and the objective are done in double-float (pairs of
// float32 with error-free products and sums, about 48 significant bits).
// Lane l owns row l of the Gram matrix (= column l: it is exactly
// symmetric) as the double-float pair per entry that the Gram kernel
// stores.  The float32 Cholesky keeps row l in registers and
// broadcasts the column of each step with shuffles.  The triangular solves
// multiply by the reciprocal of the pivots; the refinement makes the stored
// scales independent of that rounding.
// ---------------------------------------------------------------------------

// In-place lower Cholesky with lane a holding row a in A[].
__device__ __forceinline__ bool reg_cholesky(float (&A)[32], int G, float thr) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (k < G) {
            const float piv = __shfl_sync(0xffffffffu, A[k], k);
            if (!(piv > thr) || !isfinite(piv)) return false;   // warp-uniform
            const float lkk = sqrtf(piv);
            float lak = 0.f;
            if (lane > k) lak = A[k] / lkk;
            if (lane == k) A[k] = lkk;
            if (lane > k) A[k] = lak;
            // the entries above the diagonal (b > a) are never read again, so
            // they take the update as well instead of a predicate per entry
#pragma unroll
            for (int b = k + 1; b < 32; ++b) {
                const float lbk = __shfl_sync(0xffffffffu, lak, b);
                A[b] = fmaf(-lak, lbk, A[b]);
            }
        }
    }
    return true;
}

// y <- (L L^T)^{-1} y with lane a holding y_a; L row-major in Ls (stride
// 33) with zeros above the diagonal, dinv = 1 / L_aa.
__device__ __forceinline__ float reg_chol_solve(const float *Ls, int G, float dinv, float y) {
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int k = 0; k < G; ++k) {
        const float yk = __shfl_sync(0xffffffffu, __fmul_rn(y, dinv), k);
        const float t = fmaf(-Ls[lane * 33 + k], yk, y);   // lanes a < k: L_ak = 0
        y = lane == k ? yk : t;
    }
#pragma unroll 4
    for (int k = G - 1; k >= 0; --k) {
        const float xk = __shfl_sync(0xffffffffu, __fmul_rn(y, dinv), k);
        const float t = fmaf(-Ls[k * 33 + lane], xk, y);   // lanes a > k: L_ka = 0
        y = lane == k ? xk : t;
    }
    return y;
}

constexpr int kSmallWarps = 4;   // rows (warps) per block of the G <= 32 kernel

__global__ void __launch_bounds__(32 * kSmallWarps, 4) scale_solve_small_kernel(SolveArgs a) {
    __shared__ float Lsh[kSmallWarps][32 * 33];
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    const int G = a.d / a.g;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.x * kSmallWarps + w;
    if (j >= a.p) return;  // warp-uniform
    const bool own = lane < G;
    const float2 *gj = a.gram + (size_t)j * G * G;
    // row `lane` of the Gram matrix, read column-wise (coalesced) by
    // symmetry: every load (and the row's active flag) is issued before the
    // first is used
    const int act = a.eval_only ? 1 : a.active[j];
    DF gr[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        const float2 e = (own && c < G) ? gj[(size_t)c * G + lane] : make_float2(0.f, 0.f);
        gr[c] = DF{e.x, e.y};
    }
    const float so = own ? a.S[(size_t)j * G + lane] : 0.f;
    const double rhs_d = own ? a.rhs[(size_t)j * G + lane] : 0.0;
    if (!act) return;  // warp-uniform
    const DF rh = split_double(rhs_d);

    // gradient g = rhs - Gram s_old and F(s_old) = wHw - s_old^T (rhs + g)
    DF acc{0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        if (c < G) {
            const float sc = __shfl_sync(0xffffffffu, so, c);
            df_add_prod(acc, gr[c].h, sc);
            acc.l = __fmaf_rn(gr[c].l, sc, acc.l);
        }
    }
    const DF gd = df_add(rh, df_neg(acc));
    const bool bfin = isfinite(gd.h) && isfinite(gd.l);
    DF fs{0.f, 0.f};
    {
        const DF t = df_add(rh, gd);
        df_add_prod(fs, so, t.h);
        fs.l = __fmaf_rn(so, t.l, fs.l);
    }
    const double F_old = a.wHw[j] - df_to_double(df_warp_sum(fs));
    if (a.L_out && lane == 0) a.L_out[j] = F_old;
    if (a.eval_only) return;
    if (a.o.fixed_grid) {
        bool stop = false;
        if (a.o.early_stop && a.k >= 2) {
            const double dec = a.L_prev[j] - F_old;
            const double den = fmax(fabs(a.L_prev[j]), (double)a.o.eps);
            stop = (dec / den <= (double)a.o.tau_rel) || (fabs(dec) <= (double)a.o.tau_abs);
        }
        if (lane == 0) {
            a.L_prev[j] = F_old;
            a.iters[j] = a.k;
            if (stop) a.active[j] = 0;
        }
        return;
    }

    // float32 factor of the Gram matrix (entries rounded to nearest, as a
    // float64 -> float32 conversion does), with the ridge retry
    float A[32];
    bool finite = true;
    float diag = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        A[c] = gr[c].h;
        finite &= (bool)isfinite(A[c]);
        if (c == lane) diag = A[c];
    }
    finite = __all_sync(0xffffffffu, finite);
    const float md = warp_max(own ? diag : 0.f);
    bool ok = finite && reg_cholesky(A, G, a.o.rcond * fmaxf(md, a.o.eps));
    int used_ridge = 0;
    if (!ok) {
        used_ridge = 1;
#pragma unroll
        for (int c = 0; c < 32; ++c) A[c] = (c == lane) ? gr[c].h + a.o.ridge : gr[c].h;
        ok = reg_cholesky(A, G, 0.f);
    }
    ok = ok && __all_sync(0xffffffffu, bfin);
    auto fail = [&]() {
        if (lane == 0) {
            a.ridge[j] += used_ridge;
            a.rstat[j] = JARQ_ERR_NUMERICAL;
            a.active[j] = 0;
            atomicOr(a.status, ST_NUMERICAL);
        }
    };
    if (!ok) {
        fail();
        return;
    }
    float *Ls = Lsh[w];
    float ldiag = 1.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        Ls[lane * 33 + c] = c <= lane ? A[c] : 0.f;
        if (c == lane) ldiag = A[c];
    }
    __syncwarp();
    const float dinv = own ? 1.0f / ldiag : 0.f;

    // (Gram + lambda I) inc = g - lambda s_old, refined twice with
    // double-float residuals
    const float lam = used_ridge ? a.o.ridge : 0.f;
    DF b = gd;
    if (used_ridge) {
        df_add_prod(b, -lam, so);
    }
    DF inc{0.f, 0.f};
    float y = own ? __fadd_rn(b.h, b.l) : 0.f;
    for (int step = 0; step < 3; ++step) {
        y = reg_chol_solve(Ls, G, dinv, y);
        if (!own) y = 0.f;
        inc = df_add(inc, DF{y, 0.f});
        if (step == 2) break;
        DF res = b;
        if (used_ridge) {
            df_add_prod(res, -lam, inc.h);
            res.l = __fmaf_rn(-lam, inc.l, res.l);
        }
        DF q{0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            if (c < G) {
                const float ih = __shfl_sync(0xffffffffu, inc.h, c);
                const float il = __shfl_sync(0xffffffffu, inc.l, c);
                df_add_prod(q, gr[c].h, ih);
                q.l = __fmaf_rn(gr[c].h, il, q.l);
                q.l = __fmaf_rn(gr[c].l, ih, q.l);
            }
        }
        res = df_add(res, df_neg(q));
        y = own ? __fadd_rn(res.h, res.l) : 0.f;
    }
    if (!__all_sync(0xffffffffu, isfinite(inc.h) && isfinite(inc.l))) {
        fail();
        return;
    }
    // s_new = float32(s_old + inc)
    float sn = 0.f;
    if (own) {
        const DF t = df_two_sum(so, inc.h);
        sn = __fadd_rn(t.h, __fadd_rn(t.l, inc.l));
    }
    // L^{(k)} = wHw - 2 s^T rhs + s^T Gram s at the stored float32 scales
    DF gs{0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        if (c < G) {
            const float sc = __shfl_sync(0xffffffffu, sn, c);
            df_add_prod(gs, gr[c].h, sc);
            gs.l = __fmaf_rn(gr[c].l, sc, gs.l);
        }
    }
    DF t1{0.f, 0.f}, t2{0.f, 0.f};
    df_add_prod(t1, sn, rh.h);
    t1.l = __fmaf_rn(sn, rh.l, t1.l);
    df_add_prod(t2, sn, gs.h);
    t2.l = __fmaf_rn(sn, gs.l, t2.l);
    t1 = df_warp_sum(t1);
    t2 = df_warp_sum(t2);
    double L_new = a.wHw[j] - 2.0 * df_to_double(t1) + df_to_double(t2);
    const bool keep_old = used_ridge && a.o.ridge_accept && !(L_new <= F_old);
    if (keep_old) L_new = F_old;
    bool stop = false;
    if (a.o.early_stop && a.k >= 2) {
        const double dec = a.L_prev[j] - L_new;
        const double den = fmax(fabs(a.L_prev[j]), (double)a.o.eps);
        stop = (dec / den <= (double)a.o.tau_rel) || (fabs(dec) <= (double)a.o.tau_abs);
    }
    if (!keep_old && own) a.S[(size_t)j * G + lane] = sn;
    if (lane == 0) {
        a.L_prev[j] = L_new;
        a.iters[j] = a.k;
        a.ridge[j] += used_ridge;
        if (stop) a.active[j] = 0;
    }
}

template <int NT>
cudaError_t launch_big(const SolveArgs &a, bool pdl, cudaStream_t s) {
    static std::atomic<unsigned long long> attr_done{0};
    const cudaError_t e =
        set_max_dynamic_smem((const void *)scale_solve_kernel<NT>, (int)solve_bytes(NT), attr_done);
    if (e != cudaSuccess) return e;
    return launch_k(scale_solve_kernel<NT>, dim3(a.p), dim3(NT), solve_bytes(a.d / a.g), s, pdl, a);
}

}  // namespace

cudaError_t launch_scale_solve(const float2 *gram, const double *rhs, const double *wHw, float *S,
                               double *L_prev, double *L_out, int *active,
                               int *iters, int *ridge, int *rstat, int *status, int p, int d,
                               int g, int k, bool eval_only, const jarq_options &o,
                               cudaStream_t s, bool pdl) {
    const int G = d / g;
    SolveArgs a{gram, rhs, wHw, S, L_prev, L_out, active, iters, ridge, rstat,
                status, p, d, g, k, eval_only, o};
    if (G <= 32)
        return launch_k(scale_solve_small_kernel, dim3((p + kSmallWarps - 1) / kSmallWarps),
                        dim3(32 * kSmallWarps), 0, s, pdl, a);
    if (G <= 64) return launch_big<64>(a, pdl, s);
    if (G <= 96) return launch_big<96>(a, pdl, s);
    return launch_big<128>(a, pdl, s);
}

}  // namespace jarq
