// C ABI entry points: handle lifecycle, argument checks, staging of host
// buffers and the refinement loop (Sec. 3.3; App. E "Order of updates").
//
// Once per call: the target projection P = W H, w^T H w and the folded
// projection Pt_i = R_i^{-T} P_i (App. G "Computational Complexity",
// target-projection shortcut).  Per iteration k = 1..K: the Gram matrices of
// the current codes and rhs_i = c_i^T P_i, the joint scale solve (gradient
// rhs - Gram s, objective, early stop), and one Gauss-Seidel sweep over the
// groups in blocks of a few: the targets' products T_i of a block, then its
// Babai steps on y = (Pt_i - T_i) / s_i.
#include <float.h>
#include <stdlib.h>
#include <string.h>

#include <memory>
#include <vector>

#include <new>

#include "jarq_internal.cuh"

namespace jarq {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 2D tensor map of 2-byte elements (bf16 or fp16) over [rows][cols]
// (pitch = cols), box_rows x 64 boxes with 128-byte swizzle or box_rows x 32
// boxes with 64-byte swizzle, out-of-range elements read as zero.
cudaError_t make_tmap_2b(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                         uint32_t box_rows, CUtensorMapDataType dtype, uint32_t box_cols) {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                                         cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !ptr)
            return e != cudaSuccess ? e : cudaErrorSymbolNotFound;
        fn = (EncodeTiledFn)ptr;
    }
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(m, dtype, 2, const_cast<void *>(base), dims, strides,
                    box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t make_tmap_bf16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                           uint32_t box_rows, uint32_t box_cols) {
    return make_tmap_2b(m, base, rows, cols, box_rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, box_cols);
}

cudaError_t make_tmap_f16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                          uint32_t box_rows) {
    return make_tmap_2b(m, base, rows, cols, box_rows, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 64);
}

}  // namespace jarq

using namespace jarq;

namespace {

jarq_status cuda_fail(cudaError_t e) {
    return e == cudaErrorMemoryAllocation ? JARQ_ERR_NOMEM : JARQ_ERR_CUDA;
}

#define CK(x)                                  \
    do {                                       \
        cudaError_t e_ = (x);                  \
        if (e_ != cudaSuccess) {               \
            (void)cudaGetLastError();          \
            return cuda_fail(e_);              \
        }                                      \
    } while (0)

// Launch `call` (which enqueues `n` kernels on stream `strm`) under the
// profiling scope `name`.
#define RUN_ON(name, n, strm, call)     \
    do {                                \
        ProfScope ps_(name, strm);      \
        CK(call);                       \
        ps_.done();                     \
        count_launches(n);              \
    } while (0)
#define RUN(name, n, call) RUN_ON(name, n, st, call)

template <class T>
cudaError_t dalloc(T **p, size_t n) {
    *p = nullptr;
    if (n == 0) n = 1;
    return cudaMalloc((void **)p, n * sizeof(T));
}

bool is_device_ptr(const void *ptr) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Lays arrays out in one allocation: a first pass without memory adds up the
// sizes, a second one hands out the pieces.  One cudaMalloc and cudaFree
// instead of one per array: on a 4096 x 4096 layer, preparing a Hessian went
// from 3.5 to 3.1 ms, its first layer from 0.74 to 0.2 ms above a later one,
// and the release from 1.8 to 1.1 ms.
struct Arena {
    char *base = nullptr;
    size_t used = 0;
    template <class T>
    void take(T *&ptr, size_t n) {
        ptr = base ? reinterpret_cast<T *>(base + used) : nullptr;
        used += (n * sizeof(T) + 255) / 256 * 256;
    }
};

void free_ws(Workspace &w) {
    cudaFree(w.mem);
    cudaFree(w.sW);
    cudaFree(w.sS);
    cudaFree(w.sQ);
    cudaFree(w.sZ);
    w = Workspace{};
}

void layout_ws(Arena &m, Workspace &w, const jarq_hessian *h, int p, int p_pad) {
    const size_t d = h->din, G = h->G, pd = (size_t)p_pad * h->d_pad, np = p;
    m.take(w.rplanes, 3 * pd);
    m.take(w.cplane, pd);
    m.take(w.wdig, 6 * pd);
    m.take(w.Hr, np * d);
    m.take(w.r, np * d);
    m.take(w.gram, np * G * G);
    m.take(w.rhs, np * G);
    // partials of a product: one slot of 256 columns (a block of the sweep) a
    // row, or more slots while the CTAs of 128 rows x 64 columns fit the SMs
    // (target_splits), for this row count and every smaller one
    size_t t_len = (size_t)p_pad * 256;
    if (t_len < (size_t)num_sms() * 128 * 64) t_len = (size_t)num_sms() * 128 * 64;
    m.take(w.t_hi, t_len);
    m.take(w.t_lo, t_len);
    m.take(w.Pt_hi, np * d);
    m.take(w.Pt_lo, np * d);
    m.take(w.wexp, np * G);
    m.take(w.Phi, np * d);
    m.take(w.Plo, np * d);
    m.take(w.wHw, np);
    m.take(w.aux, np);
    m.take(w.own, np * G);
    m.take(w.L_prev, np);
    m.take(w.L_host, np);
    m.take(w.L_final, np);
    m.take(w.active, np);
    m.take(w.iters, np);
    m.take(w.accepted, np);
    m.take(w.ridge, np);
    m.take(w.rstat, np);
}

cudaError_t ensure_ws(jarq_hessian *h, int p, cudaStream_t st) {
    Workspace &w = h->ws;
    if (p <= w.cap_rows) return cudaSuccess;
    free_ws(w);
    const int p_pad = round_up(p, 128);
    Arena m;
    layout_ws(m, w, h, p, p_pad);
    cudaError_t e = dalloc(&m.base, m.used);
    if (e != cudaSuccess) return e;
    w.mem = m.base;
    m.used = 0;
    layout_ws(m, w, h, p, p_pad);
    // columns beyond din are read as zeros by the products; rows beyond p only
    // reach results that nobody reads
    if (h->d_pad != h->din) {
        const size_t pd = (size_t)p_pad * h->d_pad;
        if ((e = cudaMemsetAsync(w.rplanes, 0, 3 * pd * 2, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(w.cplane, 0, pd * 2, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(w.wdig, 0, 6 * pd * 2, st)) != cudaSuccess) return e;
    }
    if ((e = make_tmap_bf16(&w.mapR, w.rplanes, (uint64_t)3 * p_pad, h->d_pad, 128)) != cudaSuccess)
        return e;
    if ((e = make_tmap_f16(&w.mapC, w.cplane, (uint64_t)p_pad, h->d_pad, 128)) != cudaSuccess)
        return e;
    if ((e = make_tmap_bf16(&w.mapWd, w.wdig, (uint64_t)4 * p_pad, h->d_pad, 128, 32)) != cudaSuccess)
        return e;
    if ((e = make_tmap_bf16(&w.mapPd, w.wdig, (uint64_t)6 * p_pad, h->d_pad, 128, 32)) != cudaSuccess)
        return e;
    w.p_pad = p_pad;
    w.cap_rows = p;
    return cudaSuccess;
}

// Device views of the four layer arguments, staging host buffers.
struct LayerArgs {
    const float *W;
    float *S;
    uint8_t *Q;
    const int32_t *Z;
    bool hS = false, hQ = false;  // S / Q came from host memory
};

cudaError_t stage_layer(jarq_hessian *h, const float *W, const float *S, const uint8_t *Q,
                        const int32_t *Z, int p, LayerArgs &out, cudaStream_t st) {
    Workspace &w = h->ws;
    const size_t d = h->din, G = h->G;
    // the kernels read the codes in 16-byte vectors: a device Q that is not
    // 16-byte aligned is staged like host memory
    const bool dW = is_device_ptr(W), dS = is_device_ptr(S),
               dQ = is_device_ptr(Q) && ((uintptr_t)Q & 15) == 0, dZ = is_device_ptr(Z);
    if ((!dW || !dS || !dQ || !dZ) && w.stage_rows < p) {
        cudaFree(w.sW);
        cudaFree(w.sS);
        cudaFree(w.sQ);
        cudaFree(w.sZ);
        w.sW = nullptr;
        w.sS = nullptr;
        w.sQ = nullptr;
        w.sZ = nullptr;
        w.stage_rows = 0;
        cudaError_t e;
        if ((e = dalloc(&w.sW, (size_t)p * d)) != cudaSuccess) return e;
        if ((e = dalloc(&w.sS, (size_t)p * G)) != cudaSuccess) return e;
        if ((e = dalloc(&w.sQ, (size_t)p * d)) != cudaSuccess) return e;
        if ((e = dalloc(&w.sZ, (size_t)p * G)) != cudaSuccess) return e;
        w.stage_rows = p;
    }
    out.W = W;
    out.S = const_cast<float *>(S);
    out.Q = const_cast<uint8_t *>(Q);
    out.Z = Z;
    cudaError_t e = cudaSuccess;
    if (!dW) {
        e = cudaMemcpyAsync(w.sW, W, (size_t)p * d * sizeof(float), cudaMemcpyHostToDevice, st);
        out.W = w.sW;
    }
    if (e == cudaSuccess && !dS) {
        e = cudaMemcpyAsync(w.sS, S, (size_t)p * G * sizeof(float), cudaMemcpyHostToDevice, st);
        out.S = w.sS;
        out.hS = true;
    }
    if (e == cudaSuccess && !dQ) {
        e = cudaMemcpyAsync(w.sQ, Q, (size_t)p * d, cudaMemcpyDefault, st);
        out.Q = w.sQ;
        out.hQ = true;
    }
    if (e == cudaSuccess && !dZ) {
        e = cudaMemcpyAsync(w.sZ, Z, (size_t)p * G * sizeof(int32_t), cudaMemcpyHostToDevice,
                            st);
        out.Z = w.sZ;
    }
    return e;
}

// The arrays of a prepared Hessian (one allocation, h->mem).
void layout_hessian(Arena &m, jarq_hessian *h) {
    const size_t d = h->din, G = h->G, g = h->g, pd = (size_t)h->d_pad * h->d_pad;
    m.take(h->Hs, d * d);
    m.take(h->Hplanes, 3 * pd);
    m.take(h->Hdig8, 6 * pd);
    m.take(h->Hdig10, 4 * pd);
    m.take(h->expo, G * G);
    m.take(h->Lf, G * factor_floats((int)g));
    m.take(h->L64, G * g * g);
    m.take(h->Rinv, G * g * g);
    m.take(h->rdig, 6 * d * g);
    m.take(h->rexp, G);
    m.take(h->Htdig, 4 * pd);
    m.take(h->expoT, G * G);
    m.take(h->band, G * (sweep_block(h->g) - 1) * g * g);
    m.take(h->dstatus, 1);
}

jarq_status status_from_bits(int bits) {
    if (bits & ST_NOT_SPD) return JARQ_ERR_NOT_SPD;
    if (bits & (ST_BAD_CODE | ST_BAD_ZERO)) return JARQ_ERR_ARG;
    if (bits & ST_TIMEOUT) return JARQ_ERR_TIMEOUT;
    if (bits & ST_NUMERICAL) return JARQ_ERR_NUMERICAL;
    return JARQ_OK;
}

cudaError_t read_status(jarq_hessian *h, cudaStream_t st, int *bits) {
    cudaError_t e = cudaMemcpyAsync(h->hstatus, h->dstatus, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    *bits = (e == cudaSuccess) ? *h->hstatus : 0;
    if (e == cudaSuccess) prof_collect();
    return e;
}

ResidualView rview(jarq_hessian *h) {
    return ResidualView{h->ws.r, h->ws.rplanes, h->ws.cplane, h->din, h->d_pad, h->ws.p_pad};
}

// Common front half of refine/objective: stage, validate, residual.
jarq_status layer_front(jarq_hessian *h, const float *W, const float *S, const uint8_t *Q,
                        const int32_t *Z, int dout, int bits, LayerArgs &la, cudaStream_t st,
                        bool codes_only = false) {
    CK(cudaSetDevice(h->device));
    CK(ensure_ws(h, dout, st));
    CK(stage_layer(h, W, S, Q, Z, dout, la, st));
    CK(cudaMemsetAsync(h->dstatus, 0, sizeof(int), st));
    RUN("validate", 1, launch_validate(la.Q, la.Z, dout, h->din, h->G, (1 << bits) - 1, h->dstatus, st));
    int sb = 0;
    CK(read_status(h, st, &sb));
    if (sb) return status_from_bits(sb);
    ResidualView rv = rview(h);
    if (codes_only) rv.r = nullptr;
    RUN("residual", 1, launch_residual(la.W, la.S, la.Q, la.Z, rv, dout, h->g, st));
    return JARQ_OK;
}

bool layer_args_ok(const jarq_hessian *h, const void *W, const void *S, const void *Q,
                   const void *Z, int dout, int bits) {
    if (!h || dout < 0 || bits < 1 || bits > 8) return false;
    if (dout > 0 && (!W || !S || !Q || !Z)) return false;
    return true;
}

// Inputs of the propagation-corrected target (App. "Propagation-Corrected
// Targets and QEP"): K = X~^T X and XX = X^T X, float32 [d][d] with the
// normalisation of the prepared H, and mu, nu^2.
struct MuTarget {
    const float *K, *XX;
    float mu, nu2;
};

jarq_status refine_impl(jarq_hessian *h, const float *W, float *S, uint8_t *Q, const int32_t *Z,
                        int dout, int bits, const jarq_options *opt, jarq_stats *stats,
                        void *stream, const MuTarget *mt);

// Digits of a d x d float32 matrix M (host or device) into the handle's
// mu-target planes, then its target projection W M^T into (out_hi, out_lo).
jarq_status project_by(jarq_hessian *h, const float *M, int p, float *out_hi, float *out_lo,
                       cudaStream_t st) {
    Workspace &w = h->ws;
    const int d = h->din, g = h->g;
    if (!h->qdig) {
        // the handle takes the planes only when all that goes with them is
        // there: a call after a failed one starts again from here
        Arena m;
        __nv_bfloat16 *dig;
        int *expo;
        const size_t pd = (size_t)h->d_pad * h->d_pad;
        auto layout = [&] {
            m.take(dig, 6 * pd);
            m.take(expo, (size_t)h->G * h->G);
        };
        layout();
        CK(dalloc(&m.base, m.used));
        m.used = 0;
        layout();
        // on the call's stream: one that does not block is not ordered with
        // the default stream, whose fill could land on digits already written
        cudaError_t e = h->d_pad != d ? cudaMemsetAsync(dig, 0, 6 * pd * 2, st) : cudaSuccess;
        if (e == cudaSuccess) e = make_tmap_bf16(&h->mapQ, dig, (uint64_t)6 * h->d_pad, h->d_pad, 64, 32);
        if (e != cudaSuccess) cudaFree(m.base);
        CK(e);
        h->qdig = dig;
        h->qexp = expo;
    }
    // the digit kernels read M in 16-byte vectors: a device M that is not
    // 16-byte aligned is staged like host memory
    const float *Md = M;
    if (!is_device_ptr(M) || ((uintptr_t)M & 15)) {
        if (!h->qstage) CK(dalloc(&h->qstage, (size_t)d * d));
        CK(cudaMemcpyAsync(h->qstage, M, (size_t)d * d * sizeof(float), cudaMemcpyDefault, st));
        Md = h->qstage;
    }
    RUN("slices", 2, launch_slices8(Md, h->qexp, h->qdig, d, h->d_pad, g, st));
    RUN("proj", 1, launch_tc_proj(w.mapWd, h->mapQ, out_hi, out_lo, w.wexp, h->qexp, p, w.p_pad,
                                  d, h->d_pad, g, h->dstatus, st));
    return JARQ_OK;
}

// H w_corr and ||y(mu)||^2 in place of H w and w^T H w (Eqs. mu-target,
// w-corr): w^T XX w from the projection by XX, then the projection by K
// and the combination.
jarq_status mu_projection(jarq_hessian *h, const float *Wd, int p, const MuTarget &t,
                          cudaStream_t st) {
    Workspace &w = h->ws;
    const int d = h->din;
    jarq_status rc = project_by(h, t.XX, p, w.Pt_hi, w.Pt_lo, st);
    if (rc != JARQ_OK) return rc;
    RUN("whw", 1, launch_whw(Wd, w.Pt_hi, w.Pt_lo, w.aux, p, d, st));
    rc = project_by(h, t.K, p, w.Pt_hi, w.Pt_lo, st);
    if (rc != JARQ_OK) return rc;
    RUN("mu_combine", 1, launch_mu_combine(w.Phi, w.Plo, w.Pt_hi, w.Pt_lo, Wd, w.aux, w.wHw, p, d,
                                           (double)t.mu, (double)t.nu2, st));
    return JARQ_OK;
}

}  // namespace

extern "C" {

jarq_options jarq_default_options(void) {
    jarq_options o;
    o.max_iters = 3;
    o.early_stop = 1;
    o.tau_rel = 1e-5f;
    o.tau_abs = 1e-5f;
    o.ridge = 1e-4f;
    o.rcond = 1e-10f;
    o.eps = FLT_EPSILON;
    o.ridge_accept = 0;
    o.fixed_grid = 0;
    return o;
}

jarq_status jarq_selftest_wait_timeout(void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    int *d = nullptr;
    int bits = 0;
    if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) {
        (void)cudaGetLastError();
        return JARQ_ERR_NOMEM;
    }
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(int), st);
    if (e == cudaSuccess) e = launch_wait_timeout(d, 256, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, d, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return JARQ_ERR_CUDA;
    }
    return status_from_bits(bits);
}

const char *jarq_status_string(jarq_status s) {
    switch (s) {
        case JARQ_OK: return "ok";
        case JARQ_ERR_ARG: return "invalid argument";
        case JARQ_ERR_NOT_SPD: return "Hessian diagonal block not positive definite";
        case JARQ_ERR_NUMERICAL: return "scale system failed even with the ridge";
        case JARQ_ERR_CUDA: return "CUDA error";
        case JARQ_ERR_TIMEOUT: return "device wait timed out";
        case JARQ_ERR_NOMEM: return "device allocation failed";
    }
    return "unknown status";
}

int jarq_hessian_din(const jarq_hessian *h) { return h ? h->din : 0; }
int jarq_hessian_group_size(const jarq_hessian *h) { return h ? h->g : 0; }

void jarq_hessian_destroy(jarq_hessian *h) {
    if (!h) return;
    DeviceGuard dg(h->device);
    cudaDeviceSynchronize();
    free_ws(h->ws);
    cudaFree(h->mem);
    cudaFree(h->qdig);
    cudaFree(h->qstage);
    cudaFreeHost(h->hstatus);
    (void)cudaGetLastError();
    delete h;
}

jarq_status jarq_prepare_hessian(const float *H, int din, int group_size, float nu2,
                                 jarq_hessian **out, void *stream) {
    if (!H || !out || din <= 0 || (group_size != 64 && group_size != 128) ||
        din % group_size != 0 || din / group_size > kMaxGroups || !isfinite(nu2))
        return JARQ_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    jarq_hessian *h = new (std::nothrow) jarq_hessian();
    if (!h) return JARQ_ERR_NOMEM;
    h->din = din;
    h->g = group_size;
    h->G = din / group_size;
    h->d_pad = round_up(din, 128);
    jarq_status rc = JARQ_OK;
    float *Hdev = nullptr;
    do {
        if (cudaGetDevice(&h->device) != cudaSuccess) { rc = JARQ_ERR_CUDA; break; }
        const size_t dd = (size_t)din * din;
        cudaError_t e;
        const size_t pd = (size_t)h->d_pad * h->d_pad;
        Arena m;
        layout_hessian(m, h);
        if ((e = dalloc(&h->mem, m.used)) != cudaSuccess) { rc = cuda_fail(e); break; }
        m = Arena{h->mem};
        layout_hessian(m, h);
        // the folded rows R_i^{-T} H[grp i, :] as float pairs, only needed to
        // form their digits, and the inverse factors as float pairs, only
        // needed to form those: 8 d^2 + 8 d g bytes in the 20 d_pad^2 of H's own
        // digits (Hdig8 and behind it Hdig10), which are formed last
        float *const Ht_hi = reinterpret_cast<float *>(h->Hdig8), *const Ht_lo = Ht_hi + dd;
        float2 *const RinvF = reinterpret_cast<float2 *>(Ht_lo + dd);
        // columns beyond din are read as zeros by the products
        const bool padded = h->d_pad != din;
        if (padded) {
            if ((e = cudaMemsetAsync(h->Hplanes, 0, 3 * pd * 2, st)) != cudaSuccess) { rc = cuda_fail(e); break; }
            if ((e = cudaMemsetAsync(h->Htdig, 0, 4 * pd * 2, st)) != cudaSuccess) { rc = cuda_fail(e); break; }
        }
        if ((e = make_tmap_bf16(&h->mapH128, h->Hplanes, (uint64_t)3 * h->d_pad, h->d_pad, 128)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if ((e = make_tmap_bf16(&h->mapD8, h->Hdig8, (uint64_t)6 * h->d_pad, h->d_pad, 64, 32)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if ((e = make_tmap_f16(&h->mapD10, h->Hdig10, (uint64_t)4 * h->d_pad, h->d_pad, 64)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if ((e = make_tmap_bf16(&h->mapRi, h->rdig, (uint64_t)6 * din, group_size, 64, 32)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if ((e = make_tmap_f16(&h->mapHt, h->Htdig, (uint64_t)4 * h->d_pad, h->d_pad, 64)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if ((e = cudaMallocHost((void **)&h->hstatus, sizeof(int))) != cudaSuccess) { rc = cuda_fail(e); break; }
        const float *Hsrc = H;
        if (!is_device_ptr(H)) {
            if ((e = dalloc(&Hdev, dd)) != cudaSuccess) { rc = cuda_fail(e); break; }
            if ((e = cudaMemcpyAsync(Hdev, H, dd * sizeof(float), cudaMemcpyHostToDevice, st)) != cudaSuccess) { rc = cuda_fail(e); break; }
            Hsrc = Hdev;
        }
        if ((e = cudaMemsetAsync(h->dstatus, 0, sizeof(int), st)) != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("symmetrize", st); e = launch_symmetrize(Hsrc, h->Hs, h->Hplanes, din, h->d_pad, nu2, st); ps.done(); count_launches(1); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("group_factor", st); e = launch_group_factor(h->Hs, h->Lf, h->L64, h->Rinv, RinvF, din, group_size, h->dstatus, st); ps.done(); count_launches(2); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("slices", st); e = launch_slice_rinv(h->Rinv, h->rdig, h->rexp, din, group_size, st); ps.done(); count_launches(1); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("htilde", st); e = launch_htilde(h->Hs, RinvF, Ht_hi, Ht_lo, din, group_size, st); ps.done(); count_launches(1); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("slices", st); e = launch_slice10(Ht_hi, Ht_lo, h->expoT, h->Htdig, din, h->d_pad, group_size, st); ps.done(); count_launches(2); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("slices", st); e = launch_band(h->Htdig, h->band, din, h->d_pad, group_size, st); ps.done(); count_launches(1); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        if (padded && (e = cudaMemsetAsync(h->Hdig8, 0, 6 * pd * 2, st)) != cudaSuccess) { rc = cuda_fail(e); break; }
        if (padded && (e = cudaMemsetAsync(h->Hdig10, 0, 4 * pd * 2, st)) != cudaSuccess) { rc = cuda_fail(e); break; }
        { ProfScope ps("slices", st); e = launch_slices(h->Hs, h->expo, h->Hdig8, h->Hdig10, din, h->d_pad, group_size, st); ps.done(); count_launches(2); }
        if (e != cudaSuccess) { rc = cuda_fail(e); break; }
        int sb = 0;
        if ((e = read_status(h, st, &sb)) != cudaSuccess) { rc = cuda_fail(e); break; }
        rc = status_from_bits(sb);
    } while (0);
    if (Hdev) {
        cudaStreamSynchronize(st);
        cudaFree(Hdev);
    }
    if (rc != JARQ_OK) {
        jarq_hessian_destroy(h);
        return rc;
    }
    *out = h;
    return JARQ_OK;
}

jarq_status jarq_objective(jarq_hessian *h, const float *W, const float *S, const uint8_t *Q,
                           const int32_t *Z, int dout, int bits, double *F_per_row,
                           void *stream) {
    if (!layer_args_ok(h, W, S, Q, Z, dout, bits) || (dout > 0 && !F_per_row))
        return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    DeviceGuard dg(h->device);
    if (!dg.ok()) return JARQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    LayerArgs la;
    jarq_status rc = layer_front(h, W, S, Q, Z, dout, bits, la, st);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    CK(cudaMemsetAsync(h->dstatus, 0, sizeof(int), st));
    RUN("hr_full", 1, launch_tc_hr_full(w.mapR, h->mapH128, w.Hr, dout, w.p_pad, h->din, h->d_pad, h->dstatus, st));
    RUN("grad", 1, launch_grad(w.r, w.Hr, w.L_final, dout, h->din, st));
    CK(cudaMemcpyAsync(F_per_row, w.L_final, (size_t)dout * sizeof(double), cudaMemcpyDefault, st));
    int sb = 0;
    CK(read_status(h, st, &sb));
    return status_from_bits(sb);
}

jarq_status jarq_residual_product(jarq_hessian *h, const float *W, const float *S,
                                  const uint8_t *Q, const int32_t *Z, int dout, int bits,
                                  float *HR, void *stream) {
    if (!layer_args_ok(h, W, S, Q, Z, dout, bits) || (dout > 0 && !HR)) return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    DeviceGuard dg(h->device);
    if (!dg.ok()) return JARQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    LayerArgs la;
    jarq_status rc = layer_front(h, W, S, Q, Z, dout, bits, la, st);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    CK(cudaMemsetAsync(h->dstatus, 0, sizeof(int), st));
    RUN("hr_full", 1, launch_tc_hr_full(w.mapR, h->mapH128, w.Hr, dout, w.p_pad, h->din, h->d_pad, h->dstatus, st));
    CK(cudaMemcpyAsync(HR, w.Hr, (size_t)dout * h->din * sizeof(float), cudaMemcpyDefault, st));
    int sb = 0;
    CK(read_status(h, st, &sb));
    return status_from_bits(sb);
}

jarq_status jarq_refine_layer(jarq_hessian *h, const float *W, float *S, uint8_t *Q,
                              const int32_t *Z, int dout, int bits, const jarq_options *opt,
                              jarq_stats *stats, void *stream) {
    return refine_impl(h, W, S, Q, Z, dout, bits, opt, stats, stream, nullptr);
}

jarq_status jarq_fit_scales(jarq_hessian *h, const float *W, float *S, const uint8_t *Q,
                            const int32_t *Z, int dout, int bits, jarq_fit method, int passes,
                            double *F_before, double *F_after, void *stream) {
    if (!layer_args_ok(h, W, S, Q, Z, dout, bits)) return JARQ_ERR_ARG;
    if (method != JARQ_FIT_JOINT && method != JARQ_FIT_INDEPENDENT &&
        method != JARQ_FIT_COORDINATE)
        return JARQ_ERR_ARG;
    if (method == JARQ_FIT_COORDINATE && passes < 1) return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    DeviceGuard dg(h->device);
    if (!dg.ok()) return JARQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    LayerArgs la;
    jarq_status rc = layer_front(h, W, S, Q, Z, dout, bits, la, st, true);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    const int p = dout, d = h->din, g = h->g, G = h->G;
    RUN("init_rows", 1, launch_init_rows(w.active, w.iters, w.accepted, w.ridge, w.rstat, p, st));
    RUN("slice_rows", 1, launch_slice_rows(la.W, w.wdig, w.wexp, p, d, h->d_pad, w.p_pad, g, st));
    RUN("proj", 1, launch_tc_proj(w.mapWd, h->mapD8, w.Phi, w.Plo, w.wexp, h->expo, p, w.p_pad, d,
                                  h->d_pad, g, h->dstatus, st));
    RUN("whw", 1, launch_whw(la.W, w.Phi, w.Plo, w.wHw, p, d, st));
    RUN("gram", 1, launch_tc_gram(w.mapC, h->mapD10, la.Q, la.Z, h->expo, nullptr, w.gram, p,
                                  w.p_pad, d, h->d_pad, g, bits, h->dstatus, st));
    RUN("rhs", 1, launch_rhs(la.Q, la.Z, w.Phi, w.Plo, nullptr, w.rhs, p, d, g, st));
    if (method == JARQ_FIT_JOINT) {
        jarq_options o = jarq_default_options();
        o.early_stop = 0;
        RUN("scale_solve", 1, launch_scale_solve(w.gram, w.rhs, w.wHw, la.S, w.L_prev, w.L_host,
                                                 w.active, w.iters, w.ridge, w.rstat, h->dstatus,
                                                 p, d, g, 1, false, o, st));
        CK(cudaMemcpyAsync(w.L_final, w.L_prev, p * sizeof(double), cudaMemcpyDeviceToDevice, st));
    } else {
        if (method == JARQ_FIT_INDEPENDENT)
            RUN("own_rhs", 1, launch_own_rhs(h->Hs, la.W, la.Q, la.Z, w.own, p, d, g, st));
        RUN("scale_fit", 1, launch_scale_fit(w.gram, w.rhs, w.own, w.wHw, la.S, w.L_host,
                                             w.L_final, p, G, (int)method, passes, st));
    }
    if (la.hS) CK(cudaMemcpyAsync(S, la.S, (size_t)p * G * sizeof(float), cudaMemcpyDeviceToHost, st));
    if (F_before) CK(cudaMemcpyAsync(F_before, w.L_host, p * sizeof(double), cudaMemcpyDefault, st));
    if (F_after) CK(cudaMemcpyAsync(F_after, w.L_final, p * sizeof(double), cudaMemcpyDefault, st));
    int sb = 0;
    CK(read_status(h, st, &sb));
    return status_from_bits(sb);
}

jarq_status jarq_multicode_probe(jarq_hessian *h, const float *W, const float *S,
                                 const uint8_t *Q, const int32_t *Z, int dout, int bits,
                                 int group, uint8_t *Q_search, int32_t *moves, int32_t *accepted,
                                 int32_t *changed, double *dF, void *stream) {
    if (!layer_args_ok(h, W, S, Q, Z, dout, bits) || group < 0 || group >= h->G) return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    DeviceGuard dg(h->device);
    if (!dg.ok()) return JARQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    LayerArgs la;
    jarq_status rc = layer_front(h, W, S, Q, Z, dout, bits, la, st, true);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    const int p = dout, d = h->din, g = h->g, G = h->G;
    const int nsplit = target_splits(w.p_pad, g, G, 1);
    RUN("slice_rows", 1, launch_slice_rows(la.W, w.wdig, w.wexp, p, d, h->d_pad, w.p_pad, g, st));
    RUN("proj", 1, launch_tc_proj(w.mapWd, h->mapD8, w.Phi, w.Plo, w.wexp, h->expo, p, w.p_pad, d,
                                  h->d_pad, g, h->dstatus, st));
    // T = sum_h s_h H_ih c_h: the sweep's product with H's own digits
    RUN("sweep_product", 1, launch_tc_target(w.mapC, h->mapD10, w.t_hi, w.t_lo, la.S, h->expo, nullptr, p,
                                      w.p_pad, h->d_pad, g, G, group, 1, 0, nsplit, (1 << bits) - 1, h->dstatus, st,
                                      false));
    uint8_t *qo = reinterpret_cast<uint8_t *>(w.Hr);
    RUN("probe", 1, launch_probe(w.Phi, w.Plo, w.t_hi, w.t_lo, h->Hs, h->L64, la.S, la.Q, la.Z, qo,
                                 w.iters, w.accepted, w.ridge, w.L_final, p, w.p_pad, d, g, group,
                                 nsplit, (1 << bits) - 1, FLT_EPSILON, st));
    if (Q_search) CK(cudaMemcpyAsync(Q_search, qo, (size_t)p * g, cudaMemcpyDefault, st));
    if (moves) CK(cudaMemcpyAsync(moves, w.iters, p * sizeof(int32_t), cudaMemcpyDefault, st));
    if (accepted) CK(cudaMemcpyAsync(accepted, w.accepted, p * sizeof(int32_t), cudaMemcpyDefault, st));
    if (changed) CK(cudaMemcpyAsync(changed, w.ridge, p * sizeof(int32_t), cudaMemcpyDefault, st));
    if (dF) CK(cudaMemcpyAsync(dF, w.L_final, p * sizeof(double), cudaMemcpyDefault, st));
    int sb = 0;
    CK(read_status(h, st, &sb));
    return status_from_bits(sb);
}

jarq_status jarq_selftest_stalled_kernel(const char *kernel, void *stream) try {
    if (!kernel) return JARQ_ERR_ARG;
    auto is = [&](const char *name) { return !strcmp(kernel, name); };
    // a small layer refined and scored first, so that every buffer holds what
    // its kernel reads
    constexpr int d = 512, g = 128, G = d / g, p = 300, bits = 3, n = 1200;
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<float> H((size_t)d * d), W((size_t)p * d), S((size_t)p * G, 0.1f);
    std::vector<uint8_t> Q((size_t)p * d);
    std::vector<int32_t> Z((size_t)p * G, 3);
    std::vector<double> F(p);
    for (int i = 0; i < d; ++i) H[(size_t)i * d + i] = 1.f;
    for (size_t i = 0; i < W.size(); ++i) {
        Q[i] = (uint8_t)(i * 5 % 8);
        W[i] = 0.1f * (float)((int)Q[i] - 3) + 0.01f * (float)(i % 7);
    }
    jarq_hessian *h = nullptr;
    jarq_status rc = jarq_prepare_hessian(H.data(), d, g, 0.f, &h, stream);
    if (rc != JARQ_OK) return rc;
    std::unique_ptr<jarq_hessian, void (*)(jarq_hessian *)> owner(h, jarq_hessian_destroy);
    rc = jarq_refine_layer(h, W.data(), S.data(), Q.data(), Z.data(), p, bits, nullptr, nullptr, stream);
    if (rc == JARQ_OK)
        rc = jarq_objective(h, W.data(), S.data(), Q.data(), Z.data(), p, bits, F.data(), stream);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    CK(cudaMemsetAsync(h->dstatus, 0, sizeof(int), st));
    char *scratch = nullptr;
    if (is("target")) {
        CK(launch_tc_target(w.mapC, h->mapHt, w.t_hi, w.t_lo, w.sS, h->expoT, nullptr, p, w.p_pad, h->d_pad, g, G,
                            0, sweep_block(g), 0, 1, (1 << bits) - 1, h->dstatus, st, false, true));
    } else if (is("gram")) {
        CK(launch_tc_gram(w.mapC, h->mapD10, w.sQ, w.sZ, h->expo, nullptr, w.gram, p, w.p_pad, d, h->d_pad, g,
                          bits, h->dstatus, st, false, true));
    } else if (is("proj")) {
        CK(launch_tc_proj(w.mapWd, h->mapD8, w.Phi, w.Plo, w.wexp, h->expo, p, w.p_pad, d, h->d_pad, g, h->dstatus,
                          st, true));
    } else if (is("ptilde")) {
        CK(launch_ptilde(w.mapPd, h->mapRi, w.Phi, w.Plo, w.wdig, w.wexp, h->rexp, w.Pt_hi, w.Pt_lo, p, w.p_pad, d,
                         h->d_pad, g, h->dstatus, st, true));
    } else if (is("hr_full")) {
        CK(launch_tc_hr_full(w.mapR, h->mapH128, w.Hr, p, w.p_pad, d, h->d_pad, h->dstatus, st, true));
    } else if (is("syrk")) {
        const size_t hb = (size_t)d * d * sizeof(float), xb = (size_t)n * d * 2;
        CUtensorMap map;
        CK(dalloc(&scratch, hb + xb));
        cudaError_t e = cudaMemsetAsync(scratch, 0, hb + xb, st);
        if (e == cudaSuccess) e = make_tmap_f16(&map, scratch + hb, n, d, 64);
        if (e == cudaSuccess)
            e = launch_tc_syrk(map, reinterpret_cast<float *>(scratch), h->dstatus, 1.f, d, n, st, true);
        if (e != cudaSuccess) cudaFree(scratch);
        CK(e);
    } else {
        return JARQ_ERR_ARG;
    }
    int sb = 0;
    const cudaError_t e = read_status(h, st, &sb);
    cudaFree(scratch);
    CK(e);
    return status_from_bits(sb);
} catch (const std::bad_alloc &) {
    return JARQ_ERR_NOMEM;
}

jarq_status jarq_refine_layer_mu(jarq_hessian *h, const float *W, float *S, uint8_t *Q,
                                 const int32_t *Z, int dout, int bits, const float *K,
                                 const float *XX, float mu, float nu2, const jarq_options *opt,
                                 jarq_stats *stats, void *stream) {
    if (!(mu >= 0.f && mu <= 1.f) || !(nu2 >= 0.f) || !isfinite(nu2)) return JARQ_ERR_ARG;
    if (mu == 1.f) return refine_impl(h, W, S, Q, Z, dout, bits, opt, stats, stream, nullptr);
    if (!K || !XX) return JARQ_ERR_ARG;
    MuTarget t{K, XX, mu, nu2};
    return refine_impl(h, W, S, Q, Z, dout, bits, opt, stats, stream, &t);
}

}  // extern "C"

namespace {

jarq_status refine_impl(jarq_hessian *h, const float *W, float *S, uint8_t *Q, const int32_t *Z,
                        int dout, int bits, const jarq_options *opt, jarq_stats *stats,
                        void *stream, const MuTarget *mt) {
    if (!layer_args_ok(h, W, S, Q, Z, dout, bits)) return JARQ_ERR_ARG;
    jarq_options o = opt ? *opt : jarq_default_options();
    if (o.max_iters < 0 || !(o.ridge >= 0.f) || !(o.rcond >= 0.f) || !(o.eps >= 0.f))
        return JARQ_ERR_ARG;
    if (dout == 0) return JARQ_OK;
    DeviceGuard dg(h->device);
    if (!dg.ok()) return JARQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    LayerArgs la;
    jarq_status rc = layer_front(h, W, S, Q, Z, dout, bits, la, st, true);
    if (rc != JARQ_OK) return rc;
    Workspace &w = h->ws;
    const int p = dout, d = h->din, g = h->g, G = h->G, qmax = (1 << bits) - 1;
    RUN("init_rows", 1, launch_init_rows(w.active, w.iters, w.accepted, w.ridge, w.rstat, p, st));
    const ResidualView rv = rview(h);
    // the sweep's blocks of groups, and the split of their products over K
    const int nblk = G < sweep_block(g) ? G : sweep_block(g);
    const int nsplit = target_splits(w.p_pad, g, G, nblk);
    // target projection P = W H, w^T H w and the folded Pt, once per call
    RUN("slice_rows", 1, launch_slice_rows(la.W, w.wdig, w.wexp, p, d, h->d_pad, w.p_pad, g, st));
    RUN("proj", 1, launch_tc_proj(w.mapWd, h->mapD8, w.Phi, w.Plo, w.wexp, h->expo, p, w.p_pad, d,
                                  h->d_pad, g, h->dstatus, st));
    RUN("whw", 1, launch_whw(la.W, w.Phi, w.Plo, w.wHw, p, d, st));
    if (mt) {
        // mu-target: P <- H w_corr and w^T H w <- ||y(mu)||^2 from the two
        // extra projections W XX and W K^T (Pt's buffers hold them until
        // the folded projection is formed)
        rc = mu_projection(h, la.W, p, *mt, st);
        if (rc != JARQ_OK) return rc;
    }
    RUN("ptilde", 2, launch_ptilde(w.mapPd, h->mapRi, w.Phi, w.Plo, w.wdig, w.wexp, h->rexp, w.Pt_hi,
                                   w.Pt_lo, p, w.p_pad, d, h->d_pad, g, h->dstatus, st));
    // Gram, right-hand side and solve of a small layer are launched
    // programmatically too, so that launch latency and prologues run under the
    // kernel before: 256 x 256 455 -> 427 us, 1024 x 512 530 -> 500 us, 64 x 4096
    // 3.26 -> 3.21 ms.  Above 2^19 weights the early grids take room from the
    // running one: 1000 x 1344 1.05 -> 1.10 ms, 256 x 4096 2.82 -> 2.88 ms, 4096 x
    // 4096 13.02 -> 13.15 ms.
    constexpr long long kChainedWeights = 1ll << 19;
    const bool chained = (long long)p * d <= kChainedWeights;
    for (int k = 1; k <= o.max_iters; ++k) {
        // with the early stop off every row is refined (a row marked numerical
        // is skipped by the solve and Babai), so the Gram and the right-hand
        // side need not read the active flags
        const int *act_es = o.early_stop ? w.active : nullptr;
        RUN("gram", 1, launch_tc_gram(w.mapC, h->mapD10, la.Q, la.Z, h->expo, act_es, w.gram, p,
                                      w.p_pad, d, h->d_pad, g, bits, h->dstatus, st, chained));
        RUN("rhs", 1, launch_rhs(la.Q, la.Z, w.Phi, w.Plo, act_es, w.rhs, p, d, g, st, chained));
        double *L_out = (k == 1 && stats && stats->L_host) ? w.L_host : nullptr;
        RUN("scale_solve", 1, launch_scale_solve(w.gram, w.rhs, w.wHw, la.S, w.L_prev, L_out,
                                                 w.active, w.iters, w.ridge, w.rstat, h->dstatus,
                                                 p, d, g, k, false, o, st, chained));
        // The product reads the active flags only with the early stop on (to
        // skip pairs of tiles whose rows all stopped); a row marked numerical
        // by the scale solve is skipped by Babai, and its partials go unread.
        for (int i0 = 0; i0 < G; i0 += nblk) {
            const int nb = G - i0 < nblk ? G - i0 : nblk;
            RUN("sweep_product", 1,
                launch_tc_target(w.mapC, h->mapHt, w.t_hi, w.t_lo, la.S, h->expoT,
                                 o.early_stop ? w.active : nullptr, p, w.p_pad, h->d_pad, g, G, i0,
                                 nb, i0 ? nblk : 0, nsplit, qmax, h->dstatus, st, true));
            RUN("sweep_babai", 1,
                launch_babai(w.t_hi, w.t_lo, w.Pt_hi, w.Pt_lo, nsplit, h->Lf, h->band, h->expoT,
                             la.S, la.Q, la.Z, rv, w.active, w.accepted, h->dstatus, p, g, i0, nb,
                             qmax, o.eps, st));
        }
    }
    // objective of the returned state (and of the input state when K = 0)
    const bool want_final = stats && stats->L_final;
    const bool want_host0 = stats && stats->L_host && o.max_iters == 0;
    if (want_final || want_host0) {
        RUN("gram", 1, launch_tc_gram(w.mapC, h->mapD10, la.Q, la.Z, h->expo, nullptr, w.gram, p,
                                      w.p_pad, d, h->d_pad, g, bits, h->dstatus, st, chained));
        RUN("rhs", 1, launch_rhs(la.Q, la.Z, w.Phi, w.Plo, nullptr, w.rhs, p, d, g, st, chained));
        RUN("scale_solve", 1, launch_scale_solve(w.gram, w.rhs, w.wHw, la.S, w.L_prev, w.L_final,
                                                 w.active, w.iters, w.ridge, w.rstat, h->dstatus,
                                                 p, d, g, 0, true, o, st, chained));
        if (want_host0)
            CK(cudaMemcpyAsync(w.L_host, w.L_final, p * sizeof(double), cudaMemcpyDeviceToDevice, st));
    }
    if (la.hS) CK(cudaMemcpyAsync(S, la.S, (size_t)p * G * sizeof(float), cudaMemcpyDeviceToHost, st));
    if (la.hQ) CK(cudaMemcpyAsync(Q, la.Q, (size_t)p * d, cudaMemcpyDefault, st));
    if (stats) {
        if (stats->L_host) CK(cudaMemcpyAsync(stats->L_host, w.L_host, p * sizeof(double), cudaMemcpyDefault, st));
        if (stats->L_final) CK(cudaMemcpyAsync(stats->L_final, w.L_final, p * sizeof(double), cudaMemcpyDefault, st));
        if (stats->iters) CK(cudaMemcpyAsync(stats->iters, w.iters, p * sizeof(int), cudaMemcpyDefault, st));
        if (stats->accepted) CK(cudaMemcpyAsync(stats->accepted, w.accepted, p * sizeof(int), cudaMemcpyDefault, st));
        if (stats->ridge_hits) CK(cudaMemcpyAsync(stats->ridge_hits, w.ridge, p * sizeof(int), cudaMemcpyDefault, st));
        if (stats->row_status) CK(cudaMemcpyAsync(stats->row_status, w.rstat, p * sizeof(int), cudaMemcpyDefault, st));
    }
    int sb = 0;
    CK(read_status(h, st, &sb));
    return status_from_bits(sb);
}

}  // namespace
