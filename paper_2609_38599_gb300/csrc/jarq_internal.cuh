// Internal declarations shared by the JARQ CUDA sources (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <atomic>

#include "../../include/jarq.h"

namespace jarq {

// Device status bits (OR-ed by kernels, read back once per call).
enum : int {
    ST_NOT_SPD = 1,      // a diagonal block of H is not positive definite
    ST_NUMERICAL = 2,    // a row's scale system failed even with the ridge
    ST_BAD_CODE = 4,     // a code is outside [0, 2^b - 1]
    ST_BAD_ZERO = 8,     // a zero point is outside [0, 2^b - 1]
    ST_TIMEOUT = 16,     // a bounded device wait gave up
};

constexpr int kMaxGroups = 128;    // largest supported G for the scale solve
constexpr int kMaxGroupSize = 128; // the larger of the two group sizes
constexpr int kMaxSplit = 16;      // largest split-K factor of the sweep's product

// Groups of one block of the sweep for group size g: 256 columns.  The Babai
// kernel holds the factors of two groups and the blocks Ht_i'i of one group i
// in shared memory, which for g = 128 leaves room for one such block.  Two
// groups of 128 in one launch take 32.8 us of product and 27.6 us of Babai
// steps on 4096 x 4096; with a launch per group the start of each launch
// (about 8 us of a product, 4 us of a Babai step) is paid twice.
__host__ __device__ constexpr int sweep_block(int g) { return 256 / g; }

__host__ __device__ inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Layout of one group's factor L_i = R_i^T as the Babai kernel reads it
// (k_babai.cu), float32:
//   rows   h = 0 .. g - 1: columns 0 .. 32 (h/32 + 1) - 1 of L[h], zero from
//          column 4 (h/4) on (h's own quad and everything above the diagonal)
//   tri    per quad 4 q .. 4 q + 3 eight floats: L[3][2], L[3][1], L[3][0],
//          L[2][1], L[2][0], L[1][0] of the quad's own block, 0, 0
//   diag   L[l][l];  rdiag  1 / L[l][l]
__host__ __device__ constexpr int factor_row(int h) {
    return 512 * (h / 32) * (h / 32 + 1) + (h % 32) * 32 * (h / 32 + 1);
}
__host__ __device__ constexpr int factor_tri(int g) { return 512 * (g / 32) * (g / 32 + 1); }
__host__ __device__ constexpr int factor_diag(int g) { return factor_tri(g) + 2 * g; }
__host__ __device__ constexpr int factor_rdiag(int g) { return factor_tri(g) + 3 * g; }
__host__ __device__ constexpr int factor_floats(int g) { return factor_tri(g) + 4 * g; }

// View of the residual r = w - D_s (q - z): float32 [p][d] plus its exact
// three-plane bf16 split [3][p_pad][d_pad] read by the tensor cores, and the
// integer codes c = q - z as fp16 [p_pad][d_pad] (exact for |c| <= 2048).
struct ResidualView {
    float *r;
    __nv_bfloat16 *planes;
    __half *cplane;
    int d, d_pad, p_pad;
};

// Exact split x = x1 + x2 + x3 of a float32 into bf16 values (truncation).
__device__ __forceinline__ void split3(float x, __nv_bfloat16 &a, __nv_bfloat16 &b,
                                       __nv_bfloat16 &c) {
    const float x1 = __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
    const float rem = x - x1;
    const float x2 = __uint_as_float(__float_as_uint(rem) & 0xFFFF0000u);
    a = __float2bfloat16_rz(x1);
    b = __float2bfloat16_rz(x2);
    c = __float2bfloat16_rn(rem - x2);
}

__device__ __forceinline__ void store_code(const ResidualView &v, size_t j, int col, int c) {
    v.cplane[j * v.d_pad + col] = __int2half_rn(c);
}

__device__ __forceinline__ void store_residual(const ResidualView &v, size_t j, int col, float x) {
    v.r[j * v.d + col] = x;
    __nv_bfloat16 a, b, c;
    split3(x, a, b, c);
    const size_t plane = (size_t)v.p_pad * v.d_pad, off = j * v.d_pad + col;
    v.planes[off] = a;
    v.planes[plane + off] = b;
    v.planes[2 * plane + off] = c;
}

// Library-owned refinement workspace, sized for `cap_rows` output rows.
struct Workspace {
    int cap_rows = 0;
    char *mem = nullptr;         // the one allocation that holds the arrays below
    int p_pad = 0;               // rows of the bf16 residual planes (multiple of 128)
    float *Hr = nullptr;         // [p][d]  H r for every row (objective entry point)
    float *r = nullptr;          // [p][d]  residual r = w - D_s (q - z)
    float2 *gram = nullptr;      // [p][G][G]  Gram matrices of the current codes (float pairs)
    double *rhs = nullptr;       // [p][G]  rhs_i = c_i^T P_i (also the scratch of grad)
    float *t_hi = nullptr;       // [nsplit][p_pad][nb g]  split-K partials of the
    float *t_lo = nullptr;       //   product of a block's nb groups (double-float)
    __nv_bfloat16 *rplanes = nullptr;  // [3][p_pad][d_pad] bf16 split of r
    __half *cplane = nullptr;          // [p_pad][d_pad] codes c = q - z
    CUtensorMap mapR;            // tensor map of rplanes, 128 x 64 boxes
    CUtensorMap mapC;            // tensor map of cplane, 128 x 64 boxes
    // target projection P = W H (once per call); after it the same buffers
    // hold the six digit planes of P for the folded projection
    __nv_bfloat16 *wdig = nullptr;     // [6][p_pad][d_pad] integer digits of W (4) or P (6)
    int *wexp = nullptr;               // [p][G] exponents of those digits
    CUtensorMap mapWd;                 // tensor map of wdig's first 4 planes, 128 x 32 boxes
    CUtensorMap mapPd;                 // tensor map of all 6 planes, 128 x 32 boxes
    float *Phi = nullptr;        // [p][d]  P = Phi + Plo (double-float)
    float *Plo = nullptr;        // [p][d]
    float *Pt_hi = nullptr;      // [p][d]  folded projection Pt_i = R_i^{-T} P_i
    float *Pt_lo = nullptr;      // [p][d]
    double *wHw = nullptr;       // [p]  w_j^T H w_j (||y_j(mu)||^2 for the mu-target)
    double *aux = nullptr;       // [p]  w_j^T XX w_j of the mu-target
    double *own = nullptr;       // [p][G]  c_i^T H_ii w_i (independent scale fit)
    double *L_prev = nullptr;    // [p]  L^{(k-1)} of the early stop
    double *L_host = nullptr;    // [p]
    double *L_final = nullptr;   // [p]
    int *active = nullptr;       // [p]
    int *iters = nullptr;        // [p]
    int *accepted = nullptr;     // [p]
    int *ridge = nullptr;        // [p]
    int *rstat = nullptr;        // [p]
    // staging for host-memory arguments (allocated on first use)
    int stage_rows = 0;
    float *sW = nullptr;
    float *sS = nullptr;
    uint8_t *sQ = nullptr;
    int32_t *sZ = nullptr;
};

}  // namespace jarq

struct jarq_hessian {
    int din = 0, g = 0, G = 0;
    int device = 0;
    int d_pad = 0;
    char *mem = nullptr;          // the one allocation that holds the arrays below
    float *Hs = nullptr;          // [d][d] symmetrised H (+ nu2 I), fp32
    __nv_bfloat16 *Hplanes = nullptr;  // [3][d_pad][d_pad] exact bf16 split of Hs
    // per-block integer digits of Hs (block exponents in expo):
    __nv_bfloat16 *Hdig8 = nullptr;    // [6][d_pad][d_pad] base 2^8, |digit| <= 128
    __half *Hdig10 = nullptr;          // [4][d_pad][d_pad] base 2^10, |digit| <= 512
    int *expo = nullptr;          // [G][G] block exponents of the digits
    CUtensorMap mapH128;          // tensor map of Hplanes, 128 x 64 boxes
    CUtensorMap mapD8, mapD10;    // tensor maps of Hdig8 (64 x 32 boxes) / Hdig10 (64 x 64)
    float *Lf = nullptr;          // [G][factor_floats(g)] lower factor L_i = R_i^T, packed
    // digits of the blocks Ht_{i'i}, i' = i + 1 .. i + sweep_block(g) - 1, column by
    // column: [G][sweep_block(g) - 1][g columns of i][g rows of i'], each entry the
    // two 20-bit halves (a_0 2^10 + a_1, a_2 2^10 + a_3) of its digits
    int2 *band = nullptr;
    double *L64 = nullptr;        // [G][g][g] the same in float64
    double *Rinv = nullptr;       // [G][g][g] R_i^{-1} (upper), row-major, float64
    // R_i^{-1} in six base-2^8 digit planes, transposed per block (row i g + a,
    // column b: digit of R_i^{-1}[b][a]), one exponent per group
    __nv_bfloat16 *rdig = nullptr;     // [6][d][g]
    int *rexp = nullptr;               // [G]
    CUtensorMap mapRi;                 // tensor map of rdig, 64 x 32 boxes
    // folded rows Ht[grp i, :] = R_i^{-T} H[grp i, :] in the base-2^10 digit scheme
    __half *Htdig = nullptr;      // [4][d_pad][d_pad] fp16 digits, |digit| <= 512
    int *expoT = nullptr;         // [G][G] block exponents of Ht
    CUtensorMap mapHt;            // tensor map of Htdig, 64 x 64 boxes
    // mu-target (allocated on first use): digits of K or XX, base 2^8, six
    // planes, with a symmetric block-exponent map; staging for host K / XX
    __nv_bfloat16 *qdig = nullptr;     // [6][d_pad][d_pad], the allocation's start
    int *qexp = nullptr;               // [G][G], in qdig's allocation
    float *qstage = nullptr;           // [d][d]
    CUtensorMap mapQ;                  // tensor map of qdig, 64 x 32 boxes
    int *dstatus = nullptr;       // device status word
    int *hstatus = nullptr;       // pinned host mirror
    jarq::Workspace ws;
};

namespace jarq {

// ---- launchers (each returns the cudaError_t of its launch) ----
// `stalled`: the self-test's form of the kernel, whose MMA issuer stops early
// and whose waits give up after milliseconds
cudaError_t launch_symmetrize(const float *H, float *Hs, __nv_bfloat16 *Hplanes, int d, int d_pad,
                              float nu2, cudaStream_t s);
cudaError_t launch_group_factor(const float *Hs, float *Lf, double *L64, double *Rinv,
                                float2 *RinvF, int d, int g, int *status, cudaStream_t s);
cudaError_t launch_own_rhs(const float *Hs, const float *W, const uint8_t *Q, const int32_t *Z,
                           double *own, int p, int d, int g, cudaStream_t s);
cudaError_t launch_scale_fit(const float2 *gram, const double *rhs, const double *own,
                             const double *wHw, float *S, double *F_before, double *F_after, int p,
                             int G, int method, int passes, cudaStream_t s);
cudaError_t launch_probe(const float *Phi, const float *Plo, const float *t_hi, const float *t_lo,
                         const float *Hs, const double *L64, const float *S, const uint8_t *Q,
                         const int32_t *Z, uint8_t *q_out, int32_t *moves, int32_t *accepted,
                         int32_t *changed, double *dF, int p, int p_pad, int d, int g, int i,
                         int nsplit, int qmax, float eps, cudaStream_t s);
cudaError_t launch_htilde(const float *Hs, const float2 *RinvF, float *out_hi, float *out_lo,
                          int d, int g, cudaStream_t s);
cudaError_t launch_slice10(const float *hi, const float *lo, int *expo, __half *dig, int d,
                           int d_pad, int g, cudaStream_t s);

cudaError_t launch_validate(const uint8_t *Q, const int32_t *Z, int p, int d, int G, int qmax,
                            int *status, cudaStream_t s);
cudaError_t launch_residual(const float *W, const float *S, const uint8_t *Q, const int32_t *Z,
                            ResidualView rv, int p, int g, cudaStream_t s);
cudaError_t launch_tc_hr_full(const CUtensorMap &mapA, const CUtensorMap &mapB, float *out, int p,
                              int p_pad, int d, int d_pad, int *status, cudaStream_t s,
                              bool stalled = false);
cudaError_t launch_tc_syrk(const CUtensorMap &mapX, float *H, int *status, float scale, int d, int n,
                           cudaStream_t s, bool stalled = false);
cudaError_t launch_grad(const float *r, const float *Hr, double *F, int p, int d, cudaStream_t s);
cudaError_t launch_slices(const float *Hs, int *expo, __nv_bfloat16 *dig8, __half *dig10, int d,
                          int d_pad, int g, cudaStream_t s);
cudaError_t launch_tc_gram(const CUtensorMap &mapC, const CUtensorMap &mapS, const uint8_t *Q,
                           const int32_t *Z, const int *expo, const int *active, float2 *gram,
                           int p, int p_pad, int d, int d_pad, int g, int bits, int *status,
                           cudaStream_t s, bool pdl = false, bool stalled = false);
cudaError_t launch_slices8(const float *M, int *expo, __nv_bfloat16 *dig8, int d, int d_pad,
                           int g, cudaStream_t s);
cudaError_t launch_mu_combine(float *Phi, float *Plo, const float *Khi, const float *Klo,
                              const float *W, const double *wXXw, double *wHw, int p, int d,
                              double mu, double nu2, cudaStream_t s);
cudaError_t launch_slice_rows(const float *W, __nv_bfloat16 *planes, int *wexp, int p, int d,
                              int d_pad, int p_pad, int g, cudaStream_t s);
cudaError_t launch_tc_proj(const CUtensorMap &mapW, const CUtensorMap &mapH, float *Phi,
                           float *Plo, const int *wexp, const int *hexp, int p, int p_pad, int d,
                           int d_pad, int g, int *status, cudaStream_t s, bool stalled = false);
cudaError_t launch_whw(const float *W, const float *Phi, const float *Plo, double *out, int p,
                       int d, cudaStream_t s);
cudaError_t launch_rhs(const uint8_t *Q, const int32_t *Z, const float *Phi, const float *Plo,
                       const int *active, double *rhs, int p, int d, int g, cudaStream_t s,
                       bool pdl = false);
cudaError_t launch_scale_solve(const float2 *gram, const double *rhs, const double *wHw, float *S,
                               double *L_prev, double *L_out, int *active,
                               int *iters, int *ridge, int *rstat, int *status, int p, int d,
                               int g, int k, bool eval_only, const jarq_options &o,
                               cudaStream_t s, bool pdl = false);
cudaError_t launch_babai(float *t_hi, float *t_lo, const float *pt_hi,
                         const float *pt_lo, int nsplit, const float *Lf, const int2 *band,
                         const int *expoT, const float *S, uint8_t *Q, const int32_t *Z,
                         ResidualView rv, const int *active, int *accepted, int *status, int p,
                         int g, int i0, int nb, int qmax, float eps, cudaStream_t s);
cudaError_t launch_band(const __half *Htdig, int2 *band, int d, int d_pad, int g, cudaStream_t s);
cudaError_t launch_slice_rinv(const double *Rinv, __nv_bfloat16 *rdig, int *rexp, int d, int g,
                              cudaStream_t s);
cudaError_t launch_ptilde(const CUtensorMap &mapPd, const CUtensorMap &mapR, const float *Phi,
                          const float *Plo, __nv_bfloat16 *pdig, int *pexp, const int *rexp,
                          float *out_hi, float *out_lo, int p, int p_pad, int d, int d_pad, int g,
                          int *status, cudaStream_t s, bool stalled = false);
int target_splits(int p_pad, int g, int G, int nb);
cudaError_t launch_wait_timeout(int *status, uint32_t polls, cudaStream_t s);
cudaError_t launch_tc_target(const CUtensorMap &mapC, const CUtensorMap &mapT, float *out_hi,
                             float *out_lo, const float *S, const int *expoT, const int *active,
                             int p, int p_pad, int d_pad, int g, int G, int i0, int nb,
                             int nb_prev, int nsplit, int qmax, int *status, cudaStream_t s,
                             bool pdl, bool stalled = false);

// Launch; with `pdl` under programmatic stream serialization: the kernel may
// start while the previous kernel in the stream finishes, and must call
// griddepcontrol.wait before touching that kernel's inputs or outputs.
template <class... KArgs, class... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     bool pdl, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args &&>(args)...);
}
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args &&...args) {
    return launch_k(kernel, grid, block, smem, s, true, static_cast<Args &&>(args)...);
}
cudaError_t launch_init_rows(int *active, int *iters, int *accepted, int *ridge, int *rstat,
                             int p, cudaStream_t s);

// Multiprocessor count of the current device (cached per device ordinal).
int num_sms();

// Enable `bytes` of dynamic shared memory for `func` on the current device:
// the most that any call of it needs, since the limit is the process's and a
// smaller one, set by another thread, would refuse a launch on its way.
// The attribute is per device and a process may drive several devices, so
// `done` is a bit mask over device ordinals; ordinals of 64 and above set
// the attribute on every call.
cudaError_t set_max_dynamic_smem(const void *func, int bytes,
                                 std::atomic<unsigned long long> &done);

// True for managed memory, or device memory of the current device (a buffer
// on another GPU is false: the kernels would read a peer's memory).
bool on_device(const void *p);

// Makes `device` current for the guard's lifetime and then restores the
// caller's current device, so that an entry point never leaves the calling
// thread on another GPU.
class DeviceGuard {
  public:
    explicit DeviceGuard(int device) {
        if (cudaGetDevice(&prev_) != cudaSuccess) {
            (void)cudaGetLastError();
            return;
        }
        if (prev_ == device) {
            ok_ = true;
            return;
        }
        if (cudaSetDevice(device) == cudaSuccess) {
            ok_ = switched_ = true;
        } else {
            (void)cudaGetLastError();
        }
    }
    ~DeviceGuard() {
        if (switched_) cudaSetDevice(prev_);
    }
    bool ok() const { return ok_; }
    DeviceGuard(const DeviceGuard &) = delete;
    DeviceGuard &operator=(const DeviceGuard &) = delete;

  private:
    int prev_ = 0;
    bool ok_ = false, switched_ = false;
};

// A status word of the current device for the length of one call that has no
// handle: calls on other streams and host threads have other words, so a
// kernel may decide by its call's word whether to write.  The words are one
// static array; a call waits for a free one (each call ends by itself).
class StatusWord {
  public:
    explicit StatusWord(cudaStream_t s);
    // gives the word back, after the stream's work if read() has not waited
    ~StatusWord();
    int *ptr() const { return ptr_; }    // null: the device has no such array
    cudaError_t clear();                 // enqueued on the call's stream
    cudaError_t read(int *bits);         // the word after all of the stream's work
    StatusWord(const StatusWord &) = delete;
    StatusWord &operator=(const StatusWord &) = delete;

  private:
    cudaStream_t s_;
    int index_;
    int *ptr_ = nullptr;
    bool idle_ = true;
};

// 2D tensor map of 2-byte elements (bf16 or fp16) over [rows][cols]
// (pitch = cols elements), box_rows x box_cols boxes, box_cols = 64 with
// 128-byte swizzle or 32 with 64-byte swizzle, out-of-range elements read as
// zero.
cudaError_t make_tmap_2b(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                         uint32_t box_rows, CUtensorMapDataType dtype, uint32_t box_cols);
cudaError_t make_tmap_bf16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                           uint32_t box_rows, uint32_t box_cols = 64);
cudaError_t make_tmap_f16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                          uint32_t box_rows);

// ---- instrumentation (prof.cu) ----
void count_launches(int n);
void prof_collect();
// Records a CUDA event before construction and, on done(), after the
// launches it brackets, when profiling is enabled.
class ProfScope {
  public:
    ProfScope(const char *name, cudaStream_t s);
    void done();

  private:
    int id_;
    cudaStream_t s_;
    cudaEvent_t a_;
};

}  // namespace jarq
