// Internal declarations shared by the CUDA translation units of the library.
//
// Coordinates. Every product works on prescaled inputs xh_d = c_kind * x_d / l_d
// so that one kernel entry is a short register computation:
//   RBF:        c = sqrt(log2(e) / 2), rh2 = c^2 r^2,  k = 2^(log2 s^2 - rh2)
//   Matern-5/2: c = sqrt(5),           rh  = sqrt(5) r, k = (1 + rh + rh^2/3) 2^(log2 s^2 - rh log2 e)
// Both equal the standard forms k = s^2 exp(-r^2/2) and
// k = s^2 (1 + sqrt5 r + 5 r^2/3) exp(-sqrt5 r) with r^2 = sum_d ((x_d - x'_d)/l_d)^2.
// Lengthscale derivatives in the same coordinates: dk/dlog l_d = psi * (dxh_d)^2 with
//   RBF:        psi = 2 ln2 * k
//   Matern-5/2: psi = (1 + rh) * s^2 2^(-rh log2 e) / 3
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "device_once.cuh"
#include "lgp.h"

namespace lgp {

constexpr int kMaxD = 8;
constexpr int kMaxT = 64;
// Lanczos steps kept per column for the log-determinant quadrature (the quadrature kernel holds the
// tridiagonal in shared memory: 4 x 8 bytes per step)
constexpr int kMaxLanczos = 1024;
constexpr int kMaxRank = 32;  // largest pivoted-Cholesky preconditioner rank
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kTwoLn2 = 1.3862943611198906f;
constexpr float kLn2 = 0.6931471805599453f;

// Padded row width of the prescaled X buffer (floats): 4 for D <= 4, else 8.
inline int dpad_of(int D) { return D <= 4 ? 4 : 8; }

struct KernelParams {
    int kind;
    int D;
    int dpad;
    float log2_s2;   // log2(s^2)
    float s2;        // s^2
    float noise;     // sigma_n^2
    float scale[kMaxD];
};

// ---------------------------------------------------------------- device helpers

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Accumulates a * b into the float pair (hi, lo) without float64 arithmetic: the product's rounding
// error exactly by FMA (TwoProduct) and the running sum's by Knuth's TwoSum, as in the compensated
// dot product of Ogita, Rump and Oishi ("Accurate sum and dot product", SIAM J. Sci. Comput. 2005).
// Each operation is an explicitly rounded intrinsic, so the compiler cannot contract it into an FMA.
// hi + lo carries the partial sum to about 2^-44 relative; the block and column reductions then run in
// float64. (The float64 pipe of this GPU is slow enough that converting every element to double set
// the time of these kernels.)
__device__ __forceinline__ void acc_prod2(float &hi, float &lo, float a, float b) {
    const float p = __fmul_rn(a, b);
    const float pe = fmaf(a, b, -p);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, pe));
}

template <int KIND> struct Entry;

template <> struct Entry<LGP_RBF> {
    // k from the prescaled squared distance.
    static __device__ __forceinline__ float k(float rh2, float log2s2) { return ex2_approx(log2s2 - rh2); }
    // k and psi (dk/dlog l_d = psi * dxh_d^2).
    static __device__ __forceinline__ void k_psi(float rh2, float log2s2, float &k, float &psi) {
        k = ex2_approx(log2s2 - rh2);
        psi = kTwoLn2 * k;
    }
};

template <> struct Entry<LGP_MATERN52> {
    static __device__ __forceinline__ float k(float rh2, float log2s2) {
        const float rh = sqrt_approx(rh2);
        const float e = ex2_approx(fmaf(-rh, kLog2e, log2s2));
        const float poly = fmaf(rh2, 1.0f / 3.0f, rh) + 1.0f;
        return poly * e;
    }
    static __device__ __forceinline__ void k_psi(float rh2, float log2s2, float &k, float &psi) {
        const float rh = sqrt_approx(rh2);
        const float e = ex2_approx(fmaf(-rh, kLog2e, log2s2));
        const float poly = fmaf(rh2, 1.0f / 3.0f, rh) + 1.0f;
        k = poly * e;
        psi = (1.0f + rh) * e * (1.0f / 3.0f);
    }
};

// Matern-1/2 on x = log2(e) x / l: rh = r log2 e, k = 2^(log2 s^2 - rh). dk/dlog l_d = s^2 e^-r r_d^2 / r
// = k ln2 dxh_d^2 / rh for r > 0, and 0 at r = 0 (where every dxh_d is 0).
template <> struct Entry<LGP_MATERN12> {
    static __device__ __forceinline__ float k(float rh2, float log2s2) { return ex2_approx(log2s2 - sqrt_approx(rh2)); }
    static __device__ __forceinline__ void k_psi(float rh2, float log2s2, float &k, float &psi) {
        k = ex2_approx(log2s2 - sqrt_approx(rh2));
        psi = rh2 > 0.0f ? k * kLn2 * rsqrtf(rh2) : 0.0f;
    }
};

// Matern-3/2 on x = sqrt3 x / l: rh = sqrt3 r, k = (1 + rh) e with e = 2^(log2 s^2 - rh log2 e);
// dk/dlog l_d = 3 s^2 e^(-sqrt3 r) r_d^2 = e dxh_d^2.
template <> struct Entry<LGP_MATERN32> {
    static __device__ __forceinline__ float k(float rh2, float log2s2) {
        const float rh = sqrt_approx(rh2);
        const float e = ex2_approx(fmaf(-rh, kLog2e, log2s2));
        return fmaf(e, rh, e);
    }
    static __device__ __forceinline__ void k_psi(float rh2, float log2s2, float &k, float &psi) {
        const float rh = sqrt_approx(rh2);
        const float e = ex2_approx(fmaf(-rh, kLog2e, log2s2));
        k = fmaf(e, rh, e);
        psi = e;
    }
};

// Two entries at once from squared distances accumulated on packed float32x2 operations from acc0. The Matern entries take
// s^2 in their exponent's one multiply-add; RBF entries are k = 2^-(rh2 + acc0) with an ls2 of 0 (EntryScale), and s^2 goes
// into V or the finished sums: accumulated from -log2 s^2, each of the D additions rounds at that size (D = 8, s^2 = 100,
// entry error 2.6e-7 against 9e-8; more where the distances are small). (The start stays an operand: with a plain product for the
// first square the row kernel's schedule comes out 4% slower, N = 20000, D = 2, t = 48 1310 -> 1364 us.) Matern-5/2 uses
// k = e + e (rh + rh2 / 3). A packed operation on three different register pairs runs at half rate (mv_sym.cuh), so the
// multiply-adds by constants are scalar.
template <int KIND> struct PackedEntry;
template <> struct PackedEntry<LGP_RBF> {
    static __device__ __forceinline__ float2 acc0(float ls2) { return make_float2(-ls2, -ls2); }
    static __device__ __forceinline__ float2 k(float2 acc, float) { return make_float2(ex2_approx(-acc.x), ex2_approx(-acc.y)); }
};
template <> struct PackedEntry<LGP_MATERN52> {
    static __device__ __forceinline__ float2 acc0(float) { return make_float2(0.0f, 0.0f); }
    static __device__ __forceinline__ float2 k(float2 r2, float ls2) {
        const float2 r = make_float2(sqrt_approx(r2.x), sqrt_approx(r2.y));
        const float2 e = make_float2(ex2_approx(fmaf(r.x, -kLog2e, ls2)), ex2_approx(fmaf(r.y, -kLog2e, ls2)));
        const float2 q = make_float2(fmaf(r2.x, 1.0f / 3.0f, r.x), fmaf(r2.y, 1.0f / 3.0f, r.y));
        return __ffma2_rn(e, q, e);
    }
};
template <> struct PackedEntry<LGP_MATERN12> {
    static __device__ __forceinline__ float2 acc0(float) { return make_float2(0.0f, 0.0f); }
    static __device__ __forceinline__ float2 k(float2 r2, float ls2) {
        return make_float2(ex2_approx(ls2 - sqrt_approx(r2.x)), ex2_approx(ls2 - sqrt_approx(r2.y)));
    }
};
template <> struct PackedEntry<LGP_MATERN32> {
    static __device__ __forceinline__ float2 acc0(float) { return make_float2(0.0f, 0.0f); }
    static __device__ __forceinline__ float2 k(float2 r2, float ls2) {
        const float2 r = make_float2(sqrt_approx(r2.x), sqrt_approx(r2.y));
        const float2 e = make_float2(ex2_approx(fmaf(r.x, -kLog2e, ls2)), ex2_approx(fmaf(r.y, -kLog2e, ls2)));
        return __ffma2_rn(e, r, e);
    }
};

// The outputscale of the kernels on PackedEntry: log2 s^2 in the exponent (Matern), or for RBF s^2 as the factor of V (v, in
// the kernels) or of the finished sums (out, where the partial sums are added up), on the side where neither the products
// nor the sums can leave the float32 range that the full entries had.
struct EntryScale {
    float log2s2 = 0.0f, v = 1.0f, out = 1.0f;
};
inline EntryScale entry_scale(const KernelParams &kp) {
    EntryScale s;
    if (kp.kind != LGP_RBF) s.log2s2 = kp.log2_s2;
    else (kp.s2 < 1.0f ? s.v : s.out) = kp.s2;
    return s;
}

template <int KIND> __device__ __forceinline__ float rbf_scaled(float v, float scale) {
    if constexpr (KIND == LGP_RBF) return v * scale;
    else return v;
}

// Host: the kind is one the library implements.
inline bool kind_supported(int kind) {
    return kind == LGP_RBF || kind == LGP_MATERN52 || kind == LGP_MATERN12 || kind == LGP_MATERN32;
}

// Host: the factor c of the prescaled coordinates x = c x / l, chosen so that each entry needs one
// ex2: RBF sqrt(log2(e) / 2) (rh^2 = r^2 log2(e) / 2), M52 sqrt5, M32 sqrt3, M12 log2(e).
inline double prescale_of(int kind) {
    switch (kind) {
        case LGP_RBF: return 0.8493218002880191;     // sqrt(0.5 / ln 2)
        case LGP_MATERN52: return 2.23606797749979;  // sqrt 5
        case LGP_MATERN32: return 1.7320508075688772;  // sqrt 3
        case LGP_MATERN12: return 1.4426950408889634;  // log2 e
    }
    return 0.0;
}

// ---------------------------------------------------------------- chained launches

// A kernel whose first statement is chain_wait() may be launched with launch_chained: its CTAs are then placed while the
// previous kernel of the stream still runs its last ones, and wait here until that kernel has finished and its writes are
// visible. chain_wait comes before any access to memory and before any return (a kernel that ended without it could
// finish before its predecessor); its chain_next, from which on the successor may be placed, comes with it.
// When it came, a product call of N = 20000, D = 8, t = 16 (then with eight small kernels beside the product's): 168 -> 154 us;
// solve of N = 1024, t = 1 (two kernels an iteration): 945 -> 866 us.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

// Lets a kernel be launched with `bytes` of dynamic shared memory on the current device (set once per device).
template <class Kernel> cudaError_t allow_shared(DeviceOnce &once, Kernel kernel, int bytes) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || once.has(dev)) return e;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) == cudaSuccess) once.add(dev);
    return e;
}

// ---------------------------------------------------------------- CG state on the device

// Per-column CG scalars (float64) and flags, plus the Lanczos history.
struct CgState {
    int iter;          // iterations done (global counter)
    int done;          // 1 when no column is active or iter reached max_iter
    int status;        // 0 ok, else an lgp_status (breakdown / nonfinite)
    int max_iter;
    int hist_len;      // Lanczos steps kept per column
    int t;
    int loop_chunks;   // chunks run by the device-side while loop
    int max_chunks;    // hard cap on loop_chunks (the loop ends even if `done` were never set)
    double tol;
    int active[kMaxT];
    int iters[kMaxT];
    double bnorm2[kMaxT];
    double rr[kMaxT];
    double rz[kMaxT];  // r^T z with z = P^{-1} r (= rr without a preconditioner)
    double w0[kMaxT];  // b^T P^{-1} b: the Lanczos quadrature weight of each column
    double alpha[kMaxT];
    double beta[kMaxT];
    double thresh[kMaxT];       // a column stops once r^T r <= thresh = (tol ||b||)^2
    unsigned int rmax[kMaxT];   // float bits of max |r| after the last update (solves whose p is split here)
    unsigned int pmax[kMaxT];   // float bits of max |p|
    unsigned int ticket;        // blocks of the current kernel that have written their partial sums
};

// ---------------------------------------------------------------- launchers (defined in the .cu files)

// prep.cu
void launch_prep_x(const float *X, int64_t N, int D, int dpad, const float *scale_host, float *Xs, int64_t Np,
                   int *err_flag, cudaStream_t st, unsigned int *zero64 = nullptr, unsigned int *zero32 = nullptr);
void launch_rademacher(uint64_t seed, int64_t N, int m, float *Z, int64_t ldz, int col0, cudaStream_t st);
void launch_scan_finite(const float *A, int64_t n, int *err_flag, cudaStream_t st);
void launch_copy_cols(const float *src, int64_t lds, float *dst, int64_t ldd, int64_t rows, int cols, int dst_col0,
                      cudaStream_t st);

// predict.cu
void launch_kernel_cols(const KernelParams &kp, const float *Xh, int64_t N, int64_t Np, const float *Xsh, int64_t j0,
                        int tc, float *B, int64_t ldb, int col0, cudaStream_t st);
void launch_var_from_dots(const double *dots, int c0, int t, float s2, float *var, int64_t j0, cudaStream_t st);
void launch_var_from_probes(const float *Z, int64_t ldz, const float *Q, int64_t ldq, int64_t M, int m, float s2,
                            float *var, cudaStream_t st);

// What a product left for its caller to finish when asked to (the CG step, which reads the same rows anyway):
// S partial sums, out = scale sum_k part[k * stride + e] + noise V. part = nullptr: out is complete.
struct ProductTail {
    const float *part = nullptr;
    int S = 0;
    int64_t stride = 0;
    float scale = 1.0f, noise = 0.0f;
};

// mv_simt.cu
struct MvLaunch {
    const KernelParams *kp;
    const float *Xs;      // prescaled [Np, dpad]
    int64_t N, Np;
    const float *V;       // [N, ldv] (rows >= N are never read)
    int64_t ldv;
    float *out;           // [N, ldo]
    int64_t ldo;
    int t;
    float *partial;       // split-column partial sums (workspace) or nullptr
    int64_t partial_cap;  // floats available in partial
    const int *skip;      // device flag: skip all work when *skip != 0 (may be nullptr)
    int num_sms;
    // With tail set, column-split partial sums are left to the caller (see ProductTail).
    struct ProductTail *tail = nullptr;
    bool rows = false;    // the row-by-row kernel also where the symmetric one would run
    // Cross product out = K(Xr, Xs) V (no noise term): prescaled row points [Npr, dpad] and their
    // count; Xr == nullptr gives the square product K_y V.
    const float *Xr = nullptr;
    int64_t Nr = 0, Npr = 0;
};
cudaError_t launch_mv_simt(const MvLaunch &m, cudaStream_t st);
int64_t mv_simt_partial_floats(int64_t N, int64_t Np, int t, int D, int num_sms);
// Split partial floats of the cross product with Nr output rows (Npr padded) and N columns.
int64_t mv_simt_cross_partial_floats(int64_t Nr, int64_t Npr, int64_t N, int t, int num_sms);

cudaError_t launch_mv_grad(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, const float *W, int t,
                           float *G, float *partial, int64_t partial_cap, int num_sms, cudaStream_t st);
int64_t mv_grad_partial_floats(int64_t N, int64_t Np, int t, int D, int num_sms);

// Bilinear adjoint reduction: acc[p] = sum_ij dK_p[i,j] * (A_i . B_j) for p < D (lengthscales), p = D (log s^2).
cudaError_t launch_adjoint_bilinear(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, const float *A,
                                    const float *B, int t, double *block_partials, int64_t partial_cap, int *n_blocks,
                                    int num_sms, cudaStream_t st);
int64_t adjoint_partial_doubles(int64_t N, int t, int D, int num_sms);

// mv_tc.cu
bool tc_supported(int t);
int64_t tc_vsplit_bytes(int64_t Np, int t);
// fmt: 0 = bfloat16 halves, 1 = scaled float16 halves
// forced_splits > 0 overrides the column-split count (the autotuner's choice); 0 = wave-efficiency heuristic;
// kTcSymmetric = the symmetric-tile kernel (mv_tcs.cuh), which adds onto out instead of writing partials.
// kTcSymmetricDiff = the same, always in the difference form.
constexpr int kTcSymmetric = -1;
constexpr int kTcSymmetricDiff = -2;
// Words of tc_max_words in which nothing has been collected since launch_prep_x cleared them, but for this V and X.
struct TcZeroed {
    bool v = false, x = false;
};
// operands_ready: the operands that depend on X alone are already in vsplit (launch_tc_operands, once
// per prepared X): the transposed X and, where the symmetric product may take the dot form, its
// distance operands; otherwise the product builds them first.
// dist_form (symmetric product with the dot form allowed): -1 = not known on the host, so both distance
// instances launch and the device gate word lets one of them work; 0 / 1 = only the difference / dot
// instance launches (the caller read the gate word, which must then give the same answer).
// v_ready: V is already split in the workspace, and out of a symmetric product already holds sigma^2 V
// (launch_v_split, launch_p_split). tail (optional): see ProductTail. zeroed: see TcZeroed.
// ev_begin / ev_end (optional): recorded on st immediately before and after the product kernel's
// launch(es), after the V split and operand kernels (the kernel timing of lgp_last_kernel_ms).
cudaError_t launch_mv_tc(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, const float *V, int64_t ldv,
                         float *out, int64_t ldo, int t, int fmt, void *vsplit, float *partial, int64_t partial_cap,
                         const int *skip, int *err_flag, long long wait_budget, int num_sms, cudaStream_t st,
                         int forced_splits = 0, bool operands_ready = false, int dist_form = -1,
                         cudaEvent_t ev_begin = nullptr, cudaEvent_t ev_end = nullptr, bool v_ready = false,
                         ProductTail *tail = nullptr, TcZeroed zeroed = {});
// A CG solve's vector p as the split operand of its products (p row stride t, the workspace of one vsplit).
struct CgSplit {
    int fmt;
    uint16_t *vs;         // stacked [V_hi; V_lo]
    unsigned int *vmax;   // f16: per-column bound on |p| (float bits) that sets the scaling exponents
    float *col_scale;
    float s2;
    float *out_init;      // [N, t] set to noise * p (symmetric product), or nullptr
    float noise;
};
CgSplit tc_cg_split(const KernelParams &kp, int64_t Np, int t, int fmt, void *vsplit, float *out_init);
// The split operands of V (column maxima for f16, halves, scaling factors), and out_init = noise V if given.
cudaError_t launch_v_split(const KernelParams &kp, int64_t N, int64_t Np, const float *V, int64_t ldv, int t, int fmt,
                           void *vsplit, float *out_init, int64_t ldo, const int *skip, int num_sms, cudaStream_t st);
// p = r + beta p for the active columns and p's split operands, in one pass (the CG step's last launch).
cudaError_t launch_p_split(const CgSplit &sp, float *p, const float *r, int64_t N, int t, CgState *state, cudaStream_t st);
// The operands of the tensor-core products that depend on X alone, into the t-column V-split workspace:
// the transposed prescaled X, and with dot = true the dot-form distance data of the symmetric product
// (box, centred split operands, squared norms, the gate word).
cudaError_t launch_tc_operands(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, int t, void *vsplit, bool dot,
                               int num_sms, cudaStream_t st);
// The words in which the passes over V (64 words) and X (32 words) collect maxima
void tc_max_words(int64_t Np, int t, void *vsplit, unsigned int **vmax, unsigned int **words);
int64_t mv_tc_partial_floats(int64_t Np, int t, int num_sms);
int64_t mv_tc_partial_floats(int64_t Np, int t, int num_sms, int forced_splits);
// Up to four kernel choices worth timing: kTcSymmetric or kTcSymmetricDiff (when tc_symmetric_ok) and the three most
// wave-efficient split counts.
void tc_split_candidates(int64_t Np, int kind, int D, int num_sms, int *cand, int *n);
bool tc_symmetric_ok(int64_t Np);
// Dot-form distance of the symmetric product: whether it is considered for (kind, D), its limit on
// max |u|^2, and the byte offset of the word holding the measured max in the V-split workspace.
bool dot_form_allowed(int kind, int D);
float dot_gate_limit(int kind);
int64_t tc_dot_gate_offset(int64_t Np, int t);

// precond.cu: the rank-k pivoted-Cholesky preconditioner P = L L^T + sigma^2 I (k = 0: none).
struct Precond {
    int k = 0;
    int64_t Np = 0;                // row stride of the L columns
    const double *L64 = nullptr;   // [k][Np] (column q contiguous over rows)
    const float *L32 = nullptr;    // float32 copy used inside the CG iterations
    const double *Cinv = nullptr;  // [k][k] inverse of C = sigma^2 I + L^T L
    double *part = nullptr;        // [G][k t] block partials of L^T R
    double *U = nullptr;           // [k][t] C^{-1} L^T R
    int G = 0;                     // blocks of the L^T R reduction
    double noise = 0.0;
    double logdet = 0.0;           // log|P| = (N - k) log sigma^2 + log|C|
};

size_t pivinfo_bytes();
// k pivoted-Cholesky steps of K_ff from the raw float32 X [N, D] (float64 arithmetic): L64 [k][Np], residual d [Np]
void launch_pivchol(const float *X, int64_t N, int64_t Np, int D, const double *inv_ls_host, double s2, int kind,
                    int k, double *L64, double *d, void *pinfo, cudaStream_t st);
// Block partials [G][k * k] of L^T L
void launch_gram(const double *L64, int64_t Np, int64_t N, int k, double *partial, int G, cudaStream_t st);
void launch_to_f32(const double *src, float *dst, int64_t n, cudaStream_t st);
// Z = P^{-1} R for rows < N (t <= 32, k t <= 1024); Pcopy (may be null) receives Z too; rz_partial (may be
// null) gets [G_vec][t] block partials of r^T z; state (may be null) skips the work once the CG is done.
cudaError_t launch_precond_apply(const Precond &pc, const float *R, int64_t ldr, float *Z, int64_t ldz, float *Pcopy,
                          int64_t N, int t, double *rz_partial, int G_vec, const CgState *state, cudaStream_t st);
// rhs[:, col0 + c] = L E[N:, c] + sigma E[:N, c] for the [N + k, m] Rademacher block E
void launch_precond_probes(const double *L64, int64_t Np, int k, const float *E, int64_t N, int m, double sigma,
                           float *rhs, int64_t ldr, int col0, cudaStream_t st);

// solver.cu
struct CgBuffers {
    float *x, *r, *p, *Kp;   // [Np, t]
    float *z;                // [Np, t] P^{-1} r (preconditioned solves only)
    double *partial;         // block partial dots, cg_partial_doubles(G, t)
    int G;                   // blocks of the vector kernels
    CgState *state;
    double *hist_alpha;      // [hist_len, t]
    double *hist_beta;       // [hist_len, t]
    Precond pc;              // pc.k == 0: plain CG
};
// X0 (may be null): warm start x0 [N, ldx0], with K_y x0 already in b.Kp.
void launch_cg_init(const float *B, int64_t ldb, int64_t N, int64_t Np, int t, const CgBuffers &b, double tol,
                    int max_iter, int hist_len, cudaStream_t st, const float *X0 = nullptr, int64_t ldx0 = 0);
// cg_cluster.cu: the whole step after the product as one launch of a cluster, where the vectors and the S partial sums per
// element that the product left are few enough: its CTAs (1, 8 or 16), or 0 for three launches. wide: 16 are possible.
int cg_step_rule(int64_t N, int t, int S, bool wide);
int cg_step_ctas(int64_t N, int t, const CgBuffers &b, int S);
cudaError_t launch_cg_cluster(int ctas, int64_t N, int t, const CgBuffers &b, const ProductTail &tail, const CgSplit *split,
                              cudaStream_t st);
// One CG iteration after its product (b.Kp, or its partial sums in tail); split: p's halves for the next product.
cudaError_t launch_cg_after_matvec(int64_t N, int t, const CgBuffers &b, const ProductTail &tail, const CgSplit *split,
                                   cudaStream_t st);
void launch_cg_copy_out(const CgBuffers &b, int64_t N, int t, float *Xsol, int64_t ldx, cudaStream_t st);
// Column 0 of the single-column run b1 (state, first hist_len Lanczos coefficients) into column c of a
// t-column state and history; dst->loop_chunks accumulates.
void launch_cg_gather_column(const CgBuffers &b1, int hist_len, CgState *dst, double *dst_alpha, double *dst_beta,
                             int t, int c, cudaStream_t st);
// Body tail of the device-side CG loop: sets the while-node condition to "not done and under the chunk cap".
cudaError_t launch_cg_loop_condition(cudaGraphConditionalHandle h, CgState *state, cudaStream_t st);
// Host-driven loop (LGP_CG_GRAPH=0): counts one chunk in state->loop_chunks.
cudaError_t launch_cg_chunk_tally(CgState *state, cudaStream_t st);
int cg_num_blocks(int64_t N, int t, int num_sms);
int64_t cg_partial_doubles(int G, int t);

// Column dot products sum_i A[i,c] B[i,c] and sum_i A[i,c]^2 (float64), c < t: out[2t].
void launch_col_dots(const float *A, const float *B, int64_t N, int t, double *partial, int G, double *out,
                     cudaStream_t st);
// Stochastic Lanczos quadrature over probe columns 1..t-1 and the LML assembly.
// out: [0] lml, [1] quad, [2] logdet, [3] status flag (0 ok, else nonpositive Ritz value)
void launch_slq_lml(const CgBuffers &b, int t, int hist_len, const double *dots, int64_t N, double *out,
                    cudaStream_t st);
// B'[:,0] = A[:,0]; B'[:,c] = -Z[:,c] / m for c >= 1 (the right factor of the gradient's bilinear form)
void launch_adjoint_rhs(const float *A, const float *RHS, int64_t N, int t, float *Bp, cudaStream_t st);
// Sum block partials and form grad[p] = 1/2 acc[p] (p <= D); grad[D+1] from the noise term.
void launch_grad_finalize(const double *block_partials, int n_blocks, int D, const double *dots, int t, float noise,
                          double *grad_out, cudaStream_t st);

}  // namespace lgp
