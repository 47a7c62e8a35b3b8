// Conjugate-gradient vector updates, float64 scalar recurrences, stochastic Lanczos
// quadrature and the LML / gradient assembly.
//
// CG (Sec. 2 "CG-based inference"; Sec. 5 "our simpler CG loop"): x0 = 0, one recurrence per
// right-hand-side column, all columns advanced by the same launches. Per iteration, after
// Kp = K_y p, with z = P^{-1} r (z = r without a preconditioner):
//   alpha_c = r_c^T z_c / p_c^T Kp_c,  x_c += alpha_c p_c,  r_c -= alpha_c Kp_c,
//   z_c' = P^{-1} r_c',  beta_c = r_c'^T z_c' / r_c^T z_c,  p_c = z_c' + beta_c p_c,
// column c stops once ||r_c|| <= tol ||b_c||. The optional preconditioner is the pivoted-Cholesky
// P of precond.cu (the gap Sec. 5 names; plain CG is the paper's loop). Vectors are float32; a dot product's sum is
// carried as a float pair within a thread, without rounding across a block's threads (limb_sum.cuh) and in float64 across
// blocks, in index order, so results are reproducible run to run.
#include <math.h>

#include <algorithm>

#include "cg_reduce.cuh"

namespace lgp {

namespace {

constexpr int kVecThreads = 256;

// Threads per block for column-interleaved work: a multiple of t not above 256.
__host__ __device__ inline int vec_block(int t) { return (kVecThreads / t) * t; }

// Block-level per-column reduction of vals (one per thread, column tid % t) into out[c].
__device__ void block_col_reduce(double v, int t, double *red, double *out_row) {
    const int tid = threadIdx.x;
    const int nr = blockDim.x / t;
    red[tid] = v;
    __syncthreads();
    int s = 1;
    while (s < nr) s <<= 1;
    for (s >>= 1; s >= 1; s >>= 1) {
        const int slot = tid / t;
        if (slot < s && slot + s < nr) red[tid] += red[tid + s * t];
        __syncthreads();
    }
    if (tid < t) out_row[tid] = red[tid];
}

// Sum of partial[b * stride + c] over b < G by one warp: lane l adds b = l, l + 32, ... in order,
// then a fixed shuffle tree combines the lanes (same order every call).
__device__ __forceinline__ double warp_sum_partials(const double *__restrict__ partial, int G, int stride, int c) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int b = lane; b < G; b += 32) s += partial[(int64_t)b * stride + c];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    return __shfl_sync(0xffffffffu, s, 0);
}

// Row range of block b when G blocks share N rows.
__device__ __forceinline__ void block_rows(int64_t N, int64_t *r0, int64_t *r1) {
    const int64_t per = (N + gridDim.x - 1) / gridDim.x;
    *r0 = min(N, (int64_t)blockIdx.x * per);
    *r1 = min(N, *r0 + per);
}

__global__ void cg_init_kernel(const float *__restrict__ B, int64_t ldb, int64_t N, int t, float *__restrict__ x,
                               float *__restrict__ r, float *__restrict__ p, double *__restrict__ partial) {
    __shared__ double red[kVecThreads];
    int64_t r0, r1;
    block_rows(N, &r0, &r1);
    const int c = threadIdx.x % t;
    double s = 0.0;
    for (int64_t i = r0 + threadIdx.x / t; i < r1; i += blockDim.x / t) {
        const float b = B[i * ldb + c];
        x[i * t + c] = 0.0f;
        r[i * t + c] = b;
        p[i * t + c] = b;
        s += (double)b * (double)b;
    }
    block_col_reduce(s, t, red, partial + (int64_t)blockIdx.x * t);
}

// Warm start: x = x0, r = b - K_y x0 (KX0 = K_y x0 computed before), p = r; block partials of
// b^T b (partial) and r^T r (rr_partial).
__global__ void cg_init_x0_kernel(const float *__restrict__ B, int64_t ldb, const float *__restrict__ X0, int64_t ldx0,
                                  const float *__restrict__ KX0, int64_t N, int t, float *__restrict__ x,
                                  float *__restrict__ r, float *__restrict__ p, double *__restrict__ partial,
                                  double *__restrict__ rr_partial) {
    __shared__ double red[kVecThreads];
    int64_t r0, r1;
    block_rows(N, &r0, &r1);
    const int c = threadIdx.x % t;
    double sb = 0.0, sr = 0.0;
    for (int64_t i = r0 + threadIdx.x / t; i < r1; i += blockDim.x / t) {
        const float b = B[i * ldb + c];
        const float rv = b - KX0[i * t + c];
        x[i * t + c] = X0[i * ldx0 + c];
        r[i * t + c] = rv;
        p[i * t + c] = rv;
        sb += (double)b * (double)b;
        sr += (double)rv * (double)rv;
    }
    block_col_reduce(sb, t, red, partial + (int64_t)blockIdx.x * t);
    __syncthreads();
    block_col_reduce(sr, t, red, rr_partial + (int64_t)blockIdx.x * t);
}

// Scalar kernels run as one block of 32 * min(t, 32) threads: warp w owns columns w, w + 32.
__global__ void cg_init_scalars_kernel(CgState *st, const double *__restrict__ partial, int G, int t, double tol,
                                       int max_iter, int hist_len, const double *__restrict__ rz_partial,
                                       const double *__restrict__ rr_partial) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    int any = 0;
    int bad = 0;
    for (int c = warp; c < t; c += nw) {
        const double s = warp_sum_partials(partial, G, t, c);
        const double rr0 = rr_partial ? warp_sum_partials(rr_partial, G, t, c) : s;
        const double rz = rz_partial ? warp_sum_partials(rz_partial, G, t, c) : rr0;
        if (lane != 0) continue;
        st->bnorm2[c] = s;
        st->rr[c] = rr0;
        st->rz[c] = rz;
        st->w0[c] = rz;
        const double root = tol * sqrt(s);
        st->thresh[c] = root * root;
        st->rmax[c] = st->pmax[c] = 0u;
        st->alpha[c] = 0.0;
        st->beta[c] = 0.0;
        st->iters[c] = 0;
        const int b_ = !isfinite(s) || !isfinite(rz) || !isfinite(rr0);
        bad |= b_;
        // a warm start that already meets the tolerance leaves the column inactive
        const int act = (s > 0.0) && (rz > 0.0) && !b_ && (sqrt(rr0) > tol * sqrt(s));
        st->active[c] = act;
        any |= act;
    }
    any = __syncthreads_or(any);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        st->iter = 0;
        st->ticket = 0u;
        st->t = t;
        st->tol = tol;
        st->max_iter = max_iter;
        st->hist_len = hist_len;
        st->status = bad ? (int)LGP_ERR_NONFINITE : 0;
        st->done = (!any || bad) ? 1 : 0;
        st->loop_chunks = 0;
        st->max_chunks = max_iter / 8 + 2;
    }
}

// ---------------------------------------------------------------- one CG iteration after the product
//
// Three launches: pkp_alpha (Kp from the product's column-split partial sums if it left any, p^T Kp, and in the last
// block to finish alpha), xr_beta (x, r, r^T r, the columns' max |r|; last block: beta, convergence, the loop's done
// flag) and p (p, and for the tensor-core products its split halves and the sigma^2 p that their out starts from).
// What bounds them: up to a few MB per vector the launches and the chain of loads, block reduction and float64
// reduction, not bandwidth. Hence few launches, 16-byte loads in blocks of 1024 threads, integer sums up to one value per
// block and column (cg_reduce.cuh), and at most kStepBlocks float64 values per column: one float64 warp instruction takes 64
// cycles of a sub-partition here, so a square root per column would cost more than all the loads (the test of convergence
// compares squares).
// Measured a solve / training step: N = 1024, t = 1, ~90 iterations 2.33 -> 1.83 ms; N = 2000, D = 8, t = 16 6.5 -> 4.7 ms;
// prediction at N = 8000, t = 32 (with the product's own gain) 16.7 -> 13.2 ms.

constexpr int kStepThreads = 1024;
constexpr int kStepBlocks = 76;  // half the SMs: each SM's load rate still covers L2, and half the float64 sums

// Whether this block is the last of the grid to arrive (its partials written before); resets the counter.
__device__ bool last_block(unsigned int *ticket) {
    __shared__ int last;
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int k = atomicAdd(ticket, 1u);
        last = k == gridDim.x - 1;
        if (last) *ticket = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
}

// Column sums of partial[b * t + c] over the grid's blocks, in a fixed order; valid in threads c < t after the call.
__device__ double grid_col_sum(const double *partial, int t, double *red) {
    const int G = gridDim.x, tid = threadIdx.x;
    if (G == 1) return tid < t ? partial[tid] : 0.0;
    int slots = 128 / t;  // t <= 64
    if (slots > 8) slots = 8;
    if (slots > G) slots = G;
    if (tid < slots * t) {
        const int slot = tid / t, c = tid - slot * t;
        double s = 0.0;
        for (int b = slot; b < G; b += slots) s += __ldcg(partial + (int64_t)b * t + c);
        red[tid] = s;
    }
    __syncthreads();
    double s = 0.0;
    if (tid < t)
        for (int k = 0; k < slots; ++k) s += red[k * t + tid];
    return s;
}

// Elements e (multiples of VEC) of a block's grid-stride loop over [0, N t). The vectors hold Np t >= N t values, so
// a last float4 that crosses N t stays inside them; its elements past N t are left out of the sums.
#define LGP_STEP_LOOP(e)                                                                                              \
    for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * VEC; e < total;                                \
         e += (int64_t)gridDim.x * blockDim.x * VEC)

// LANES > 0: Kp = scale sum_k part[k] + noise p first (S partial sums, part_stride apart), LANES lanes of a warp sharing the
// partial sums of each VEC elements (8 where there are many, so that their loads overlap).
template <int VEC, int LANES>
__global__ void __launch_bounds__(kStepThreads) cg_pkp_alpha_kernel(const float *__restrict__ p, float *__restrict__ Kp,
                                                                    const float *__restrict__ part, int S,
                                                                    int64_t part_stride, float scale, float noise, int64_t N, int t,
                                                                    CgState *st, double *__restrict__ partial,
                                                                    double *__restrict__ hist_alpha) {
    __shared__ float2 red[kStepThreads / 8 * 4];  // LANES = 8: element threads' sums; the grid sum's 128 doubles
    __shared__ ColSums acc;
    chain_wait();
    chain_next();
    if (st->done) return;
    clear_sums(acc);
    __syncthreads();
    const int64_t total = N * t;
    // LANES = 8: element thread u of the block's blockDim / 8 is lanes with (lane & 3) = u mod 4 of warp u / 4
    constexpr int L = LANES > 1 ? LANES : 1;
    const int sub = L > 1 ? (threadIdx.x & 31) / (32 / L) : 0;
    const int u = L > 1 ? (int)(threadIdx.x >> 5) * (32 / L) + (int)(threadIdx.x & (32 / L - 1)) : (int)threadIdx.x;
    const int nu = blockDim.x / L;
    float hi[VEC], lo[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) hi[k] = lo[k] = 0.0f;
    // (with L > 1 every lane of a warp runs the same rounds: the bound is its first element thread's)
    for (int64_t e0 = ((int64_t)blockIdx.x * nu + (L > 1 ? u - (u & (32 / L - 1)) : u)) * VEC; e0 < total;
         e0 += (int64_t)gridDim.x * nu * VEC) {
        const int64_t e = e0 + (L > 1 ? (u & (32 / L - 1)) * VEC : 0);
        const bool in = L == 1 || e < total;
        float pv[VEC], kv[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) pv[k] = kv[k] = 0.0f;
        if (in) load_vec<VEC>(p + e, pv);
        if constexpr (LANES > 0) {
            if (in) {
#pragma unroll 4
                for (int q = sub; q < S; q += L) {
                    float w[VEC];
                    load_vec<VEC>(part + q * part_stride + e, w);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) kv[k] += w[k];
                }
            }
            if constexpr (L > 1) {
#pragma unroll
                for (int off = 32 / L; off < 32; off <<= 1)
#pragma unroll
                    for (int k = 0; k < VEC; ++k) kv[k] += __shfl_xor_sync(0xffffffffu, kv[k], off);
            }
#pragma unroll
            for (int k = 0; k < VEC; ++k) kv[k] = fmaf(noise, pv[k], scale * kv[k]);
            if (in && sub == 0) store_vec<VEC>(Kp + e, kv);
        } else {
            load_vec<VEC>(Kp + e, kv);
        }
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < VEC; ++k)
                if (VEC == 1 || e + k < total) acc_prod2(hi[k], lo[k], pv[k], kv[k]);
        }
    }
    if constexpr (L > 1) {
        // element thread u's sums to thread u, whose columns they have
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) red[u * VEC + k] = make_float2(hi[k], lo[k]);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float2 v = (int)threadIdx.x < nu ? red[threadIdx.x * VEC + k] : make_float2(0.0f, 0.0f);
            hi[k] = v.x;
            lo[k] = v.y;
        }
        __syncthreads();
    }
    block_col_sums<VEC>(hi, lo, t, acc, partial + (int64_t)blockIdx.x * t);
    if (!last_block(&st->ticket)) return;
    const double pkp = grid_col_sum(partial, t, reinterpret_cast<double *>(red));
    const int c = threadIdx.x;
    int bad = 0, nonfinite = 0;
    if (c < t) {
        double alpha = 0.0;
        if (st->active[c]) {
            if (!isfinite(pkp)) {
                nonfinite = 1;
                st->active[c] = 0;
            } else if (!(pkp > 0.0)) {
                bad = 1;
                st->active[c] = 0;
            } else {
                alpha = st->rz[c] / pkp;
            }
        }
        st->alpha[c] = alpha;
        if (st->iter < st->hist_len) hist_alpha[(int64_t)st->iter * t + c] = alpha;
    }
    bad = __syncthreads_or(bad);
    nonfinite = __syncthreads_or(nonfinite);
    if (threadIdx.x == 0 && (bad || nonfinite) && st->status == 0)
        st->status = nonfinite ? (int)LGP_ERR_NONFINITE : (int)LGP_ERR_BREAKDOWN;
}

// beta, convergence and the done flag from the columns' r^T r and r^T z (threads c < t of one block). vbound (may be
// null): the bound on max |p| after the update, |r| + |beta| |p|, from which the tensor-core products scale p's columns.
__device__ void finish_beta(CgState *st, double rr, double rz, int t, double *hist_beta, unsigned int *vbound) {
    const int c = threadIdx.x;
    int any = 0;
    if (c < t) {
        double beta = 0.0;
        if (st->active[c]) {
            beta = rz / st->rz[c];
            st->rr[c] = rr;
            st->rz[c] = rz;
            st->iters[c] += 1;
            if (!(rr > st->thresh[c])) st->active[c] = 0;
            if (vbound && st->active[c]) {
                const float b = fmaf((float)beta, __uint_as_float(st->pmax[c]), __uint_as_float(st->rmax[c]));
                vbound[c] = __float_as_uint(b * 1.000001f);  // above the rounding of the update itself
                st->pmax[c] = 0u;
            }
        }
        st->rmax[c] = 0u;
        st->beta[c] = beta;
        if (st->iter < st->hist_len) hist_beta[(int64_t)st->iter * t + c] = beta;
        any = st->active[c];
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        st->iter += 1;
        if (!any || st->iter >= st->max_iter) st->done = 1;
    }
}

// FINISH: the last block computes beta (plain CG; the preconditioned one needs r^T z first, cg_beta_kernel).
template <int VEC, bool FINISH>
__global__ void __launch_bounds__(kStepThreads) cg_xr_beta_kernel(float *__restrict__ x, float *__restrict__ r,
                                                                  const float *__restrict__ p,
                                                                  const float *__restrict__ Kp, int64_t N, int t,
                                                                  CgState *st, double *__restrict__ partial,
                                                                  double *__restrict__ hist_beta, unsigned int *vbound) {
    __shared__ double red[128];
    __shared__ ColSums acc;
    __shared__ unsigned int rmax[kMaxT];
    chain_wait();
    chain_next();
    if (st->done) return;
    const int64_t total = N * t;
    float alpha[VEC], hi[VEC], lo[VEC], m[VEC];
    bool any = false;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        alpha[k] = (float)st->alpha[col_of<VEC>(threadIdx.x, k, t)];
        any |= alpha[k] != 0.0f;
        hi[k] = lo[k] = m[k] = 0.0f;
    }
    if (threadIdx.x < kMaxT) rmax[threadIdx.x] = 0u;
    clear_sums(acc);
    __syncthreads();
    LGP_STEP_LOOP(e) {
        float rv[VEC];
        load_vec<VEC>(r + e, rv);
        if (any) {
            float xv[VEC], pv[VEC], kv[VEC];
            load_vec<VEC>(x + e, xv);
            load_vec<VEC>(p + e, pv);
            load_vec<VEC>(Kp + e, kv);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (alpha[k] != 0.0f) {
                    xv[k] = fmaf(alpha[k], pv[k], xv[k]);
                    rv[k] = fmaf(-alpha[k], kv[k], rv[k]);
                }
            }
            store_vec<VEC>(x + e, xv);
            store_vec<VEC>(r + e, rv);
        }
#pragma unroll
        for (int k = 0; k < VEC; ++k)
            if (VEC == 1 || e + k < total) {
                acc_prod2(hi[k], lo[k], rv[k], rv[k]);
                m[k] = fmaxf(m[k], fabsf(rv[k]));
            }
    }
    if (vbound) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) atomicMax(&rmax[col_of<VEC>(threadIdx.x, k, t)], __float_as_uint(m[k]));
    }
    block_col_sums<VEC>(hi, lo, t, acc, partial + (int64_t)blockIdx.x * t);
    if (vbound && (int)threadIdx.x < t) atomicMax(&st->rmax[threadIdx.x], rmax[threadIdx.x]);
    if constexpr (FINISH) {
        if (!last_block(&st->ticket)) return;
        const double rr = grid_col_sum(partial, t, red);
        finish_beta(st, rr, rr, t, hist_beta, vbound);
    }
}

// Preconditioned CG: one block sums the r^T r partials (G_rr blocks) and the r^T z partials (G_rz) and finishes beta.
__global__ void __launch_bounds__(1024) cg_beta_kernel(CgState *st, const double *__restrict__ rr_partial, int G_rr,
                                                       const double *__restrict__ rz_partial, int G_rz, int t,
                                                       double *hist_beta) {
    __shared__ double srr[kMaxT], srz[kMaxT];
    chain_wait();
    chain_next();
    if (st->done) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int c = warp; c < t; c += nw) {
        const double rr = warp_sum_partials(rr_partial, G_rr, t, c);
        const double rz = warp_sum_partials(rz_partial, G_rz, t, c);
        if (lane == 0) {
            srr[c] = rr;
            srz[c] = rz;
        }
    }
    __syncthreads();
    const int c = threadIdx.x < t ? threadIdx.x : 0;
    finish_beta(st, srr[c], srz[c], t, hist_beta, nullptr);
}

template <int VEC>
__global__ void __launch_bounds__(kStepThreads) cg_p_kernel(float *__restrict__ p, const float *__restrict__ z, int64_t N,
                                                            int t, const CgState *st) {
    chain_wait();
    chain_next();
    if (st->done) return;
    const int64_t total = N * t;
    float beta[VEC];
    int act[VEC];
    int any = 0;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        const int c = col_of<VEC>(threadIdx.x, k, t);
        act[k] = st->active[c];
        any |= act[k];
        beta[k] = (float)st->beta[c];
    }
    if (!any) return;
    LGP_STEP_LOOP(e) {
        float pv[VEC], zv[VEC];
        load_vec<VEC>(p + e, pv);
        load_vec<VEC>(z + e, zv);
#pragma unroll
        for (int k = 0; k < VEC; ++k)
            if (act[k]) pv[k] = fmaf(beta[k], pv[k], zv[k]);
        store_vec<VEC>(p + e, pv);
    }
}

__global__ void cg_loop_condition_kernel(cudaGraphConditionalHandle h, CgState *st) {
    st->loop_chunks += 1;
    const bool more = !st->done && st->loop_chunks < st->max_chunks;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

// Host-driven form of the loop tail (no graph): only counts the chunk.
__global__ void cg_chunk_tally_kernel(CgState *st) { st->loop_chunks += 1; }

// Single-column solves assembled into one t-column result: column 0 of a t = 1 CG run (its state
// and the first hist_len Lanczos coefficients) becomes column c of dst; chunk counts add up.
__global__ void cg_gather_column_kernel(const CgState *__restrict__ src, const double *__restrict__ src_alpha,
                                        const double *__restrict__ src_beta, int hist_len, CgState *dst,
                                        double *__restrict__ dst_alpha, double *__restrict__ dst_beta, int t, int c) {
    for (int k = threadIdx.x; k < hist_len; k += blockDim.x) {
        dst_alpha[(int64_t)k * t + c] = src_alpha[k];
        dst_beta[(int64_t)k * t + c] = src_beta[k];
    }
    if (threadIdx.x == 0) {
        dst->active[c] = src->active[0];
        dst->iters[c] = src->iters[0];
        dst->bnorm2[c] = src->bnorm2[0];
        dst->rr[c] = src->rr[0];
        dst->rz[c] = src->rz[0];
        dst->w0[c] = src->w0[0];
        dst->alpha[c] = src->alpha[0];
        dst->beta[c] = src->beta[0];
        dst->loop_chunks += src->loop_chunks;
        dst->iter = max(dst->iter, src->iter);
        if (src->status != 0 && dst->status == 0) dst->status = src->status;
        dst->t = t;
        dst->hist_len = hist_len;
    }
}

__global__ void copy_out_kernel(const float *__restrict__ x, int64_t N, int t, float *__restrict__ out, int64_t ldo) {
    const int64_t total = N * t;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / t;
        const int c = (int)(e - i * t);
        out[i * ldo + c] = x[e];
    }
}

__global__ void col_dots_kernel(const float *__restrict__ A, const float *__restrict__ B, int64_t N, int t,
                                double *__restrict__ partial) {
    __shared__ double red[kVecThreads];
    int64_t r0, r1;
    block_rows(N, &r0, &r1);
    const int c = threadIdx.x % t;
    double sab = 0.0, saa = 0.0;
    for (int64_t i = r0 + threadIdx.x / t; i < r1; i += blockDim.x / t) {
        const double a = A[i * t + c];
        sab += a * (double)B[i * t + c];
        saa += a * a;
    }
    block_col_reduce(sab, t, red, partial + (int64_t)blockIdx.x * 2 * t);
    __syncthreads();
    block_col_reduce(saa, t, red, partial + (int64_t)blockIdx.x * 2 * t + t);
}

__global__ void col_dots_final_kernel(const double *__restrict__ partial, int G, int t, double *out) {
    const int c = threadIdx.x;
    if (c >= 2 * t) return;
    double s = 0.0;
    for (int b = 0; b < G; ++b) s += partial[(int64_t)b * 2 * t + c];
    out[c] = s;
}

// e_1^T log(T) e_1 of each probe's Lanczos tridiagonal, the Gauss quadrature of the stochastic
// log-determinant (Sec. 3 "Inference"), without an eigendecomposition of T. For lambda > 0,
//   log lambda = int_R [s(v) - s(v - log lambda)] dv,   s(v) = 1 / (1 + e^-v),
// so with x = e^v and g(x) = e_1^T (T + x I)^{-1} e_1 = sum_j u_1j^2 / (lambda_j + x),
//   e_1^T log(T) e_1 = int_R [x / (1 + x) - x g(x)] dv.
// The integrand is a sum of differences of logistic functions: analytic in the strip |Im v| < pi
// and decaying like e^-|v| outside [log lambda_min, log lambda_max], so the trapezoidal rule with
// step h on [log lambda_lo - 36, log lambda_hi + 36] has discretisation error ~exp(-2 pi^2 / h)
// (8e-18 at h = 0.5) and truncation error ~e^-36 (Trefethen & Weideman, "The exponentially
// convergent trapezoidal rule", SIAM Review 2014). Bounds: lambda_max <= the Gershgorin bound of T;
// lambda_min >= 1 / tr(T^-1), where T = L D L^T with D = diag(1/alpha_k) and unit lower bidiagonal L
// of subdiagonal sqrt(beta_k) (the CG-Lanczos factorisation), which gives
// tr(T^-1) = sum_i alpha_i s_i, s_0 = 1, s_i = 1 + beta_{i-1} s_{i-1}.
// At each node g(x) = P_2 / P_1 with the trailing minors P_k = det((T + x I)[k:m, k:m]) from the
// division-free recurrence P_k = (a_k + x) P_{k+1} - b_k^2 P_{k+2}, rescaled by powers of two, and
//   x / (1 + x) - x P_2 / P_1 = x ((a_1 - 1) P_2 - b_1^2 P_3) / ((1 + x) P_1)
// (P_1 expanded along its first row), which has no cancellation between the two terms. All of it is
// float64: every thread of the block evaluates its own nodes, so each float64 instruction does the
// work of all its lanes on a part whose float64 rate is low.
constexpr int kSlqThreads = 256;
constexpr double kSlqStep = 0.5;   // h
constexpr double kSlqTail = 36.0;  // trapezoidal range beyond the spectrum bounds, in log units

// (p0, p1, p2) scaled by the power of two that brings max(|p0|, |p1|) into [1, 2): exact.
__device__ __forceinline__ void rescale_pow2(double &p0, double &p1, double &p2) {
    const double mx = fmax(fabs(p0), fabs(p1));
    if (!(mx > 0.0) || !isfinite(mx)) return;
    const int e = ((__double2hiint(mx) >> 20) & 0x7ff) - 1023;
    if (e <= -1022 || e >= 1023) return;
    const double sc = __hiloint2double((1023 - e) << 20, 0);
    p0 *= sc;
    p1 *= sc;
    p2 *= sc;
}

// One block per probe column c = blockIdx.x + 1: gamma_c = w_c e_1^T log(T_c) e_1 with
// w_c = z_c^T P^{-1} z_c (||z_c||^2 without a preconditioner), T_c from the first
// m = min(L, iterations of c) CG coefficients: T[k,k] = 1/alpha_k + beta_{k-1}/alpha_{k-1},
// T[k,k+1] = sqrt(beta_k)/alpha_k. Writes gamma[c] and bad[c] (1 if T_c is not positive definite
// or a value is not finite). Summation order is fixed.
__global__ void __launch_bounds__(kSlqThreads) slq_quad_kernel(const CgState *st, const double *__restrict__ hist_alpha,
                                                               const double *__restrict__ hist_beta, int t,
                                                               int hist_len, double *__restrict__ gamma,
                                                               double *__restrict__ bad) {
    __shared__ double sa[kMaxLanczos], sbb[kMaxLanczos], sal[kMaxLanczos], sbe[kMaxLanczos];
    __shared__ double red[kSlqThreads];
    __shared__ double s_vlo;
    __shared__ int s_nodes, s_bad;
    const int c = blockIdx.x + 1;
    const int tid = threadIdx.x;
    const int m = min(hist_len, st->iters[c]);
    if (m <= 0) {
        if (tid == 0) {
            gamma[c] = 0.0;
            bad[c] = 0.0;
        }
        return;
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int k = tid; k < m; k += kSlqThreads) {
        const double al = hist_alpha[(int64_t)k * t + c];
        const double be = hist_beta[(int64_t)k * t + c];
        sal[k] = al;
        sbe[k] = be;
        if (!(al > 0.0) || !isfinite(al) || (k + 1 < m && (!(be >= 0.0) || !isfinite(be)))) atomicOr(&s_bad, 1);
    }
    __syncthreads();
    for (int k = tid; k < m; k += kSlqThreads) {
        double a = 1.0 / sal[k];
        if (k > 0) a += sbe[k - 1] / sal[k - 1];
        sa[k] = a;
        sbb[k] = k + 1 < m ? sbe[k] / (sal[k] * sal[k]) : 0.0;  // b_k^2
    }
    __syncthreads();
    // Gershgorin upper bound of the spectrum (max reduction over the rows)
    double g = 0.0;
    for (int k = tid; k < m; k += kSlqThreads) {
        double gk = sa[k];
        if (k > 0) gk += sqrt(sbb[k - 1]);
        if (k + 1 < m) gk += sqrt(sbb[k]);
        g = fmax(g, gk);
    }
    red[tid] = g;
    __syncthreads();
    for (int s = kSlqThreads / 2; s > 0; s >>= 1) {
        if (tid < s) red[tid] = fmax(red[tid], red[tid + s]);
        __syncthreads();
    }
    if (tid == 0) {
        const double lam_hi = red[0];
        double sk = 1.0, tr = sal[0];
        for (int i = 1; i < m; ++i) {
            sk = fma(sbe[i - 1], sk, 1.0);
            tr = fma(sal[i], sk, tr);
        }
        const double lam_lo = 1.0 / tr;
        if (!(lam_hi > 0.0) || !isfinite(lam_hi) || !(lam_lo > 0.0) || !isfinite(tr)) s_bad = 1;
        const double vlo = log(lam_lo) - kSlqTail;
        const double vhi = log(lam_hi) + kSlqTail;
        s_vlo = vlo;
        s_nodes = s_bad ? 0 : (int)ceil((vhi - vlo) / kSlqStep) + 1;
    }
    __syncthreads();
    const int nodes = s_nodes;
    const double a1m1 = sa[0] - 1.0, b1sq = sbb[0];
    double acc = 0.0;
    int nonpos = 0;
    for (int n = tid; n < nodes; n += kSlqThreads) {
        const double x = exp(s_vlo + n * kSlqStep);
        double p0 = sa[m - 1] + x, p1 = 1.0, p2 = 0.0;  // (P_k, P_{k+1}, P_{k+2}) at k = m
        for (int k = m - 2, q = 0; k >= 0; --k, ++q) {
            p2 = p1;
            p1 = p0;
            p0 = fma(sa[k] + x, p1, -sbb[k] * p2);
            if ((q & 3) == 3) rescale_pow2(p0, p1, p2);
        }
        if (!(p0 > 0.0)) nonpos = 1;  // T + x I positive definite: every trailing minor is positive
        acc += x * fma(a1m1, p1, -b1sq * p2) / ((1.0 + x) * p0);
    }
    if (nonpos) atomicOr(&s_bad, 1);
    red[tid] = acc;
    __syncthreads();
    for (int s = kSlqThreads / 2; s > 0; s >>= 1) {
        if (tid < s) red[tid] += red[tid + s];
        __syncthreads();
    }
    if (tid == 0) {
        const double v = st->w0[c] * kSlqStep * red[0];
        gamma[c] = v;
        bad[c] = (s_bad || !isfinite(v)) ? 1.0 : 0.0;
    }
}

// logdet = logdet_P + mean_c gamma_c (logdet_P = log|P|, 0 without a preconditioner);
// LML = -1/2 (y^T K_y^{-1} y + logdet + N log 2 pi). Sums in column order.
__global__ void slq_lml_finish_kernel(const double *__restrict__ gamma, const double *__restrict__ bad, int t,
                                      const double *__restrict__ dots, int64_t N, double logdet_p, double *out) {
    double s = 0.0;
    int any_bad = 0;
    for (int k = 1; k < t; ++k) {
        s += gamma[k];
        any_bad |= bad[k] != 0.0;
    }
    const double logdet = logdet_p + (t > 1 ? s / (t - 1) : 0.0);
    const double quad = dots[0];
    out[0] = -0.5 * (quad + logdet + (double)N * 1.8378770664093453);  // log(2 pi)
    out[1] = quad;
    out[2] = logdet;
    out[3] = any_bad ? 1.0 : 0.0;
}

__global__ void adjoint_rhs_kernel(const float *__restrict__ A, const float *__restrict__ RHS, int64_t N, int t,
                                   float *__restrict__ Bp) {
    const int64_t total = N * t;
    const float inv_m = t > 1 ? -1.0f / (float)(t - 1) : 0.0f;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / t;
        const int c = (int)(e - i * t);
        Bp[e] = c == 0 ? A[i * t] : inv_m * RHS[e];
    }
}

__global__ void grad_finalize_kernel(const double *__restrict__ bp, int n_blocks, int D, const double *__restrict__ dots,
                                     int t, float noise, double *grad_out) {
    const int p = threadIdx.x;
    if (p <= D) {
        double s = 0.0;
        for (int b = 0; b < n_blocks; ++b) s += bp[(int64_t)b * (D + 1) + p];
        grad_out[p] = 0.5 * s;
    } else if (p == D + 1) {
        double tr = 0.0;
        for (int c = 1; c < t; ++c) tr += dots[c];
        const double m = t > 1 ? (double)(t - 1) : 1.0;
        grad_out[p] = 0.5 * (double)noise * (dots[t] - tr / m);
    }
}

inline int grid_for(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 4096 ? 4096 : g));
}

}  // namespace

int cg_num_blocks(int64_t N, int t, int num_sms) {
    int64_t g = (N * t + 4095) / 4096;
    if (g > 2 * num_sms) g = 2 * num_sms;
    if (g < 1) g = 1;
    return (int)g;
}

int64_t cg_partial_doubles(int G, int t) { return (int64_t)std::max(3 * G, kStepBlocks) * t; }

void launch_cg_init(const float *B, int64_t ldb, int64_t N, int64_t Np, int t, const CgBuffers &b, double tol,
                    int max_iter, int hist_len, cudaStream_t st, const float *X0, int64_t ldx0) {
    (void)Np;
    double *rr_partial = nullptr;
    if (X0) {
        // b.Kp holds K_y x0; the r^T r partials go to the third slot of the partial buffer
        rr_partial = b.partial + (int64_t)2 * b.G * t;
        cg_init_x0_kernel<<<b.G, vec_block(t), 0, st>>>(B, ldb, X0, ldx0, b.Kp, N, t, b.x, b.r, b.p, b.partial,
                                                        rr_partial);
    } else {
        cg_init_kernel<<<b.G, vec_block(t), 0, st>>>(B, ldb, N, t, b.x, b.r, b.p, b.partial);
    }
    double *rz_partial = nullptr;
    if (b.pc.k > 0) {
        // z0 = P^{-1} b, p0 = z0, and the r^T z partials in the second half of the partial buffer
        rz_partial = b.partial + (int64_t)b.G * t;
        launch_precond_apply(b.pc, b.r, t, b.z, t, b.p, N, t, rz_partial, b.G, nullptr, st);
    }
    cg_init_scalars_kernel<<<1, 32 * (t < 32 ? t : 32), 0, st>>>(b.state, b.partial, b.G, t, tol, max_iter, hist_len,
                                                                 rz_partial, rr_partial);
}

namespace {

int step_blocks(int64_t N, int t) {
    // never more than cg_num_blocks, for which the partial sums are sized
    return std::min(kStepBlocks, cg_num_blocks(N, t, kStepBlocks));
}

template <int VEC>
cudaError_t launch_step(int64_t N, int t, const CgBuffers &b, const ProductTail &tail, const CgSplit *split, cudaStream_t st) {
    const int bd = VEC == 4 ? kStepThreads : (kStepThreads / t) * t;
    const int G = step_blocks(N, t);
    unsigned int *vbound = split ? split->vmax : nullptr;
    cudaError_t e;
    if (tail.part && tail.S >= 16 && VEC == 4) {
        const int64_t per = kStepThreads / 8 * VEC;  // elements of a block's round
        const int G8 = (int)std::min<int64_t>(kStepBlocks, (N * t + per - 1) / per);
        e = launch_chained(cg_pkp_alpha_kernel<VEC, VEC == 4 ? 8 : 1>, G8, bd, 0, st, b.p, b.Kp, tail.part, tail.S,
                           tail.stride, tail.scale, tail.noise, N, t, b.state, b.partial, b.hist_alpha);
    } else if (tail.part) {
        e = launch_chained(cg_pkp_alpha_kernel<VEC, 1>, G, bd, 0, st, b.p, b.Kp, tail.part, tail.S, tail.stride, tail.scale, tail.noise, N,
                           t, b.state, b.partial, b.hist_alpha);
    } else {
        e = launch_chained(cg_pkp_alpha_kernel<VEC, 0>, G, bd, 0, st, b.p, b.Kp, nullptr, 0, 0, 1.0f, 0.0f, N, t, b.state, b.partial,
                           b.hist_alpha);
    }
    if (e != cudaSuccess) return e;
    if (b.pc.k > 0) {
        double *rz_partial = b.partial + (int64_t)b.G * t;
        if ((e = launch_chained(cg_xr_beta_kernel<VEC, false>, G, bd, 0, st, b.x, b.r, b.p, b.Kp, N, t, b.state, b.partial,
                                b.hist_beta, nullptr)) != cudaSuccess ||
            (e = launch_precond_apply(b.pc, b.r, t, b.z, t, nullptr, N, t, rz_partial, b.G, b.state, st)) != cudaSuccess)
            return e;
        e = launch_chained(cg_beta_kernel, 1, 1024, 0, st, b.state, b.partial, G, rz_partial, b.G, t, b.hist_beta);
    } else {
        e = launch_chained(cg_xr_beta_kernel<VEC, true>, G, bd, 0, st, b.x, b.r, b.p, b.Kp, N, t, b.state, b.partial,
                           b.hist_beta, vbound);
    }
    if (e != cudaSuccess) return e;
    return split ? launch_p_split(*split, b.p, b.r, N, t, b.state, st)
                 : launch_chained(cg_p_kernel<VEC>, G, bd, 0, st, b.p, b.pc.k > 0 ? b.z : b.r, N, t, b.state);
}

}  // namespace

cudaError_t launch_cg_after_matvec(int64_t N, int t, const CgBuffers &b, const ProductTail &tail, const CgSplit *split,
                                   cudaStream_t st) {
    const int ctas = cg_step_ctas(N, t, b, tail.part ? tail.S : 0);
    if (ctas > 0) return launch_cg_cluster(ctas, N, t, b, tail, split, st);
    return t <= 64 && (t & (t - 1)) == 0 ? launch_step<4>(N, t, b, tail, split, st) : launch_step<1>(N, t, b, tail, split, st);
}

cudaError_t launch_cg_loop_condition(cudaGraphConditionalHandle h, CgState *state, cudaStream_t st) {
    cg_loop_condition_kernel<<<1, 1, 0, st>>>(h, state);
    return cudaPeekAtLastError();
}

cudaError_t launch_cg_chunk_tally(CgState *state, cudaStream_t st) {
    cg_chunk_tally_kernel<<<1, 1, 0, st>>>(state);
    return cudaPeekAtLastError();
}

void launch_cg_gather_column(const CgBuffers &b1, int hist_len, CgState *dst, double *dst_alpha, double *dst_beta,
                             int t, int c, cudaStream_t st) {
    cg_gather_column_kernel<<<1, 64, 0, st>>>(b1.state, b1.hist_alpha, b1.hist_beta, hist_len, dst, dst_alpha,
                                              dst_beta, t, c);
}

void launch_cg_copy_out(const CgBuffers &b, int64_t N, int t, float *Xsol, int64_t ldx, cudaStream_t st) {
    copy_out_kernel<<<grid_for(N * t), 256, 0, st>>>(b.x, N, t, Xsol, ldx);
}

void launch_col_dots(const float *A, const float *B, int64_t N, int t, double *partial, int G, double *out,
                     cudaStream_t st) {
    col_dots_kernel<<<G, vec_block(t), 0, st>>>(A, B, N, t, partial);
    col_dots_final_kernel<<<1, 2 * kMaxT, 0, st>>>(partial, G, t, out);
}

void launch_slq_lml(const CgBuffers &b, int t, int hist_len, const double *dots, int64_t N, double *out,
                    cudaStream_t st) {
    // per-column gamma and bad flags in the CG partial-sum buffer (3 G t >= 2 t doubles, free after
    // the column dots have been reduced)
    double *gamma = b.partial;
    double *bad = b.partial + t;
    if (t > 1)
        slq_quad_kernel<<<t - 1, kSlqThreads, 0, st>>>(b.state, b.hist_alpha, b.hist_beta, t, hist_len, gamma, bad);
    slq_lml_finish_kernel<<<1, 1, 0, st>>>(gamma, bad, t, dots, N, b.pc.k > 0 ? b.pc.logdet : 0.0, out);
}

void launch_adjoint_rhs(const float *A, const float *RHS, int64_t N, int t, float *Bp, cudaStream_t st) {
    adjoint_rhs_kernel<<<grid_for(N * t), 256, 0, st>>>(A, RHS, N, t, Bp);
}

void launch_grad_finalize(const double *block_partials, int n_blocks, int D, const double *dots, int t, float noise,
                          double *grad_out, cudaStream_t st) {
    grad_finalize_kernel<<<1, 32, 0, st>>>(block_partials, n_blocks, D, dots, t, noise, grad_out);
}

}  // namespace lgp
