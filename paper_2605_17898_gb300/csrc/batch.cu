// Many independent GP solves of uneven size advanced together.
//
// Per CG iteration, one persistent launch computes K_y(g) p(g) for every problem g:
// its CTAs pull work items (problem, block of 256 rows, column split) from a list sorted by cost
// (longest first) through an atomic counter, so large and small problems share the
// GPU without one launch per problem. Problems whose columns have all converged are
// skipped. One more launch is the rest of the iteration: a thread-block cluster (or one CTA) per problem
// adds the product's partial sums and runs the problem's whole CG step, its column sums exchanged
// through distributed shared memory in a fixed order, so the results do not depend on which CTA took which item.
#include <cooperative_groups.h>

#include "batch.cuh"
#include "cg_reduce.cuh"
#include "mv_simt.cuh"

namespace lgp {

namespace {

constexpr int kBatchBM = 256;  // rows of a work item
template <int TT> using BatchTile = RowTile<TT, 2, 128>;

// One 256-row block of one problem: K_y p for those rows over all of the problem's columns (or one split of them). The
// distance runs over the problem's own D coordinates (the rows are stored padded to DP).
template <int KIND, int D, int TT>
__device__ void batch_item(const BatchGp &g, int64_t row0, int split, const BatchArgs &a, float *xs, float *vs, float *tot) {
    using S = BatchTile<TT>;
    static_assert(S::kRows == kBatchBM, "an item is one block of rows");
    const int t = a.t;
    const float *Xs = a.Xs + g.xs_off;
    const float *V = a.p + g.vec_off * t;
    float *out = a.kp + g.vec_off * t;
    const int64_t jb = (int64_t)split * g.cols_per_split;
    const int64_t je = min(g.N, jb + g.cols_per_split);
    float sum[S::R][TT];
    simt_rows<KIND, D, S>(Xs, row0, g.Np, Xs, g.Np, V, t, 0, t, jb, je, g.scale.log2s2, g.scale.v, xs, vs, tot, sum);
#pragma unroll
    for (int r = 0; r < S::R; ++r) {
        const int64_t i = row0 + r * S::kThreads + threadIdx.x;
        if (i >= g.N) continue;
        if (g.splits > 1) {
            float *dst = a.part + g.part_off + ((int64_t)split * g.Np + i) * t;
#pragma unroll
            for (int c = 0; c < TT; ++c)
                if (c < t) dst[c] = sum[r][c];
        } else {
#pragma unroll
            for (int c = 0; c < TT; ++c)
                if (c < t) out[i * t + c] = fmaf(g.noise, V[i * t + c], rbf_scaled<KIND>(sum[r][c], g.scale.out));
        }
    }
}

template <int KIND, int TT>
__device__ __forceinline__ void batch_item_d(const BatchGp &g, int64_t row0, int split, const BatchArgs &a, float *xs,
                                             float *vs, float *tot) {
    switch (g.D) {
        case 1: batch_item<KIND, 1, TT>(g, row0, split, a, xs, vs, tot); break;
        case 2: batch_item<KIND, 2, TT>(g, row0, split, a, xs, vs, tot); break;
        case 3: batch_item<KIND, 3, TT>(g, row0, split, a, xs, vs, tot); break;
        case 4: batch_item<KIND, 4, TT>(g, row0, split, a, xs, vs, tot); break;
        case 5: batch_item<KIND, 5, TT>(g, row0, split, a, xs, vs, tot); break;
        case 6: batch_item<KIND, 6, TT>(g, row0, split, a, xs, vs, tot); break;
        case 7: batch_item<KIND, 7, TT>(g, row0, split, a, xs, vs, tot); break;
        default: batch_item<KIND, 8, TT>(g, row0, split, a, xs, vs, tot);
    }
}

template <int TT>
__global__ void __launch_bounds__(BatchTile<TT>::kThreads) batch_mv_kernel(BatchArgs a) {
    __shared__ __align__(16) float xs[kSimtBN * 8];
    __shared__ __align__(16) float vs[kSimtBN * TT];
    __shared__ float tot[BatchTile<TT>::kTotFloats];
    __shared__ int item_s;
    chain_wait();
    chain_next();
    if (*a.done || *a.n_done >= a.n_gp) return;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) item_s = atomicAdd(a.item_counter, 1);
        __syncthreads();
        const int item = item_s;
        if (item >= a.n_items) break;
        const BatchItem it = a.items[item];
        if (a.gp_done[it.gp]) continue;
        const BatchGp g = a.gps[it.gp];
        const int64_t row0 = (int64_t)it.row_block * kBatchBM;
        switch (g.kind) {
            case LGP_RBF: batch_item_d<LGP_RBF, TT>(g, row0, it.split, a, xs, vs, tot); break;
            case LGP_MATERN52: batch_item_d<LGP_MATERN52, TT>(g, row0, it.split, a, xs, vs, tot); break;
            case LGP_MATERN12: batch_item_d<LGP_MATERN12, TT>(g, row0, it.split, a, xs, vs, tot); break;
            default: batch_item_d<LGP_MATERN32, TT>(g, row0, it.split, a, xs, vs, tot);
        }
    }
}

// ---------------------------------------------------------------- segmented CG kernels

constexpr int kVec = 256;
constexpr int kMaxBatchT = 16;

__device__ void seg_col_reduce(double v, int t, double *red, double *out_row) {
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

__global__ void binit_kernel(BatchArgs a) {
    __shared__ double red[kVec];
    const BatchVecBlock vb = a.vblocks[blockIdx.x];
    const BatchGp g = a.gps[vb.gp];
    const int t = a.t;
    const int c = threadIdx.x % t;
    double s = 0.0;
    for (int64_t i = vb.r0 + threadIdx.x / t; i < vb.r1; i += blockDim.x / t) {
        const float b = g.B[i * t + c];
        const int64_t e = (g.vec_off + i) * t + c;
        a.x[e] = 0.0f;
        a.r[e] = b;
        a.p[e] = b;
        s += (double)b * (double)b;
    }
    seg_col_reduce(s, t, red, a.partial + (int64_t)blockIdx.x * t);
}

__global__ void bscal_init_kernel(BatchArgs a, double tol, int max_iter) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0) {
        a.st->max_iter = max_iter;
        a.st->tol = tol;
        a.st->status = 0;
        a.st->loop_chunks = 0;
        a.st->max_chunks = max_iter / 8 + 2;
    }
    if (k >= a.n_gp * a.t) return;
    const int gi = k / a.t, c = k % a.t;
    const BatchGp g = a.gps[gi];
    double s = 0.0;
    for (int b = g.blk0; b < g.blk1; ++b) s += a.partial[(int64_t)b * a.t + c];
    a.bnorm2[k] = s;
    a.rr[k] = s;
    a.iters[k] = 0;
    const bool bad = !isfinite(s);
    a.active[k] = (s > 0.0) && !bad;
    if (bad) atomicOr(&a.st->status, 1);
}

// Problems without an active column are done from the start; a non-finite right-hand side ends the whole call.
__global__ void bdone_kernel(BatchArgs a) {
    __shared__ int n_s;
    if (threadIdx.x == 0) n_s = 0;
    __syncthreads();
    int n = 0;
    for (int gi = threadIdx.x; gi < a.n_gp; gi += blockDim.x) {
        int act = 0;
        for (int c = 0; c < a.t; ++c) act |= a.active[gi * a.t + c];
        a.gp_done[gi] = !act;
        n += !act;
    }
    atomicAdd(&n_s, n);
    __syncthreads();
    if (threadIdx.x == 0) {
        *a.n_done = n_s;
        *a.item_counter = 0;
        *a.done = a.st->status ? 1 : 0;
    }
}

// ---------------------------------------------------------------- the CG step

// One problem's CG step after the product: Kp = scale sum_k part[k] + noise p (or as the product left it), alpha, x, r, beta,
// p and the problem's state, by one cluster of CL CTAs whose three passes over the problem's vectors meet at the
// cluster barrier. As segmented kernels the step took seven launches an iteration (with the product's memset nine),
// each a few microseconds for vectors that fit L2 many times over: 48 problems of 200..2000 rows, t = 8, 11.2 -> 6.8 ms a call.

// Block of VEC = 4 (t a power of two): kVec threads; VEC = 1: a multiple of t. (A problem's vectors hold Np t >= N t
// values from a multiple of 16 bytes, so a last float4 that crosses N t stays inside them.)
template <int VEC, int CL>
__global__ void __launch_bounds__(kVec) batch_step_kernel(BatchArgs a) {
    __shared__ ColSums acc1, acc2;
    __shared__ double sum1[kMaxBatchT], sum2[kMaxBatchT];
    __shared__ float s_alpha[kMaxBatchT], s_beta[kMaxBatchT];
    __shared__ int s_act[kMaxBatchT];
    chain_wait();
    chain_next();
    const int gi = blockIdx.x / CL, rank = blockIdx.x % CL;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.item_counter = 0;
    if (*a.done || a.gp_done[gi]) return;  // the same for the whole cluster: its rank 0 sets gp_done after the last barrier
    clear_sums(acc1);
    clear_sums(acc2);
    __syncthreads();
    const BatchGp g = a.gps[gi];
    const int tid = threadIdx.x, t = a.t, k = gi * t + (tid < t ? tid : 0);
    const int active = a.active[k], iters = a.iters[k];
    const double rr0 = a.rr[k];
    const int64_t total = g.N * t, base = g.vec_off * t;
    float *x = a.x + base, *r = a.r + base, *p = a.p + base, *kp = a.kp + base;
    const float *part = a.part + g.part_off;
    const int64_t stride = g.Np * t;
    const int64_t e0 = ((int64_t)rank * blockDim.x + tid) * VEC, step = (int64_t)CL * blockDim.x * VEC;

    float hi[VEC], lo[VEC];
    auto clear = [&]() {
#pragma unroll
        for (int q = 0; q < VEC; ++q) hi[q] = lo[q] = 0.0f;
    };
    clear();
    for (int64_t e = e0; e < total; e += step) {
        float pv[VEC], kv[VEC];
        load_vec<VEC>(p + e, pv);
        if (g.splits > 1) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) kv[q] = 0.0f;
#pragma unroll 8
            for (int s = 0; s < g.splits; ++s) {
                float w[VEC];
                load_vec<VEC>(part + s * stride + e, w);
#pragma unroll
                for (int q = 0; q < VEC; ++q) kv[q] += w[q];
            }
#pragma unroll
            for (int q = 0; q < VEC; ++q) kv[q] = fmaf(g.noise, pv[q], g.scale.out * kv[q]);
            store_vec<VEC>(kp + e, kv);
        } else {
            load_vec<VEC>(kp + e, kv);
        }
#pragma unroll
        for (int q = 0; q < VEC; ++q)
            if (VEC == 1 || e + q < total) acc_prod2(hi[q], lo[q], pv[q], kv[q]);
    }
    block_col_sums<VEC>(hi, lo, t, acc1, sum1);
    const double pkp = cluster_sum<CL>(sum1, t);
    int failed = 0;
    if (tid < t) {
        double alpha = 0.0;
        if (active) {
            if (!isfinite(pkp)) failed = 1;
            else if (!(pkp > 0.0)) failed = 2;
            else alpha = rr0 / pkp;
        }
        s_alpha[tid] = (float)alpha;
    }
    __syncthreads();

    float al[VEC];
    clear();
#pragma unroll
    for (int q = 0; q < VEC; ++q) al[q] = s_alpha[col_of<VEC>(tid, q, t)];
    for (int64_t e = e0; e < total; e += step) {
        float xv[VEC], rv[VEC], pv[VEC], kv[VEC];
        load_vec<VEC>(x + e, xv);
        load_vec<VEC>(r + e, rv);
        load_vec<VEC>(p + e, pv);
        load_vec<VEC>(kp + e, kv);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            if (al[q] != 0.0f) {
                xv[q] = fmaf(al[q], pv[q], xv[q]);
                rv[q] = fmaf(-al[q], kv[q], rv[q]);
            }
            if (VEC == 1 || e + q < total) acc_prod2(hi[q], lo[q], rv[q], rv[q]);
        }
        store_vec<VEC>(x + e, xv);
        store_vec<VEC>(r + e, rv);
    }
    block_col_sums<VEC>(hi, lo, t, acc2, sum2);
    const double rr = cluster_sum<CL>(sum2, t);
    int act = 0;
    if (tid < t) {
        double beta = 0.0;
        if (active && !failed) {
            beta = rr / rr0;
            const double root = a.st->tol * sqrt(a.bnorm2[k]);
            act = rr > root * root;
        }
        s_beta[tid] = (float)beta;
        s_act[tid] = act;
    }
    __syncthreads();

    float be[VEC];
    int ac[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) {
        be[q] = s_beta[col_of<VEC>(tid, q, t)];
        ac[q] = s_act[col_of<VEC>(tid, q, t)];
    }
    for (int64_t e = e0; e < total; e += step) {
        float pv[VEC], rv[VEC];
        load_vec<VEC>(p + e, pv);
        load_vec<VEC>(r + e, rv);
#pragma unroll
        for (int q = 0; q < VEC; ++q)
            if (ac[q]) pv[q] = fmaf(be[q], pv[q], rv[q]);
        store_vec<VEC>(p + e, pv);
    }
    // the state, by rank 0 once every CTA has read the old one and nobody reads this CTA's sums any more
    if constexpr (CL == 1) __syncthreads();
    else cooperative_groups::this_cluster().sync();
    if (rank == 0) {
        int stop = 0;
        if (tid < t && active) {
            if (failed) {
                atomicOr(&a.st->status, failed);
            } else {
                a.rr[k] = rr;
                a.iters[k] = iters + 1;
            }
            a.active[k] = act;
            stop = iters + 1 >= a.st->max_iter;
        }
        stop = __syncthreads_or(stop);
        const int any = __syncthreads_or(act);
        if (tid == 0 && (stop || !any)) {
            a.gp_done[gi] = 1;
            atomicAdd(a.n_done, 1);
        }
    }
}

__global__ void bcopy_out_kernel(BatchArgs a) {
    const BatchVecBlock vb = a.vblocks[blockIdx.x];
    const BatchGp g = a.gps[vb.gp];
    const int t = a.t;
    const int c = threadIdx.x % t;
    for (int64_t i = vb.r0 + threadIdx.x / t; i < vb.r1; i += blockDim.x / t)
        g.Xsol[i * t + c] = a.x[(g.vec_off + i) * t + c];
}

__global__ void batch_loop_condition_kernel(cudaGraphConditionalHandle h, BatchArgs a) {
    a.st->loop_chunks += 1;
    const bool more = !*a.done && *a.n_done < a.n_gp && a.st->loop_chunks < a.st->max_chunks;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

inline int vec_threads(int t) { return (kVec / t) * t; }

}  // namespace

int batch_item_rows() { return kBatchBM; }

cudaError_t launch_batch_init(const BatchArgs &a, double tol, int max_iter, cudaStream_t st) {
    binit_kernel<<<a.n_vblocks, vec_threads(a.t), 0, st>>>(a);
    const int n = a.n_gp * a.t;
    bscal_init_kernel<<<(n + 255) / 256, 256, 0, st>>>(a, tol, max_iter);
    bdone_kernel<<<1, 256, 0, st>>>(a);
    return cudaGetLastError();
}

namespace {

template <int VEC, int CL> cudaError_t launch_step(const BatchArgs &a, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.n_gp * CL), 1, 1);
    cfg.blockDim = dim3(VEC == 4 ? kVec : vec_threads(a.t), 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CL;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, batch_step_kernel<VEC, CL>, a);
}

}  // namespace

cudaError_t launch_batch_iteration(const BatchArgs &a, int num_sms, cudaStream_t st) {
    const int grid = std::max(1, std::min(a.n_items, num_sms * 6));
    cudaError_t e;
    switch (a.tt) {
        case 1: e = launch_chained(batch_mv_kernel<1>, grid, BatchTile<1>::kThreads, 0, st, a); break;
        case 2: e = launch_chained(batch_mv_kernel<2>, grid, BatchTile<2>::kThreads, 0, st, a); break;
        case 4: e = launch_chained(batch_mv_kernel<4>, grid, BatchTile<4>::kThreads, 0, st, a); break;
        case 8: e = launch_chained(batch_mv_kernel<8>, grid, BatchTile<8>::kThreads, 0, st, a); break;
        case 16: e = launch_chained(batch_mv_kernel<16>, grid, BatchTile<16>::kThreads, 0, st, a); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    // One CTA per problem where its vectors are at most two loads per thread, or up to four when there is a problem for
    // every SM anyway; else a cluster of 8. Solve of 64 problems with N = 200, t = 8: one CTA 2237 us, cluster 2418;
    // 200 with N = 500, t = 8: 7239 and 8621; one with N = 1000, t = 8: 3277 and 2467.
    const bool pow2 = (a.t & (a.t - 1)) == 0;
    if (a.max_elems <= 8 * kVec || (a.max_elems <= 16 * kVec && a.n_gp >= num_sms))
        return pow2 ? launch_step<4, 1>(a, st) : launch_step<1, 1>(a, st);
    return pow2 ? launch_step<4, 8>(a, st) : launch_step<1, 8>(a, st);
}

cudaError_t launch_batch_loop_condition(cudaGraphConditionalHandle h, const BatchArgs &a, cudaStream_t st) {
    batch_loop_condition_kernel<<<1, 1, 0, st>>>(h, a);
    return cudaGetLastError();
}

cudaError_t launch_batch_copy_out(const BatchArgs &a, cudaStream_t st) {
    bcopy_out_kernel<<<a.n_vblocks, vec_threads(a.t), 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace lgp
