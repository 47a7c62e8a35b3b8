// One CG step after the product as a single launch, for vectors of at most 262144 elements (plain CG, t a power of two):
// the step's three grid-wide stages (p^T Kp, r^T r, the update of p) are stages of one thread-block cluster, which
// exchanges its column sums through distributed shared memory and meets at the hardware's cluster barrier.
//
// What bounds it: latency. The three launches of solver.cu cost about 2 us each beyond their work, and between them
// every vector goes to L2 and back; here up to 65536 elements of x, r, p and Kp are read once into the registers of 8
// CTAs (the portable cluster size; one CTA, without a barrier, where a single SM can take the product's partial sums in
// about a microsecond). Up to 262144 elements 16 CTAs keep p and r and read x and Kp once more.
//
// The product's partial sums (S per element) are read by the cluster's SMs alone, so they bound each size (cg_step_rule): 8
// CTAs take 2^20 of them, 16 CTAs 2^22, beyond that the three launches' 76 blocks are faster. Time of an iteration with its
// product (us), 8 CTAs / 16 CTAs / three launches: N = 8000, t = 2, 1.0M 47.9 / 49.8 / 54.8; N = 4500, t = 4, 1.3M 52.0 / 47.9 /
// 52.8; N = 4000, t = 8, 2.0M 39.8 / 36.2 / 41.9; N = 12000, t = 2, 2.3M 93.1 / 84.9 / 90.7; N = 16000, t = 4, 4.0M 165.8 / 155.7 /
// 158.0; N = 8000, t = 8, 8M 108 / - / 82.8; N = 9000, t = 8, 5.1M - / 98.8 / 93.6.
//
// Measured against the three launches: solve of N = 1024, t = 1, ~90 iterations 1.62 -> 0.95 ms; training step of N = 2000,
// D = 8, t = 16 4.65 -> 3.73 ms; with 16 CTAs, solves at t = 32 of N = 3000 4.54 -> 4.18 ms, N = 8000 8.02 -> 7.53; at
// N = 4099, t = 16 6.66 -> 5.89. Larger vectors keep the three launches, whose blocks spread over more SMs.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "cg_reduce.cuh"
#include "split.cuh"

namespace lgp {

namespace {

namespace cg = cooperative_groups;

constexpr int kClThreads = 512;
constexpr int kClVecs = 4;  // float4s per thread and vector that are all held in registers
constexpr int kClWide = 16, kClWideVecs = 8;  // larger vectors
// partial sums that a cluster of 1, 8 and 16 CTAs takes (about 1.3, 4 and 8 us of its SMs' loads)
constexpr int64_t kClusterOneParts = 1 << 15, kClParts = 1 << 20, kClWideParts = 1 << 22;

struct ClusterArgs {
    float *x, *r, *p, *Kp;
    const float *part;  // the product's partial sums (nullptr: Kp is complete)
    int S;
    int64_t part_stride;
    float scale, noise;
    int total, t;  // N t
    CgState *st;
    double *hist_alpha, *hist_beta;
    int split;  // p is split for the next product
    CgSplit sp;
    int64_t N;
};

template <int CL, int T, int FMT>
__device__ void split_tile(const ClusterArgs &a, const float *tile, int row0, int rows, const int *s_exp, const int *s_act) {
    // rows row0 .. row0 + rows - 1 (a multiple of 8) x T columns of p in shared memory: one (8-row group, column) each
    for (int e = threadIdx.x; e < rows / 8 * T; e += kClThreads) {
        const int g = e / T, c = e - g * T;
        if (!s_act[c]) continue;
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = row0 + 8 * g + k < a.N ? tile[(8 * g + k) * T + c] : 0.0f;
        store_split<T, FMT>(a.sp.vs, row0 / 8 + g, c, v, s_exp[c]);
    }
}

// VECS float4s per thread and vector; above kClVecs only p and r stay in registers, Kp and x come from the L2 cache again.
template <int CL, int VECS>
__global__ void __launch_bounds__(kClThreads, 1) cg_cluster_kernel(const ClusterArgs a) {
    __shared__ ColSums acc1, acc2;
    __shared__ double sum1[kMaxT], sum2[kMaxT];
    __shared__ unsigned int rmax[kMaxT], pmax[kMaxT];
    __shared__ float s_alpha[kMaxT], s_beta[kMaxT];
    __shared__ int s_exp[kMaxT], s_act[kMaxT];
    __shared__ __align__(16) float tile[4 * kClThreads];
    CgState *st = a.st;
    chain_wait();
    chain_next();
    if (st->done) return;
    const int tid = threadIdx.x, t = a.t;
    const int rank = CL == 1 ? 0 : (int)cg::this_cluster().block_rank();
    const int c = tid < t ? tid : 0;
    // per-column state, read before the last barrier (rank 0 rewrites it after that)
    const int active = st->active[c];
    const double rz0 = st->rz[c], thresh = st->thresh[c];
    const float pmax0 = __uint_as_float(st->pmax[c]);
    const int iter = st->iter, hist_len = st->hist_len, max_iter = st->max_iter;
    const float vbound0 = a.split && a.sp.fmt == 1 ? __uint_as_float(a.sp.vmax[c]) : 0.0f;
    if (tid < kMaxT) rmax[tid] = pmax[tid] = 0u;
    clear_sums(acc1);
    clear_sums(acc2);
    __syncthreads();

    // ---- p, Kp (with the product's partial sums), r, x into registers; p^T Kp
    constexpr bool kHold = VECS <= kClVecs;
    constexpr int kHeld = kHold ? VECS : 1;
    float4 pv[VECS], rv[VECS], kv[kHeld], xv[kHeld];
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
    auto index = [&](int m) { return ((m * CL + rank) * kClThreads + tid) * 4; };
    auto load = [](const float *q) { return *reinterpret_cast<const float4 *>(q); };
    // elements past N t (the last float4 of t = 1, 2) stay out of the sums
    auto add = [&](int m, const float4 &u, const float4 &v) {
        const int e = index(m);
        if (e < a.total) acc_prod2(hi[0], lo[0], u.x, v.x);
        if (e + 1 < a.total) acc_prod2(hi[1], lo[1], u.y, v.y);
        if (e + 2 < a.total) acc_prod2(hi[2], lo[2], u.z, v.z);
        if (e + 3 < a.total) acc_prod2(hi[3], lo[3], u.w, v.w);
    };
    auto sum_parts = [&](int e, const float4 &p4) {
        float4 k4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int q = 0; q < a.S; ++q) {
            const float4 w = load(a.part + q * a.part_stride + e);
            k4.x += w.x;
            k4.y += w.y;
            k4.z += w.z;
            k4.w += w.w;
        }
        k4.x = fmaf(a.noise, p4.x, a.scale * k4.x);
        k4.y = fmaf(a.noise, p4.y, a.scale * k4.y);
        k4.z = fmaf(a.noise, p4.z, a.scale * k4.z);
        k4.w = fmaf(a.noise, p4.w, a.scale * k4.w);
        return k4;
    };
#pragma unroll
    for (int m = 0; m < VECS; ++m) {
        const int e = index(m);
        pv[m] = rv[m] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (kHold) kv[m] = xv[m] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < a.total) {
            pv[m] = load(a.p + e);
            rv[m] = load(a.r + e);
            if constexpr (kHold) {
                xv[m] = load(a.x + e);
                if (!a.part) kv[m] = load(a.Kp + e);
            }
        }
    }
    if constexpr (kHold) {
        if (a.part) {
#pragma unroll
            for (int m = 0; m < VECS; ++m)
                if (index(m) < a.total) kv[m] = sum_parts(index(m), pv[m]);
        }
#pragma unroll
        for (int m = 0; m < VECS; ++m) add(m, pv[m], kv[m]);
    } else {
#pragma unroll
        for (int m = 0; m < VECS; ++m) {
            const int e = index(m);
            if (e >= a.total) continue;
            float4 k4;
            if (a.part) {
                k4 = sum_parts(e, pv[m]);
                *reinterpret_cast<float4 *>(a.Kp + e) = k4;
            } else {
                k4 = load(a.Kp + e);
            }
            add(m, pv[m], k4);
        }
    }
    block_col_sums<4>(hi, lo, t, acc1, sum1);
    const double pkp = cluster_sum<CL>(sum1, t);
    int bad = 0, nonfinite = 0;
    double alpha = 0.0;
    if (tid < t) {
        if (active) {
            if (!isfinite(pkp)) nonfinite = 1;
            else if (!(pkp > 0.0)) bad = 1;
            else alpha = rz0 / pkp;
        }
        s_alpha[tid] = (float)alpha;
    }
    __syncthreads();

    // ---- x, r; r^T r and max |r|
    float al[4], m4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        al[k] = s_alpha[col_of<4>(tid, k, t)];
        hi[k] = lo[k] = 0.0f;
    }
    auto axpy = [](float s, float u, float v) { return s != 0.0f ? fmaf(s, u, v) : v; };
#pragma unroll
    for (int m = 0; m < VECS; ++m) {
        const int e = index(m);
        if (e >= a.total) continue;
        float4 x4, k4;
        if constexpr (kHold) {
            x4 = xv[m];
            k4 = kv[m];
        } else {
            x4 = load(a.x + e);
            k4 = load(a.Kp + e);
        }
        x4 = make_float4(axpy(al[0], pv[m].x, x4.x), axpy(al[1], pv[m].y, x4.y), axpy(al[2], pv[m].z, x4.z),
                         axpy(al[3], pv[m].w, x4.w));
        rv[m] = make_float4(axpy(-al[0], k4.x, rv[m].x), axpy(-al[1], k4.y, rv[m].y), axpy(-al[2], k4.z, rv[m].z),
                            axpy(-al[3], k4.w, rv[m].w));
        *reinterpret_cast<float4 *>(a.x + e) = x4;
        *reinterpret_cast<float4 *>(a.r + e) = rv[m];
        add(m, rv[m], rv[m]);
        m4[0] = fmaxf(m4[0], fabsf(rv[m].x));
        if (e + 1 < a.total) m4[1] = fmaxf(m4[1], fabsf(rv[m].y));
        if (e + 2 < a.total) m4[2] = fmaxf(m4[2], fabsf(rv[m].z));
        if (e + 3 < a.total) m4[3] = fmaxf(m4[3], fabsf(rv[m].w));
    }
    if (a.split) {
#pragma unroll
        for (int k = 0; k < 4; ++k) atomicMax(&rmax[col_of<4>(tid, k, t)], __float_as_uint(m4[k]));
    }
    block_col_sums<4>(hi, lo, t, acc2, sum2);
    const double rr = cluster_sum<CL>(sum2, t);
    double beta = 0.0;
    int act = 0;
    float bound = vbound0;
    if (tid < t) {
        act = active && !bad && !nonfinite;
        if (act) {
            beta = rr / rz0;
            if (!(rr > thresh)) act = 0;
        }
        if (a.split && act) {
            unsigned int mx = 0u;
            if constexpr (CL == 1) {
                mx = rmax[tid];
            } else {
                for (int q = 0; q < CL; ++q) mx = max(mx, cg::this_cluster().map_shared_rank(rmax, q)[tid]);
            }
            bound = fmaf(fabsf((float)beta), pmax0, __uint_as_float(mx)) * 1.000001f;
        }
        s_beta[tid] = (float)beta;
        s_act[tid] = act;
        s_exp[tid] = col_exponent(__float_as_uint(bound));
    }
    __syncthreads();

    // ---- p, and its halves for the next product
    float be[4];
    int ac[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int cc = col_of<4>(tid, k, t);
        be[k] = s_beta[cc];
        ac[k] = s_act[cc];
        m4[k] = 0.0f;
    }
#pragma unroll
    for (int m = 0; m < VECS; ++m) {
        const int e = index(m);
        if (e < a.total) {
            if (ac[0]) pv[m].x = fmaf(be[0], pv[m].x, rv[m].x);
            if (ac[1]) pv[m].y = fmaf(be[1], pv[m].y, rv[m].y);
            if (ac[2]) pv[m].z = fmaf(be[2], pv[m].z, rv[m].z);
            if (ac[3]) pv[m].w = fmaf(be[3], pv[m].w, rv[m].w);
            *reinterpret_cast<float4 *>(a.p + e) = pv[m];
        }
        if (a.split) {
            if (e < a.total) {
                m4[0] = fmaxf(m4[0], fabsf(pv[m].x));
                m4[1] = fmaxf(m4[1], fabsf(pv[m].y));
                m4[2] = fmaxf(m4[2], fabsf(pv[m].z));
                m4[3] = fmaxf(m4[3], fabsf(pv[m].w));
                if (a.sp.out_init)
                    *reinterpret_cast<float4 *>(a.sp.out_init + e) = make_float4(a.sp.noise * pv[m].x, a.sp.noise * pv[m].y,
                                                                               a.sp.noise * pv[m].z, a.sp.noise * pv[m].w);
            }
            const int e0 = (m * CL + rank) * kClThreads * 4;  // the CTA's rows of this round are contiguous
            if (e0 < a.total) {
                *reinterpret_cast<float4 *>(tile + 4 * tid) = pv[m];
                __syncthreads();
                const int rows = 4 * kClThreads / t;
                if (t == 16) {
                    if (a.sp.fmt == 1) split_tile<CL, 16, 1>(a, tile, e0 / 16, rows, s_exp, s_act);
                    else split_tile<CL, 16, 0>(a, tile, e0 / 16, rows, s_exp, s_act);
                } else {
                    if (a.sp.fmt == 1) split_tile<CL, 32, 1>(a, tile, e0 / 32, rows, s_exp, s_act);
                    else split_tile<CL, 32, 0>(a, tile, e0 / 32, rows, s_exp, s_act);
                }
                __syncthreads();
            }
        }
    }
    if (a.split) {
#pragma unroll
        for (int k = 0; k < 4; ++k) atomicMax(&pmax[col_of<4>(tid, k, t)], __float_as_uint(m4[k]));
    }

    // ---- state, by rank 0 once every CTA has read the old one (and nobody reads this CTA's sums any more)
    if constexpr (CL == 1) __syncthreads();
    else cg::this_cluster().sync();
    if (rank == 0) {
        if (tid < t) {
            if (active) {
                st->alpha[tid] = alpha;
                st->beta[tid] = beta;
                if (!bad && !nonfinite) {
                    st->rr[tid] = rr;
                    st->rz[tid] = rr;
                    st->iters[tid] += 1;
                }
                st->active[tid] = act;
            } else {
                st->alpha[tid] = st->beta[tid] = 0.0;
            }
            if (a.split && act) {
                unsigned int mx = 0u;
                if constexpr (CL == 1) {
                    mx = pmax[tid];
                } else {
                    for (int q = 0; q < CL; ++q) mx = max(mx, cg::this_cluster().map_shared_rank(pmax, q)[tid]);
                }
                st->pmax[tid] = mx;
                if (a.sp.fmt == 1) {
                    a.sp.vmax[tid] = __float_as_uint(bound);
                    a.sp.col_scale[tid] = ldexpf(a.sp.s2, -15 - s_exp[tid]);
                }
            }
            if (iter < hist_len) {
                a.hist_alpha[(int64_t)iter * t + tid] = alpha;
                a.hist_beta[(int64_t)iter * t + tid] = beta;
            }
        }
        bad = __syncthreads_or(bad);
        nonfinite = __syncthreads_or(nonfinite);
        const int any = __syncthreads_or(act);
        if (tid == 0) {
            if ((bad || nonfinite) && st->status == 0)
                st->status = nonfinite ? (int)LGP_ERR_NONFINITE : (int)LGP_ERR_BREAKDOWN;
            st->iter = iter + 1;
            if (!any || iter + 1 >= max_iter) st->done = 1;
        }
    }
    if constexpr (CL > 1) cg::this_cluster().sync();  // rank 0 has read the others' maxima
}

template <int CL, int VECS>
cudaLaunchConfig_t cluster_config(cudaLaunchAttribute (&at)[2], cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL, 1, 1);
    cfg.blockDim = dim3(kClThreads, 1, 1);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CL;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 2 : 1;
    return cfg;
}

template <int CL, int VECS> cudaError_t launch_cluster(const ClusterArgs &a, cudaStream_t st) {
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t cfg = cluster_config<CL, VECS>(at, st);
    return cudaLaunchKernelEx(&cfg, cg_cluster_kernel<CL, VECS>, a);
}

// Whether the current device takes clusters of 16 CTAs of the step (above the portable size of 8); asked once per device.
bool wide_cluster_ok() {
    static std::atomic<signed char> known[64];  // 0 not asked, 1 yes, -1 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    signed char k = known[dev].load();
    if (k == 0) {
        auto kernel = cg_cluster_kernel<kClWide, kClWideVecs>;
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = cluster_config<kClWide, kClWideVecs>(at, nullptr);
        int n = 0;
        const bool fits = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                          cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0;
        if (!fits) (void)cudaGetLastError();
        known[dev].store(k = fits ? 1 : -1);
    }
    return k > 0;
}

constexpr int64_t floats_of(int cl, int vecs) { return (int64_t)cl * kClThreads * 4 * vecs; }

}  // namespace

int cg_step_rule(int64_t N, int t, int S, bool wide) {
    if (t > 64 || (t & (t - 1)) != 0) return 0;
    const int64_t elems = N * t, parts = elems * S;
    if (elems <= floats_of(1, kClVecs) && std::max(elems, parts) <= kClusterOneParts) return 1;
    if (elems <= floats_of(8, kClVecs) && parts <= kClParts) return 8;
    return wide && elems <= floats_of(kClWide, kClWideVecs) && parts <= kClWideParts ? kClWide : 0;
}

int cg_step_ctas(int64_t N, int t, const CgBuffers &b, int S) {
    return b.pc.k > 0 ? 0 : cg_step_rule(N, t, S, wide_cluster_ok());
}

cudaError_t launch_cg_cluster(int ctas, int64_t N, int t, const CgBuffers &b, const ProductTail &tail, const CgSplit *split,
                              cudaStream_t st) {
    ClusterArgs a = {};
    a.x = b.x;
    a.r = b.r;
    a.p = b.p;
    a.Kp = b.Kp;
    a.part = tail.part;
    a.S = tail.S;
    a.part_stride = tail.stride;
    a.scale = tail.scale;
    a.noise = tail.noise;
    a.total = (int)(N * t);
    a.t = t;
    a.st = b.state;
    a.hist_alpha = b.hist_alpha;
    a.hist_beta = b.hist_beta;
    a.split = split ? 1 : 0;
    if (split) a.sp = *split;
    a.N = N;
    return ctas == 1 ? launch_cluster<1, kClVecs>(a, st)
         : ctas == 8 ? launch_cluster<8, kClVecs>(a, st)
                     : launch_cluster<kClWide, kClWideVecs>(a, st);
}

}  // namespace lgp
