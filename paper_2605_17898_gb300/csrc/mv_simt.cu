// Host launchers of the FP32 SIMT product family: tile choice, column splits and the split reductions.
#include <algorithm>

#include "mv_simt.cuh"
#include "mv_sym.cuh"

namespace lgp {

namespace {

// CTAs per SM that the row kernel's splits aim at (64 threads each), down to one column tile per split: at small N the
// tiles of a split are a serial chain of loads and barriers. Against at least 4 tiles per split: N = 1200, D = 6, t = 8
// 35 -> 15 us, N = 4099, D = 5, t = 5 39 -> 25 us; 16 -> 32 CTAs: N = 20000, D = 8, t = 8 410 -> 388 us. (The partial
// sums stay at that many CTAs x SMs x rows of a CTA x t floats.)
// From 16 columns on a split's partial sums cost more than its share of the entries, so there it is 8 CTAs (6 from 32
// columns on), 16 where the row blocks and column groups alone give every second SM a CTA and 32 where they give every SM one
// (the last wave is long): N = 6000, D = 8, t = 32 6 CTAs 111 us, 8 122, 16 134, 32 163; t = 16 8 77, 16 and 32 87; N = 16000, t = 32
// 8 711, 16 618, 32 638; N = 20000, D = 2, t = 32 16 734, 32 707. At t = 12 (N = 10000, D = 8) 8 169, 16 149, 32 160.
int row_ctas(int t, int64_t ctas, int num_sms) {
    if (t < 16 || ctas >= num_sms) return 32;
    if (2 * ctas >= num_sms) return 16;
    return t < 32 ? 8 : 6;
}

// Padded columns of a launch and its CTA's rows.
struct SimtShape {
    int TT, BM;
};

template <int TT> constexpr SimtShape shape_of() { return {TT, RowShape<TT>::kRows}; }

SimtShape simt_shape(int t) {
    if (t == 1) return shape_of<1>();
    if (t == 2) return shape_of<2>();
    if (t <= 4) return shape_of<4>();
    if (t <= 8) return shape_of<8>();
    if (t <= 16) return shape_of<16>();
    return shape_of<32>();
}

// Column splits so that row blocks x splits x column groups fill the GPU a few
// times over; each split covers a whole number of BN tiles.
int64_t choose_split(int64_t N, int64_t row_blocks, int64_t col_groups, int num_sms, int64_t *cols_per_split,
                     int ctas_per_sm = 8, int64_t tiles_per_split = 4) {
    const int64_t col_tiles = (N + kSimtBN - 1) / kSimtBN;
    const int64_t want = (int64_t)num_sms * ctas_per_sm;
    int64_t s = (want + row_blocks * col_groups - 1) / (row_blocks * col_groups);
    s = std::max<int64_t>(1, std::min<int64_t>(s, std::max<int64_t>(1, col_tiles / tiles_per_split)));
    const int64_t tiles_per = (col_tiles + s - 1) / s;
    *cols_per_split = tiles_per * kSimtBN;
    return (N + *cols_per_split - 1) / *cols_per_split;
}

// Symmetric product (mv_sym.cuh): block edge E, blocks G and padded column count TT for a square product of N rows
// and t columns, or E = 0 where the row-by-row kernel runs: t > 4; or N so large that the partial sums, G per row,
// would take more than 256 MiB with E = 512 and E = 1024 does not help. Blocks of 1024 need two CTAs of 4 warps on an SM:
// with one (114 KB of shared memory at D = 8, 4 padded columns) N = 100000, D = 8, t = 4, Matern-5/2 took 10.3 ms, the row
// kernel takes 7.2; at D = 7 they take 6.8 against 8.1 (N = 110000), at t = 1, N = 200000, D = 4 10.0 against 17.2.
struct SymGrid {
    int E = 0, G = 0, TT = 0;
};

constexpr int64_t kSymMaxPartial = 256ll << 20;
constexpr int kSmShared = 228 * 1024, kCtaReserved = 1024;  // bytes of shared memory of an SM, and the system's share per CTA

SymGrid sym_grid(int64_t N, int64_t Np, int t, int D, int num_sms) {
    SymGrid g;
    if (t > 4) return g;
    // The largest blocks that still give every SM enough tiles to even out the last ones (a tile's set-up and its
    // sums are paid per tile, and each block is one more partial sum per row: N = 50000, D = 4, t = 1 with
    // E = 256 535 us, 512 476); larger ones only to keep the partial sums in bounds. (A solve's vector step reads every
    // partial sum, so that blocks of 128 from one tile per SM on would make its iterations faster, N = 2500, t = 1 21.8 ->
    // 18.2 us; but their sums' chains are twice as long, and the products' errors 10% larger there.)
    auto tiles_per_sm = [&](int64_t E) {
        const int64_t G = (N + E - 1) / E;
        return G * (G + 1) / 2 / num_sms;
    };
    const int TT = t <= 2 ? t : 4;
    int64_t E = 64;
    if (tiles_per_sm(512) >= 16) E = 512;
    else if (tiles_per_sm(256) >= 8) E = 256;
    else if (tiles_per_sm(128) >= 5) E = 128;
    auto bytes = [&](int64_t e) { return (N + e - 1) / e * Np * t * (int64_t)sizeof(float); };
    if (E == 512 && bytes(E) > kSymMaxPartial && 2 * (sym_smem_bytes(D, TT, 1024) + kCtaReserved) <= kSmShared) E = 1024;
    if (bytes(E) > kSymMaxPartial) return g;
    g.E = (int)E;
    g.G = (int)((N + E - 1) / E);
    g.TT = TT;
    return g;
}

// out = scale sum_k partial[k] + noise V. Rows are the output's (N, padded Np); cross = 1 drops the noise term (V has other rows).
__global__ void reduce_split_kernel(const float *__restrict__ partial, int S, int64_t Np, int64_t N, int t,
                                    const float *__restrict__ V, int64_t ldv, float *__restrict__ out, int64_t ldo,
                                    float scale, float noise, int cross, const int *skip) {
    chain_wait();
    chain_next();
    if (skip && *skip) return;
    const int64_t total = N * t;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / t;
        const int c = (int)(e - i * t);
        float s = 0.0f;
        for (int k = 0; k < S; ++k) s += partial[((int64_t)k * Np + i) * t + c];
        s *= scale;
        out[i * ldo + c] = cross ? s : fmaf(noise, V[i * ldv + c], s);
    }
}

// The same for many splits (S >= 8): 8 lanes share 4 consecutive elements, lane q taking splits q, q + 8, ... as 16-byte
// loads, so that the loads of one element's splits overlap (product at t = 1: N = 5000, 40 splits 22 -> 19 us; N = 50000, 98
// splits 476 -> 472 us).
__global__ void __launch_bounds__(256) reduce_many_kernel(const float *__restrict__ partial, int S, int64_t Np, int64_t N,
                                                          int t, const float *__restrict__ V, int64_t ldv,
                                                          float *__restrict__ out, int64_t ldo, float scale, float noise,
                                                          int cross, const int *skip) {
    chain_wait();
    chain_next();
    if (skip && *skip) return;
    const int lane = threadIdx.x & 31, q = lane >> 2;
    const int64_t total = N * t;
    const int64_t e = 4 * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32 * 4 + (lane & 3));
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < total) {
#pragma unroll 4
        for (int k = q; k < S; k += 8) {
            const float4 v = *reinterpret_cast<const float4 *>(partial + (int64_t)k * Np * t + e);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, off);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, off);
    }
    if (q < 4 && e + q < total) {
        const float v = scale * (q == 0 ? s.x : q == 1 ? s.y : q == 2 ? s.z : s.w);
        const int64_t i = (e + q) / t;
        const int c = (int)(e + q - i * t);
        out[i * ldo + c] = cross ? v : fmaf(noise, V[i * ldv + c], v);
    }
}

__global__ void reduce_grad_kernel(const float *__restrict__ partial, int S, int NB, int64_t Np, int64_t N, int t,
                                   const float *__restrict__ W, float noise, float *__restrict__ G) {
    const int64_t total = (int64_t)(NB + 1) * N * t;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = e / (N * t);
        const int64_t rem = e - p * N * t;
        const int64_t i = rem / t;
        const int c = (int)(rem - i * t);
        if (p == NB) {
            G[e] = noise * W[i * t + c];
            continue;
        }
        float s = 0.0f;
        for (int k = 0; k < S; ++k) s += partial[(((int64_t)k * NB + p) * Np + i) * t + c];
        G[e] = s;
    }
}

inline int grid_for(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 4096));
}

}  // namespace

int64_t mv_simt_partial_floats(int64_t N, int64_t Np, int t, int D, int num_sms) {
    const SymGrid sg = sym_grid(N, Np, t, D, num_sms);
    if (sg.E) return (int64_t)sg.G * Np * t;
    const SimtShape sh = simt_shape(t);
    const int64_t BM = sh.BM;
    const int64_t rb = (N + BM - 1) / BM;
    const int64_t cg = (t + sh.TT - 1) / sh.TT;
    int64_t cps;
    const int64_t S = choose_split(N, rb, cg, num_sms, &cps, row_ctas(t, rb * cg, num_sms), 1);
    return S > 1 ? S * Np * t : 0;
}

int64_t mv_simt_cross_partial_floats(int64_t Nr, int64_t Npr, int64_t N, int t, int num_sms) {
    const SimtShape sh = simt_shape(t);
    const int64_t BM = sh.BM;
    const int64_t rb = (Nr + BM - 1) / BM;
    const int64_t cg = (t + sh.TT - 1) / sh.TT;
    int64_t cps;
    const int64_t S = choose_split(N, rb, cg, num_sms, &cps, row_ctas(t, rb * cg, num_sms), 1);
    return S > 1 ? S * Npr * t : 0;
}

// The sum of S partial results and the noise term, or, with m.tail, what the caller needs to take it over.
static cudaError_t finish_splits(const MvLaunch &m, int S, int64_t Nr, int64_t Npr, int cross, cudaStream_t st) {
    const float scale = entry_scale(*m.kp).out;
    if (m.tail) {
        m.tail->part = m.partial;
        m.tail->S = S;
        m.tail->stride = Npr * m.t;
        m.tail->scale = scale;
        m.tail->noise = m.kp->noise;
        return cudaSuccess;
    }
    if (S >= 8)
        return launch_chained(reduce_many_kernel, (unsigned)((Nr * m.t + 127) / 128), 256, 0, st, m.partial, S, Npr, Nr, m.t,
                              m.V, m.ldv, m.out, m.ldo, scale, m.kp->noise, cross, m.skip);
    return launch_chained(reduce_split_kernel, grid_for(Nr * m.t), 256, 0, st, m.partial, S, Npr, Nr, m.t, m.V, m.ldv, m.out,
                          m.ldo, scale, m.kp->noise, cross, m.skip);
}

cudaError_t launch_mv_simt(const MvLaunch &m, cudaStream_t st) {
    const bool cross = m.Xr != nullptr;
    const int64_t Nr = cross ? m.Nr : m.N, Npr = cross ? m.Npr : m.Np;
    if (m.tail) *m.tail = ProductTail();
    const SymGrid sg = cross || m.rows ? SymGrid() : sym_grid(m.N, m.Np, m.t, m.kp->D, m.num_sms);
    if (sg.E && m.partial != nullptr && (int64_t)sg.G * m.Np * m.t <= m.partial_cap) {
        SymArgs a;
        a.Xs = m.Xs;
        a.V = m.V;
        a.part = m.partial;
        a.skip = m.skip;
        a.N = m.N;
        a.Np = m.Np;
        a.ldv = m.ldv;
        a.E = sg.E;
        a.G = sg.G;
        a.t = m.t;
        a.scale = entry_scale(*m.kp);
        cudaError_t e;
        switch (m.kp->kind) {
            case LGP_RBF: e = mv_sym_dispatch_rbf(m.kp->D, sg.TT, a, st); break;
            case LGP_MATERN52: e = mv_sym_dispatch_m52(m.kp->D, sg.TT, a, st); break;
            case LGP_MATERN12: e = mv_sym_dispatch_m12(m.kp->D, sg.TT, a, st); break;
            case LGP_MATERN32: e = mv_sym_dispatch_m32(m.kp->D, sg.TT, a, st); break;
            default: e = cudaErrorInvalidValue;
        }
        return e != cudaSuccess ? e : finish_splits(m, sg.G, m.N, m.Np, 0, st);
    }
    const SimtShape sh = simt_shape(m.t);
    const int64_t BM = sh.BM;
    const int64_t rb = (Nr + BM - 1) / BM;
    const int64_t cg = (m.t + sh.TT - 1) / sh.TT;
    int64_t cps;
    int64_t S = choose_split(m.N, rb, cg, m.num_sms, &cps, row_ctas(m.t, rb * cg, m.num_sms), 1);
    if (S > 1 && (m.partial == nullptr || S * Npr * m.t > m.partial_cap)) {
        S = 1;
        cps = m.N;
    }
    SimtArgs a;
    a.Xs = m.Xs;
    a.Xr = cross ? m.Xr : m.Xs;
    a.Nr = Nr;
    a.Npr = Npr;
    a.cross = cross ? 1 : 0;
    a.V = m.V;
    a.out = m.out;
    a.partial = S > 1 ? m.partial : nullptr;
    a.skip = m.skip;
    a.N = m.N;
    a.Np = m.Np;
    a.ldv = m.ldv;
    a.ldo = m.ldo;
    a.cols_per_split = cps;
    a.t = m.t;
    const EntryScale es = entry_scale(*m.kp);
    a.log2s2 = es.log2s2;
    a.v_scale = es.v;
    a.out_scale = es.out;
    a.noise = m.kp->noise;
    const dim3 grid((unsigned)rb, (unsigned)S, (unsigned)cg);
    cudaError_t e;
    switch (m.kp->kind) {
        case LGP_RBF: e = mv_simt_dispatch_rbf(m.kp->D, sh.TT, grid, a, st); break;
        case LGP_MATERN52: e = mv_simt_dispatch_m52(m.kp->D, sh.TT, grid, a, st); break;
        case LGP_MATERN12: e = mv_simt_dispatch_m12(m.kp->D, sh.TT, grid, a, st); break;
        case LGP_MATERN32: e = mv_simt_dispatch_m32(m.kp->D, sh.TT, grid, a, st); break;
        default: e = cudaErrorInvalidValue;
    }
    if (e != cudaSuccess || S == 1) return e;
    return finish_splits(m, (int)S, Nr, Npr, a.cross, st);
}

int64_t mv_grad_partial_floats(int64_t N, int64_t Np, int t, int D, int num_sms) {
    const int TT = t == 1 ? 1 : 4;
    const int64_t rb = (N + kSimtThreads - 1) / kSimtThreads;
    const int64_t cg = (t + TT - 1) / TT;
    int64_t cps;
    const int64_t S = choose_split(N, rb, cg, num_sms, &cps);
    return S > 1 ? S * (D + 1) * Np * t : 0;
}

cudaError_t launch_mv_grad(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, const float *W, int t,
                           float *G, float *partial, int64_t partial_cap, int num_sms, cudaStream_t st) {
    const int TT = t == 1 ? 1 : 4;
    const int64_t rb = (N + kSimtThreads - 1) / kSimtThreads;
    const int64_t cg = (t + TT - 1) / TT;
    int64_t cps;
    int64_t S = choose_split(N, rb, cg, num_sms, &cps);
    const int NB = kp.D + 1;
    if (S > 1 && (partial == nullptr || S * NB * Np * t > partial_cap)) {
        S = 1;
        cps = N;
    }
    GradArgs a;
    a.Xs = Xs;
    a.W = W;
    a.G = G;
    a.partial = S > 1 ? partial : nullptr;
    a.N = N;
    a.Np = Np;
    a.cols_per_split = cps;
    a.t = t;
    a.log2s2 = kp.log2_s2;
    a.noise = kp.noise;
    const dim3 grid((unsigned)rb, (unsigned)S, (unsigned)cg);
    cudaError_t e;
    switch (kp.kind) {
        case LGP_RBF: e = mv_grad_dispatch_rbf(kp.D, TT, grid, a, st); break;
        case LGP_MATERN52: e = mv_grad_dispatch_m52(kp.D, TT, grid, a, st); break;
        case LGP_MATERN12: e = mv_grad_dispatch_m12(kp.D, TT, grid, a, st); break;
        case LGP_MATERN32: e = mv_grad_dispatch_m32(kp.D, TT, grid, a, st); break;
        default: e = cudaErrorInvalidValue;
    }
    if (e != cudaSuccess || S == 1) return e;
    reduce_grad_kernel<<<grid_for((int64_t)(NB + 1) * N * t), 256, 0, st>>>(partial, (int)S, NB, Np, N, t, W,
                                                                           kp.noise, G);
    return cudaGetLastError();
}

static int adjoint_tt(int t) {
    int TT = 1;
    while (TT < t) TT *= 2;
    return TT;
}

int64_t adjoint_partial_doubles(int64_t N, int t, int D, int num_sms) {
    const int64_t rb = (N + kSimtThreads - 1) / kSimtThreads;
    int64_t cps;
    const int64_t S = choose_split(N, rb, 1, num_sms, &cps);
    return rb * S * (D + 1);
}

cudaError_t launch_adjoint_bilinear(const KernelParams &kp, const float *Xs, int64_t N, int64_t Np, const float *A,
                                    const float *B, int t, double *block_partials, int64_t partial_cap, int *n_blocks,
                                    int num_sms, cudaStream_t st) {
    const int64_t rb = (N + kSimtThreads - 1) / kSimtThreads;
    int64_t cps;
    const int64_t S = choose_split(N, rb, 1, num_sms, &cps);
    if (rb * S * (kp.D + 1) > partial_cap) return cudaErrorInvalidValue;
    AdjArgs a;
    a.Xs = Xs;
    a.A = A;
    a.B = B;
    a.partial = block_partials;
    a.N = N;
    a.Np = Np;
    a.cols_per_split = cps;
    a.t = t;
    a.log2s2 = kp.log2_s2;
    *n_blocks = (int)(rb * S);
    const dim3 grid((unsigned)rb, (unsigned)S, 1);
    const int TT = adjoint_tt(t);
    switch (kp.kind) {
        case LGP_RBF: return adjoint_dispatch_rbf(kp.D, TT, grid, a, st);
        case LGP_MATERN52: return adjoint_dispatch_m52(kp.D, TT, grid, a, st);
        case LGP_MATERN12: return adjoint_dispatch_m12(kp.D, TT, grid, a, st);
        case LGP_MATERN32: return adjoint_dispatch_m32(kp.D, TT, grid, a, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lgp
