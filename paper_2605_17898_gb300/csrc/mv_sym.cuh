// Symmetric FP32 product K_y V for t <= 4 columns (templates; one translation unit per kernel kind).
//
// The row-by-row kernel (mv_simt.cuh) generates every entry twice and is bound by the issue of its scalar float32
// operations. Here each unordered pair's entry is generated once and used for both rows, on packed float32x2
// operations, so that per pair the FMA pipe does 2D + kernel + 2t operations where it did twice (2D + kernel + t):
//   - the points are cut into G blocks of E rows, and one CTA computes the E x E block tile (I, J), I <= J:
//     its row sums go to part[J][rows of I], its column sums to part[I][rows of J]. Every (slot, row) is written by
//     exactly one CTA, and out = sum_s part[s] + noise V adds the G slots in order: no atomics, the same result at
//     every run. (Diagonal tiles compute all E x E entries and only row sums.)
//   - a warp sweeps columns for 8R rows at a time: 8 row lanes x R rows and 4 column lanes x C columns per step. Each
//     thread keeps R rows of x and V and their sums in registers; the column side is staged in shared memory once
//     per tile. The 4 warps take different rows, and all columns (long sweeps pay for a sweep's loads and row sums); in
//     tiles of fewer than 4 row sweeps they share the columns of one sweep instead.
//   - a packed operation with three different register pairs takes four cycles of the FMA pipe, one with two takes two
//     (microbenchmark: FFMA2 a*b+c 3.96 cycles, FFMA2 d*d+a 2.15, FADD2 2.17, scalar FFMA 1.09). So the distances are
//     packed, as (-x_j) + x_i and d*d + r^2; the entry's and V's multiply-adds are scalar.
//   - a shared-memory load costs the floats it delivers to the registers (128 bytes per SM and clock, broadcast or
//     not), so nothing is stored twice there: the pairs are two neighbouring columns, and a packed operation's missing
//     broadcast is made up by keeping each row's coordinates twice in registers.
//   - a column's sum over the warp's rows is folded over the 8 row lanes by a transposing butterfly (C t values in
//     4, 7 or 14 shuffles instead of 3 each) and added by one lane, always the same, to its row set's column sums in
//     shared memory. This costs 3 of 15 cycles per pair at D = 4, t = 1; a copy of the sums per row lane, without any
//     shuffle, measured 11% slower (its loads and stores, and fewer CTAs per SM).
// Sums are short: at most E / 4 terms per lane and chain (a lane's four columns in each of E / 16 steps), then trees and G
// slots.
//
// Measured against the row kernel (product call, us): N = 50000, t = 1, RBF D = 4 970 -> 475, Matern-5/2 D = 8
// 1824 -> 939; N = 20000, D = 8, Matern-5/2: t = 2 336 -> 197, t = 4 362 -> 271; N = 2000, D = 8, t = 1 33 -> 19. The
// distances alone (FADD2, FFMA2) are 8.7 of the 15 cycles of an FP32 sub-partition per pair and warp at D = 4. At
// t = 8 the folds and V's loads outweigh the saved distances (N = 20000, D = 3 269 -> 285 us): the row kernel keeps t > 4.
#pragma once

#include "lgp_internal.cuh"

namespace lgp {

struct SymArgs {
    const float *Xs;   // prescaled points [Np, DP]
    const float *V;    // [N, ldv]
    float *part;       // [G, Np, t]
    const int *skip;
    int64_t N, Np, ldv;
    int E, G, t;
    EntryScale scale;
};

constexpr int kSymThreads = 128;  // 4 warps: row sets, or in small tiles shares of the columns

// Rows per thread, columns per thread and step, by dimension and padded column count (what the registers hold).
template <int D, int TT> struct SymShape {
    static constexpr int R = D <= 4 && TT <= 2 ? 8 : 4;
    static constexpr int C = 4;  // one 16-byte load per coordinate
    static constexpr int RB = 8 * R;  // rows of one sweep
};

// Row sets of the 4 warps (the others share a sweep's columns).
template <int D, int TT> __host__ __device__ constexpr int sym_row_sets(int E) {
    return E >= 4 * SymShape<D, TT>::RB ? 4 : E / SymShape<D, TT>::RB;
}
// Shared memory of a CTA: column side, column sums of the row sets, row sums.
constexpr int sym_smem_bytes(int D, int TT, int E) {
    const int RB = D <= 4 && TT <= 2 ? 64 : 32, sets = E >= 4 * RB ? 4 : E / RB;
    return (E * (D + TT + TT * sets) + 4 * RB * TT) * 4;
}

// v[0..NV) summed over the 8 lanes that differ in bits 0..2: the lane keeps values sym_fold_index(lane) + 0 ..
// NV / 8 - 1 in v[0], v[1]. NV = 4: lanes that differ in bit 2 hold the same value.
template <int NV>
__device__ __forceinline__ void sym_fold(float (&v)[NV], int lane) {
    int n = NV;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const bool up = (lane >> s) & 1;
        if (n > 1) {
            n >>= 1;
#pragma unroll
            for (int k = 0; k < NV / 2; ++k) {
                if (k >= n) break;
                const float send = up ? v[k] : v[k + n];
                const float keep = up ? v[k + n] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << s);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1 << s);
        }
    }
}
template <int NV> __device__ __forceinline__ int sym_fold_index(int lane) {
    const int b0 = lane & 1, b1 = (lane >> 1) & 1, b2 = (lane >> 2) & 1;
    return NV == 4 ? 2 * b0 + b1 : b0 * (NV / 2) + b1 * (NV / 4) + b2 * (NV / 8);
}

template <int KIND, int D, int TT>
__global__ void __launch_bounds__(kSymThreads) mv_sym_kernel(SymArgs a) {
    constexpr int DP = D <= 4 ? 4 : 8;
    using S = SymShape<D, TT>;
    constexpr int R = S::R, C = S::C, RB = S::RB, NV = C * TT;
    extern __shared__ float4 sym_smem[];
    const int E = a.E;
    float *xs = reinterpret_cast<float *>(sym_smem);        // [D][E]
    float *vs = xs + D * E;                                 // [E][TT]
    // warps: WR row sets x WC column sets
    const int WR = sym_row_sets<D, TT>(E), WC = 4 / WR;
    float *col = vs + E * TT;                               // [WR][E][TT] column sums of the row sets
    float *rowbuf = col + WR * E * TT;                      // [4][RB][TT] row sums of warps that share a sweep

    // tile (I, J) of the triangle, numbered row by row
    const int G = a.G;
    int I = (int)((2 * G + 1 - sqrtf((float)(2 * G + 1) * (2 * G + 1) - 8.0f * blockIdx.x)) * 0.5f);
    I = max(0, min(I, G - 1));
    auto row_start = [G](int i) { return i * G - i * (i - 1) / 2; };
    while (I > 0 && row_start(I) > (int)blockIdx.x) --I;
    while (I + 1 < G && row_start(I + 1) <= (int)blockIdx.x) ++I;
    const int J = I + ((int)blockIdx.x - row_start(I));
    const bool diag = I == J;
    const int64_t i0 = (int64_t)I * E, j0 = (int64_t)J * E;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rl = lane & 7, cl = lane >> 3;

    chain_wait();
    chain_next();
    if (a.skip && *a.skip) return;
    // column side: -x_j and V_j; column sums zero
    for (int e = tid; e < E * (DP / 4); e += kSymThreads) {
        const int j = e / (DP / 4), q = e - j * (DP / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j0 + j < a.Np) v = *reinterpret_cast<const float4 *>(a.Xs + (j0 + j) * DP + 4 * q);
        const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * q + k < D) xs[(4 * q + k) * E + j] = -f[k];
    }
    for (int e = tid; e < E * TT; e += kSymThreads) {
        const int j = e / TT, c = e - j * TT;
        vs[e] = (j0 + j < a.N && c < a.t) ? rbf_scaled<KIND>(a.V[(j0 + j) * a.ldv + c], a.scale.v) : 0.0f;
    }
    for (int e = tid; e < WR * E * TT; e += kSymThreads) col[e] = 0.0f;
    __syncthreads();

    const float ls2 = a.scale.log2s2;
    const float2 acc_init = PackedEntry<KIND>::acc0(ls2);
    const int wr = warp / WC, wc = warp % WC;
    const int cw = E / WC, c_lo = wc * cw;  // columns of this warp
    float *mycol = col + wr * E * TT + sym_fold_index<NV>(lane);

    for (int rb0 = 0; rb0 < E; rb0 += WR * RB) {
        const int rb = rb0 + wr * RB;
        if (WC == 1 && i0 + rb >= a.N) break;  // (rows past N count as zero where warps meet at barriers)
        // this thread's rows rl R .. rl R + R - 1 of the sweep, each coordinate twice
        float2 xi[R][D];
        float vi[R][TT], acc[R][TT];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = i0 + rb + rl * R + r;
            float x[DP];
#pragma unroll
            for (int q = 0; q < DP; q += 4) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < a.Np) v = *reinterpret_cast<const float4 *>(a.Xs + i * DP + q);
                x[q] = v.x;
                x[q + 1] = v.y;
                x[q + 2] = v.z;
                x[q + 3] = v.w;
            }
#pragma unroll
            for (int d = 0; d < D; ++d) xi[r][d] = make_float2(x[d], x[d]);
#pragma unroll
            for (int c = 0; c < TT; ++c) {
                vi[r][c] = i < a.N && c < a.t ? rbf_scaled<KIND>(a.V[i * a.ldv + c], a.scale.v) : 0.0f;
                acc[r][c] = 0.0f;
            }
        }
#pragma unroll 1
        for (int s = c_lo; s < c_lo + cw; s += 4 * C) {
            const int j = s + C * cl;  // this lane's C columns
            float2 xj[C / 2][D];
            float vj[C * TT], cs[NV];
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const float4 q = *reinterpret_cast<const float4 *>(xs + d * E + j);
                xj[0][d] = make_float2(q.x, q.y);
                xj[1][d] = make_float2(q.z, q.w);
            }
#pragma unroll
            for (int q = 0; q < C * TT; q += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(vs + j * TT + q);
                vj[q] = v.x;
                vj[q + 1] = v.y;
                vj[q + 2] = v.z;
                vj[q + 3] = v.w;
            }
#pragma unroll
            for (int h = 0; h < C / 2; ++h) {
                const int c0 = 2 * h * TT, c1 = c0 + TT;  // the pair's columns in vj and cs
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float2 dd = __fadd2_rn(xj[h][0], xi[r][0]);
                    float2 r2 = __ffma2_rn(dd, dd, acc_init);
#pragma unroll
                    for (int d = 1; d < D; ++d) {
                        dd = __fadd2_rn(xj[h][d], xi[r][d]);
                        r2 = __ffma2_rn(dd, dd, r2);
                    }
                    const float2 k = PackedEntry<KIND>::k(r2, ls2);
#pragma unroll
                    for (int q = 0; q < TT; ++q) {
                        acc[r][q] = fmaf(k.y, vj[c1 + q], fmaf(k.x, vj[c0 + q], acc[r][q]));
                        cs[c0 + q] = r == 0 ? k.x * vi[r][q] : fmaf(k.x, vi[r][q], cs[c0 + q]);
                        cs[c1 + q] = r == 0 ? k.y * vi[r][q] : fmaf(k.y, vi[r][q], cs[c1 + q]);
                    }
                }
            }
            if (!diag) {
                sym_fold<NV>(cs, lane);
                float *dst = mycol + j * TT;
                if constexpr (NV == 4) {
                    if ((lane & 4) == 0) dst[0] += cs[0];
                } else {
#pragma unroll
                    for (int k = 0; k < NV / 8; ++k) dst[k] += cs[k];
                }
            }
        }
        // row sums: over the 4 column lanes, then, where warps share the sweep, over them in order
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < TT; ++q) {
                float v = acc[r][q];
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                const int64_t i = i0 + rb + rl * R + r;
                if (cl == (r & 3)) {
                    if (WC > 1) rowbuf[(warp * RB + rl * R + r) * TT + q] = v;
                    else if (i < a.N && q < a.t) a.part[((int64_t)J * a.Np + i) * a.t + q] = v;
                }
            }
        if (WC > 1) {
            __syncthreads();
            for (int e = tid; e < WR * RB * TT; e += kSymThreads) {
                const int w0 = e / (RB * TT), c = e % TT;  // row set
                const int64_t i = i0 + rb0 + e / TT;
                float v = 0.0f;
                for (int k = 0; k < WC; ++k) v += rowbuf[(w0 * WC + k) * RB * TT + e - w0 * RB * TT];
                if (i < a.N && c < a.t) a.part[((int64_t)J * a.Np + i) * a.t + c] = v;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    if (diag) return;
    for (int e = tid; e < E * TT; e += kSymThreads) {
        const int j = e / TT, c = e - j * TT;
        float v = 0.0f;
        for (int w = 0; w < WR; ++w) v += col[w * E * TT + e];
        if (j0 + j < a.N && c < a.t) a.part[((int64_t)I * a.Np + j0 + j) * a.t + c] = v;
    }
}

cudaError_t mv_sym_dispatch_rbf(int D, int TT, const SymArgs &a, cudaStream_t st);
cudaError_t mv_sym_dispatch_m52(int D, int TT, const SymArgs &a, cudaStream_t st);
cudaError_t mv_sym_dispatch_m12(int D, int TT, const SymArgs &a, cudaStream_t st);
cudaError_t mv_sym_dispatch_m32(int D, int TT, const SymArgs &a, cudaStream_t st);

template <int KIND, int D, int TT>
cudaError_t launch_mv_sym_inst(const SymArgs &a, cudaStream_t st) {
    static_assert(SymShape<D, TT>::RB == (D <= 4 && TT <= 2 ? 64 : 32), "sym_smem_bytes and SymShape agree");
    const int bytes = sym_smem_bytes(D, TT, a.E);
    if (bytes > 48 * 1024) {  // set at every such launch: the attribute belongs to the current device
        const cudaError_t e = cudaFuncSetAttribute(mv_sym_kernel<KIND, D, TT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   200 * 1024);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(mv_sym_kernel<KIND, D, TT>, dim3((unsigned)(a.G * (a.G + 1) / 2)), kSymThreads, bytes, st, a);
}

template <int KIND, int TT>
cudaError_t dispatch_mv_sym_d(int D, const SymArgs &a, cudaStream_t st) {
    switch (D) {
        case 1: return launch_mv_sym_inst<KIND, 1, TT>(a, st);
        case 2: return launch_mv_sym_inst<KIND, 2, TT>(a, st);
        case 3: return launch_mv_sym_inst<KIND, 3, TT>(a, st);
        case 4: return launch_mv_sym_inst<KIND, 4, TT>(a, st);
        case 5: return launch_mv_sym_inst<KIND, 5, TT>(a, st);
        case 6: return launch_mv_sym_inst<KIND, 6, TT>(a, st);
        case 7: return launch_mv_sym_inst<KIND, 7, TT>(a, st);
        case 8: return launch_mv_sym_inst<KIND, 8, TT>(a, st);
    }
    return cudaErrorInvalidValue;
}

template <int KIND>
cudaError_t dispatch_mv_sym(int D, int TT, const SymArgs &a, cudaStream_t st) {
    switch (TT) {
        case 1: return dispatch_mv_sym_d<KIND, 1>(D, a, st);
        case 2: return dispatch_mv_sym_d<KIND, 2>(D, a, st);
        case 4: return dispatch_mv_sym_d<KIND, 4>(D, a, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lgp
