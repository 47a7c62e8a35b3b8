// Column sums of the CG kernels: compensated float pairs per thread, fixed point across a block's threads, float64 across
// the CTAs of a cluster.
#pragma once

#include <cooperative_groups.h>

#include "lgp_internal.cuh"
#include "limb_sum.cuh"

namespace lgp {

__device__ __forceinline__ void pair_add(float &h, float &l, float h2, float l2) {
    const float s = __fadd_rn(h, h2);
    const float bb = __fsub_rn(s, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
    h = s;
    l = __fadd_rn(__fadd_rn(l, l2), e);
}

// Column layout of the element-wise loops. VEC = 4 (t a power of two): thread x of the block handles float4s at
// a stride that is a multiple of t, so its four elements always have the columns (4 x + k) mod t. VEC = 1: any t,
// the block has a multiple of t threads and thread x owns column x mod t.
template <int VEC> __device__ __forceinline__ int col_of(int tid, int k, int t) { return (VEC * tid + k) % t; }

template <int VEC> __device__ __forceinline__ void load_vec(const float *p, float (&v)[VEC]) {
    if constexpr (VEC == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        v[0] = *p;
    }
}
template <int VEC> __device__ __forceinline__ void store_vec(float *p, const float (&v)[VEC]) {
    if constexpr (VEC == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else *p = v[0];
}

// Working memory of one block_col_sums call; cleared, and a barrier passed, before it.
struct ColSums {
    unsigned int mx[kMaxT];  // largest magnitude per column
    int limb[3][kMaxT];
};
__device__ __forceinline__ void clear_sums(ColSums &s) {
    if (threadIdx.x < kMaxT) {
        s.mx[threadIdx.x] = 0u;
        s.limb[0][threadIdx.x] = s.limb[1][threadIdx.x] = s.limb[2][threadIdx.x] = 0;
    }
}

// v[k] of the lanes that hold the same columns (those that agree mod group, group = 1 .. 16) combined by op, each step
// halving what a lane carries: for group <= 8 the result in r[0] is that of k = 2 bit4 + bit3 of the lane (the same in lanes
// that differ only in the bits from group to 4), for group = 16 r[0] and r[1] are those of k = 2 bit4 and the next.
template <class T, class Op> __device__ __forceinline__ void fold_columns(const T (&v)[4], int group, int lane, Op op, T (&r)[2]) {
    const bool up = lane & 16, second = lane & 8;
    const T s0 = up ? v[0] : v[2], s1 = up ? v[1] : v[3];
    r[0] = op(up ? v[2] : v[0], __shfl_xor_sync(0xffffffffu, s0, 16));
    r[1] = op(up ? v[3] : v[1], __shfl_xor_sync(0xffffffffu, s1, 16));
    if (group > 8) return;
    const T s = second ? r[0] : r[1];
    r[0] = op(second ? r[1] : r[0], __shfl_xor_sync(0xffffffffu, s, 8));
    for (int off = group; off < 8; off <<= 1) r[0] = op(r[0], __shfl_xor_sync(0xffffffffu, r[0], off));
}

// Sums the float pairs of every column over the block: out_row[c] = their float64 value, c < t, written by thread c.
// The sum across threads is the block's largest magnitude per column, then integer sums (limb_sum.cuh): float64 additions
// would take 64 cycles of a sub-partition per warp (a tree over 512 threads 1650 cycles), float pairs lose bits and
// overflow where float64 does not. At 1 and 2 columns a warp's maximum and sums are one reduction instruction each (at 4
// their 16 are slower than folding: N = 500, t = 4 15.3 and 14.7 us an iteration). An iteration with its product, pairs by
// shuffles -> this: N = 2000, D = 6, t = 1 18.2 -> 16.6 us, t = 8 20.3 -> 20.1; N = 500, t = 4 14.2 -> 14.7; N = 4000, t = 32 40.5 ->
// 39.0; N = 20000, D = 8, t = 32 156.3 -> 153.8.
template <int VEC>
__device__ void block_col_sums(float (&hi)[VEC], float (&lo)[VEC], int t, ColSums &s, double *out_row) {
    const int tid = threadIdx.x;
    if constexpr (VEC == 1) {
        const int c = tid % t;
        atomicMax(&s.mx[c], max(magnitude_bits(hi[0]), magnitude_bits(lo[0])));
        __syncthreads();
        const float scale = limb_scale(s.mx[c]);
        int l[3] = {0, 0, 0};
        add_limbs(hi[0], scale, l);
        add_limbs(lo[0], scale, l);
#pragma unroll
        for (int j = 0; j < 3; ++j) atomicAdd(&s.limb[j][c], l[j]);
    } else {
        const int lane = tid & 31;
        if (t == 1) {
            pair_add(hi[0], lo[0], hi[1], lo[1]);
            pair_add(hi[2], lo[2], hi[3], lo[3]);
            pair_add(hi[0], lo[0], hi[2], lo[2]);
        } else if (t == 2) {
            pair_add(hi[0], lo[0], hi[2], lo[2]);
            pair_add(hi[1], lo[1], hi[3], lo[3]);
        }
        const int group = t > 4 ? t / 4 : 1;  // lanes that hold one row of columns
        if (t < 4) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (k >= t) break;
                const unsigned int m = __reduce_max_sync(0xffffffffu, max(magnitude_bits(hi[k]), magnitude_bits(lo[k])));
                if (lane == 0) atomicMax(&s.mx[k], m);
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (k >= t) break;
                const float scale = limb_scale(s.mx[k]);
                int l[3] = {0, 0, 0};
                add_limbs(hi[k], scale, l);
                add_limbs(lo[k], scale, l);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int v = __reduce_add_sync(0xffffffffu, l[j]);
                    if (lane == 0) atomicAdd(&s.limb[j][k], v);
                }
            }
        } else {
            // this lane's columns after fold_columns, and whether it is the one that adds them
            const int col = 4 * (lane & (group - 1)) + 2 * (lane >> 4) + (group > 8 ? 0 : (lane >> 3) & 1);
            const bool adds = group > 8 || (lane & 7) < group;
            unsigned int m[4], mr[2];
#pragma unroll
            for (int k = 0; k < 4; ++k) m[k] = max(magnitude_bits(hi[k]), magnitude_bits(lo[k]));
            fold_columns(m, group, lane, [](unsigned int a, unsigned int b) { return max(a, b); }, mr);
            if (adds) atomicMax(&s.mx[col], mr[0]);
            if (group > 8) atomicMax(&s.mx[col + 1], mr[1]);
            __syncthreads();
            int l[3][4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float scale = limb_scale(s.mx[(4 * lane + k) & (t - 1)]);
                int p[3] = {0, 0, 0};
                add_limbs(hi[k], scale, p);
                add_limbs(lo[k], scale, p);
#pragma unroll
                for (int j = 0; j < 3; ++j) l[j][k] = p[j];
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                int r[2];
                fold_columns(l[j], group, lane, [](int a, int b) { return a + b; }, r);
                if (adds) atomicAdd(&s.limb[j][col], r[0]);
                if (group > 8) atomicAdd(&s.limb[j][col + 1], r[1]);
            }
        }
    }
    __syncthreads();
    if (tid < t) out_row[tid] = limb_total(s.limb[0][tid], s.limb[1][tid], s.limb[2][tid], s.mx[tid]);
}

// Sum over the cluster's CTAs of mine[c] (shared memory, written before), c < t, in rank order, for threads c < t.
template <int CL> __device__ double cluster_sum(double *mine, int t) {
    double s = 0.0;
    if constexpr (CL == 1) {
        __syncthreads();
        if ((int)threadIdx.x < t) s = mine[threadIdx.x];
    } else {
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        cl.sync();
        if ((int)threadIdx.x < t) {
#pragma unroll
            for (int q = 0; q < CL; ++q) s += cl.map_shared_rank(mine, q)[threadIdx.x];
        }
    }
    return s;
}

}  // namespace lgp
