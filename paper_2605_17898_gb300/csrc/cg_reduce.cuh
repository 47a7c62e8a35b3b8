// Column sums of the CG kernels: compensated float pairs within a block.
#pragma once

#include "lgp_internal.cuh"

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

// Sums the float pairs of every column over the block: out_row[c] = their float64 value, c < t (valid after the next
// barrier). red: 64 x 32 pairs.
template <int VEC>
__device__ void block_pairs_reduce(float (&hi)[VEC], float (&lo)[VEC], int t, float2 *red, double *out_row) {
    const int tid = threadIdx.x;
    if constexpr (VEC == 1) {
        const int nr = blockDim.x / t;
        red[tid] = make_float2(hi[0], lo[0]);
        __syncthreads();
        int s = 1;
        while (s < nr) s <<= 1;
        for (s >>= 1; s >= 1; s >>= 1) {
            const int slot = tid / t;
            if (slot < s && slot + s < nr) {
                float2 a = red[tid];
                const float2 b = red[tid + s * t];
                pair_add(a.x, a.y, b.x, b.y);
                red[tid] = a;
            }
            __syncthreads();
        }
        if (tid < t) out_row[tid] = (double)red[tid].x + (double)red[tid].y;
    } else {
        const int lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
        if (t == 1) {
            pair_add(hi[0], lo[0], hi[1], lo[1]);
            pair_add(hi[2], lo[2], hi[3], lo[3]);
            pair_add(hi[0], lo[0], hi[2], lo[2]);
        } else if (t == 2) {
            pair_add(hi[0], lo[0], hi[2], lo[2]);
            pair_add(hi[1], lo[1], hi[3], lo[3]);
        }
        const int group = t > 4 ? t / 4 : 1;  // lanes that hold one row of columns
        for (int off = group; off < 32; off <<= 1) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                const float h2 = __shfl_xor_sync(0xffffffffu, hi[k], off), l2 = __shfl_xor_sync(0xffffffffu, lo[k], off);
                pair_add(hi[k], lo[k], h2, l2);
            }
        }
        if (lane < group) {
#pragma unroll
            for (int k = 0; k < VEC; ++k)
                if (4 * lane + k < t) red[(4 * lane + k) * 32 + warp] = make_float2(hi[k], lo[k]);
        }
        __syncthreads();
        for (int c = warp; c < t; c += nw) {
            float2 v = lane < nw ? red[c * 32 + lane] : make_float2(0.0f, 0.0f);
            for (int off = 16; off > 0; off >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, v.x, off), l2 = __shfl_xor_sync(0xffffffffu, v.y, off);
                pair_add(v.x, v.y, h2, l2);
            }
            if (lane == 0) out_row[c] = (double)v.x + (double)v.y;
        }
    }
}

}  // namespace lgp
