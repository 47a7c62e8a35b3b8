// The tensor-core products' split of V: 16-bit halves in the order the MMA reads (mv_tc.cu, cg_cluster.cu).
#pragma once

#include "mv_tc.cuh"

namespace lgp {

// Power-of-two exponent e_c with max_c * 2^e_c < 2^15 (clamped to keep the epilogue factor normal).
__device__ __forceinline__ int col_exponent(unsigned int maxbits) {
    const float m = __uint_as_float(maxbits);
    if (!(m > 0.0f) || !isfinite(m)) return 0;
    int ex;
    frexpf(m, &ex);  // m = f * 2^ex, f in [0.5, 1): m < 2^ex
    return min(60, max(-60, 15 - ex));
}

// The halves of column c of rows 8g .. 8g + 7 (values v, scaled by 2^ec for f16): V is stacked as B rows c' = c (hi) or
// t + c (lo), element (j, c') of chunk q = j / 64 at q*64*2t + ((j%64)/8 * 2t/8 + c'/8) * 64 + (c'%8) * 8 + j%8.
template <int T, int FMT>
__device__ __forceinline__ void store_split(uint16_t *__restrict__ vs, int64_t g, int c, const float (&vals)[8], int ec) {
    uint32_t hw[4], lw[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint16_t h, l;
        if (FMT == kFmtBF16) {
            const float v = vals[k];
            const __nv_bfloat16 hb = __float2bfloat16_rn(v);
            const __nv_bfloat16 lb = __float2bfloat16_rn(v - __bfloat162float(hb));
            h = *reinterpret_cast<const uint16_t *>(&hb);
            l = *reinterpret_cast<const uint16_t *>(&lb);
        } else {
            const float v = ldexpf(vals[k], ec);
            const __half hh = __float2half_rn(v);
            const __half lh = __float2half_rn(v - __half2float(hh));
            h = *reinterpret_cast<const uint16_t *>(&hh);
            l = *reinterpret_cast<const uint16_t *>(&lh);
        }
        if (k & 1) {
            hw[k >> 1] |= (uint32_t)h << 16;
            lw[k >> 1] |= (uint32_t)l << 16;
        } else {
            hw[k >> 1] = h;
            lw[k >> 1] = l;
        }
    }
    const int64_t q = (8 * g) / tc::kBK;
    const int jj = (int)(8 * g - q * tc::kBK);  // multiple of 8
    const int64_t chunk = q * tc::kBK * 2 * T + (int64_t)(jj >> 3) * (2 * T / 8) * 64 + (c & 7) * 8;
    *reinterpret_cast<uint4 *>(vs + chunk + (int64_t)(c >> 3) * 64) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    *reinterpret_cast<uint4 *>(vs + chunk + (int64_t)((T + c) >> 3) * 64) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

}  // namespace lgp
