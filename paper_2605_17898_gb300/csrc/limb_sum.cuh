// Sums of up to 2048 float32 values as three 32-bit integers in fixed point: plain arithmetic shared by the CG kernels
// (cg_reduce.cuh) and its host check.
//
// With e such that every |v| < 2^e, v is written as l0 2^(e-19) + l1 2^(e-39) + l2 2^(e-59), |l| <= 2^19 each, rounded once in
// the last place (half of 2^(e-59), or exactly for e <= -90, where that is below the smallest float). 2048 of them add up
// in 32 bits without overflow and without rounding, in any order, and the three sums make one float64. So the sum is as
// exact as a float64 tree's and, unlike a sum of float32 pairs, neither rounds at 2^-48 nor overflows at 3.4e38.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define LGP_HD __host__ __device__ __forceinline__
#else
#define LGP_HD inline
#endif

namespace lgp {

template <class To, class From> LGP_HD To bits_as(From v) {
    static_assert(sizeof(To) == sizeof(From), "same size");
    To r;
    memcpy(&r, &v, sizeof r);
    return r;
}

// Magnitude of v as an integer that orders like |v| (NaN above infinity).
LGP_HD uint32_t magnitude_bits(float v) { return bits_as<uint32_t>(v) & 0x7FFFFFFFu; }

// Exponent field that stands for e = field - 126, from the largest magnitude; at least 18, so that 2^(19-e) is a float.
LGP_HD uint32_t limb_field(uint32_t max_bits) { return max_bits >> 23 > 18u ? max_bits >> 23 : 18u; }
LGP_HD float limb_scale(uint32_t max_bits) { return bits_as<float>((272u - limb_field(max_bits)) << 23); }  // 2^(19-e)

// l += the three parts of v. Adding 1.5 2^23 rounds a value below 2^22 to an integer, in the low bits of the sum.
LGP_HD void add_limbs(float v, float scale, int (&l)[3]) {
    const float magic = 12582912.0f;
    float a = v * scale;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
        const float r = a + magic;
        l[k] += bits_as<int32_t>(r) - 0x4B400000;
        a = (a - (r - magic)) * 1048576.0f;
    }
}

// The sum of the values whose parts add up to l: float64, infinity or NaN if a value was.
LGP_HD double limb_total(int l0, int l1, int l2, uint32_t max_bits) {
    if (max_bits >= 0x7F800000u) return (double)bits_as<float>(max_bits);
    const double s = ((double)l0 * 1048576.0 + (double)l1) * 1048576.0 + (double)l2;
    return s * bits_as<double>((uint64_t)(limb_field(max_bits) + 1023u - 185u) << 52);  // 2^(e-59)
}

}  // namespace lgp
