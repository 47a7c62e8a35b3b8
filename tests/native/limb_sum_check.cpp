// csrc/limb_sum.cuh on the host: the sum of n pairs (hi, lo) as a block of the CG kernels forms it.
#include "limb_sum.cuh"

extern "C" double limb_block_sum(const float *hi, const float *lo, int n) {
    uint32_t mx = 0;
    for (int i = 0; i < n; ++i) {
        const uint32_t a = lgp::magnitude_bits(hi[i]), b = lgp::magnitude_bits(lo[i]);
        mx = a > mx ? a : mx;
        mx = b > mx ? b : mx;
    }
    const float scale = lgp::limb_scale(mx);
    int l[3] = {0, 0, 0};
    for (int i = 0; i < n; ++i) {
        int p[3] = {0, 0, 0};
        lgp::add_limbs(hi[i], scale, p);
        lgp::add_limbs(lo[i], scale, p);
        for (int j = 0; j < 3; ++j) {
            if (mx < 0x7F800000u && (p[j] > 1 << 20 || p[j] < -(1 << 20))) return -1.0;  // two parts of at most 2^19
            l[j] = (int)((unsigned)l[j] + (unsigned)p[j]);
        }
    }
    return lgp::limb_total(l[0], l[1], l[2], mx);
}
