// Symmetric split tensor-core product K_y V on tcgen05 (sm_103a), for t in {16, 32}.
//
// K is symmetric, so the upper triangle of 128 x 128 tiles (I <= J) holds every entry. Each
// tile's entries are generated once, split into 16-bit hi/lo halves exactly as in mv_tc.cuh and
// stored to shared memory in the K-major no-swizzle layout; the MMA then reads that one copy
// twice:
//   out_I += K_IJ [V_J]     A = the tile read K-major (M = i, K = j),
//   out_J += K_IJ^T [V_I]   A = the same bytes read MN-major (M = j, K = i), I != J only,
// so each entry costs half the generation work of the row-by-row product. The contraction per
// direction is the same three-product split (K_hi [V_hi V_lo] as one N = 2t MMA, K_lo V_hi as an
// N = t MMA) into float32 accumulators in tensor memory, drained after every tile (K = 128).
//
// Work split (tile_walk.cuh): the nb (nb + 1) / 2 tiles of the triangle, numbered row by row within
// column bands of W tiles, are cut into one contiguous range per CTA and band (persistent grid of
// min(SMs, tiles) CTAs, equal tile counts to within one per band). W keeps a band's column-side
// operands within a share of L2, so that every CTA sweeping the same band reuses them; at the
// sizes where they fit L2 whole (N up to about 157000 at t = 32, 262000 at t = 16) there is one
// band. A CTA's range crosses a few tile rows; within one row segment, out_I accumulates in the
// drain warps' registers and is added to HBM when the segment ends, while out_J is added after
// every tile. Both additions are float32 adds onto out, which the V-splitting kernel initialised to
// sigma^2 V: each drain warp writes its 32-row slab to swizzled shared memory and hands it to the TMA
// unit as a bulk tensor reduce-add (cp.reduce.async.bulk.tensor), so the drain warps release the
// accumulator after their tensor-memory reads alone. (Outputs whose rows are not 16-byte aligned take
// per-thread red.global.add instead.) The order of the additions across CTAs is not fixed, so the
// result can differ between runs in the last bits.
//
// CTA: one per SM, 28 warps at 72 registers, up to 226 KB of shared memory:
//   warps 0-15   generation of the tile's entries into one of two entry buffers;
//   warp 16      producer: lane 0 the V_J ring and the V_I slots, lane 1 the distance operands;
//   warp 17      tensor-memory allocation and the out_I MMAs;  warp 18  the out_J MMAs;
//   warp 19      the Gram MMAs (dot form only);
//   warps 20-27  drain: tensor memory -> registers -> staging slab -> TMA reduce-add, half the columns each.
// Two forms of the squared distance, one kernel template (DOT):
//   difference form (every kernel and D): each generation thread computes 2 rows x 16 columns (two 8-column
//     passes, r^2 from 2D float32 operations on a transposed x_J tile);
//   dot form (RBF, Matern-3/2, Matern-5/2, when the data's spread allows): r^2 = a_i + a_j - 2 u_i . u_j for
//     the box-centred coordinates u, as one 128 x 128 tensor-core Gram tile per tile whose float16 hi/lo operand
//     rows also carry the squared norms a (built once per X by mv_tc.cu), so the tensor core returns -r^2 and an
//     entry costs the kernel value and the split; one row x 32 columns per thread.
//
// What bounds a tile (clock64 stamps of one CTA, N = 100000, t = 32): not a pipe but the latencies between
// the roles. The two entry buffers and the two accumulator buffers each close a loop (generate, multiply,
// release; multiply, drain, release), and a period is half of the longer loop or the slowest role alone. Hence:
//   - the issuers run warp-uniform loops and elect a lane for each pair of MMAs: from a divergent
//     one-lane branch each operand has to be moved to the uniform registers first (microbenchmark with the
//     kernel's N = 64 / N = 32 mix: one issuer 108 -> 55 cycles per MMA, two issuers 108 -> 100 each, which is
//     the tensor pipe's own operand rate of (A + B bytes) / 128 per cycle);
//   - they test all their barriers at once (a test takes ~140 cycles to answer under load, whatever its answer);
//   - out_I and out_J halves of an accumulator are handed over separately, and eight drain warps without
//     barriers among them read half the columns each, with the epilogue factors in registers;
//   - the dot form's generation keeps the next 16 Gram columns in flight while it computes 16, and U_I has two
//     slots so that the next tile row's Gram tiles don't wait for this row's products.
// Together, kernel time at N = 100000, D = 8, t = 32: Matern-5/2 2941 -> 2744 us, RBF 2680 -> 2206 us; N = 20000:
// 151.6 -> 129.1 us; difference form N = 20000, D = 3, t = 16: 176 -> 139 us, N = 50000, D = 8, t = 32 Matern-1/2:
// 1255 -> 1180 us. The generation of the Matern kernels now binds (2420 us alone): its square root and exponential
// take 1536 of ~2800 cycles per tile on the MUFU pipe, the rest is the latency of each warp's chain.
//
// Both instances are launched; a device word (max |u|^2, written by the operand kernel) makes
// exactly one of them work.
// Waits are bounded and abort the CTA as in mv_tc.cuh.
#pragma once

#include <type_traits>

#include "mv_tc.cuh"
#include "tile_walk.cuh"

namespace lgp {
namespace tcs {

using tc::elect_one;
using tc::tmem_free;
using tc::fence_async_smem;
using tc::kDrainBudget;
using tc::kErrWaitAcc;
using tc::kErrWaitEmpty;
using tc::kErrWaitFull;
using tc::kErrWaitReady;
using tc::kGenWarps;
using tc::kMmaWarp;
using tc::kProducerWarp;
using tc::mbar_arrive;
using tc::mbar_arrive_expect_tx;
using tc::mbar_init;
using tc::mbar_wait;
using tc::mbar_wait_all_warp;
using tc::mbar_wait_warp;
using tc::mma_commit;
using tc::mma_ss;
using tc::smem_desc;
using tc::smem_u32;
using tc::tc_fence_after;
using tc::tc_fence_before;
using tc::tma_load_2d;
using tc::tmem_ld;
using tc::tmem_wait_ld;

constexpr int kTile = 128;          // tile rows = tile columns = MMA M
constexpr int kErrWaitVi = 0x100;
constexpr int kErrWaitGram = 0x200;
// Warps 0-15 generate, then the service warps and the drain.
constexpr int kMmaWarpJ = 18;
constexpr int kGramWarp = 19;
constexpr int kTcsDrainWarp0 = 20;  // 8 drain warps
constexpr int kTcsThreads = 896;

// Shared memory: every operand that a copy brings in lives in a ring of its own, so that no copy waits on the
// entry tiles. Two entry buffers [hi | lo], a V_J ring [hi; lo] (released with the entry buffers), a ring of
// the column side's distance operand (dot form: the B-role Gram operand U_J, released by the Gram MMA;
// difference form: the transposed x_J, two [DP][64] boxes, released by the generation), the tile-row slots of
// V_I (and of U_I in the dot form) and the drain's staging tile.
// Tensor memory: two accumulator buffers of [out_I | out_J], 2t columns each (K_lo V_hi accumulates into the
// K_hi V_lo block: both are the small split corrections, summed in float32 by the tensor pipe instead of by
// the drain), then, in the dot form, two 128 x 128 float32 Gram tiles.
template <int T, int DP, bool DOT>
struct TcsLayout {
    static constexpr int kA = kTile * kTile * 2;  // one 16-bit half of the entry tile
    static constexpr int kB = T * kTile * 2;      // one 16-bit half of a 128-row V tile (stacked: 2 kB)
    static constexpr int kKg = 32;                // Gram operand width (16-bit values per row)
    static constexpr int kU = DOT ? kTile * kKg * 2 : kTile * DP * 4;
    static constexpr int kViSlots = DOT ? 1 : 2;  // V_I slots (what fits)
    static constexpr int kK = 0;
    static constexpr int kV = 4 * kA;
    static constexpr int kUr = kV + 4 * kB;
    static constexpr int kVi = kUr + 2 * kU;
    static constexpr int kUi = kVi + kViSlots * 2 * kB;
    static constexpr int kStaging = kUi + (DOT ? 2 * kU : 0);
    static constexpr int kBar = kStaging + kTile * T * 4;
    static constexpr int kBytes = kBar + 1024 + 1024;  // barriers and column factors, alignment slack
    static constexpr int kAccStride = 128;             // accumulator buffer stride
    static constexpr int kAccJ = 64;                   // out_J block inside a buffer
    static constexpr int kGramCol = 256;
    static constexpr int kTmemCols = DOT ? 512 : 256;
};

// Instruction descriptor with A read MN-major (bit 15), B K-major, M = 128, N = NCOLS.
template <int NCOLS, int FMT>
__device__ __forceinline__ uint32_t instr_desc_amn() {
    return tc::instr_desc<NCOLS, FMT>() | (1u << 15);
}

struct TcsArgs {
    const float *Xs;         // prescaled x [Np, DP] row-major (x_I rows for the generation threads)
    float *out;              // [N, ldo], holds sigma^2 V on entry
    const int *skip;
    int *err;
    int64_t N, Np, ldo;
    int nb;                  // Np / 128
    int64_t tiles;           // nb (nb + 1) / 2
    int band;                // column-band width of the tile order, in tiles (tile_walk.cuh)
    float log2s2;            // exponent offset of the entries: log2 s^2 (bf16) or 15 (f16)
    const float *col_scale;  // [T] multiplier per column (f16 mode), or nullptr
    int add_mode;            // kAddTma (tm_out is valid), kAddVec4 or kAddScalar
    long long budget;
    // Distance form. gate (device word, float bits) holds the largest squared norm of the centred
    // prescaled rows; with gate set, the dot-form kernel runs only when *gate <= gate_lim and the
    // difference-form kernel only otherwise (both are launched; the other returns at once).
    const unsigned int *gate;
    float gate_lim;
    int dot;                 // host side: launch the dot-form instance
    const float *arow;       // dot form: a_i, the squared norm of centred row i, [Np]
    const uint8_t *ua;       // dot form: A-role Gram operand, kU bytes per 128-row tile
    const uint8_t *ub;       // dot form: B-role Gram operand
};

// How the drain adds its blocks onto out: TMA bulk tensor reduce (out 16-byte aligned with a row
// stride that is a multiple of 16 bytes), red.global.add.v4.f32 (16-byte aligned rows), or one
// red.global.add.f32 per element.
constexpr int kAddTma = 2, kAddVec4 = 1, kAddScalar = 0;

// Byte offset of 16-byte chunk c of row r in a drain warp's staging slab, in the TMA swizzle pattern of a
// row of W floats (W = 16: 64-byte swizzle, chunk ^= (r / 2) mod 4; W = 8: 32-byte swizzle, chunk ^= (r / 4)
// mod 2), which spreads a warp's rows over all banks.
template <int W>
__device__ __forceinline__ uint32_t staging_off(int r, int c) {
    if constexpr (W == 16) return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
    else return (uint32_t)(r * 32 + ((c ^ ((r >> 2) & 1)) << 4));
}

__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap *map, int c0, int c1, uint32_t src) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(src)
                 : "memory");
}
// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16), completing on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

__device__ __forceinline__ void red_add1(float *p, float a) {
    asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(a) : "memory");
}

// out[0..n) += s[0..n)
template <int NV>
__device__ __forceinline__ void red_row(float *dst, const float (&s)[NV], bool vec4) {
#pragma unroll
    for (int c = 0; c < NV; c += 4) {
        if (vec4) {
            red_add4(dst + c, s[c], s[c + 1], s[c + 2], s[c + 3]);
        } else {
            red_add1(dst + c, s[c]);
            red_add1(dst + c + 1, s[c + 1]);
            red_add1(dst + c + 2, s[c + 2]);
            red_add1(dst + c + 3, s[c + 3]);
        }
    }
}

// Entries from the dot-form Gram value g = -|u_i - u_j|^2 (tensor memory; the operand rows carry both
// squared norms, mv_tc.cu): RBF k = 2^(g + ls2). The Matern forms take |g| as the squared distance:
// near r = 0, where rounding can make g slightly positive, their entries are smooth in r^2
// (k = s^2 (1 - rh^2 / 6 + ...) for Matern-5/2, s^2 (1 - rh^2 / 2 + ...) for Matern-3/2), so |g| and a
// clamp give the same entry up to that rounding; measured, the absolute value makes the Matern-5/2
// product 3% faster than a clamp. (The Matern forms are those of Entry2 in mv_tc.cuh.)
template <int KIND> struct DotEntry2;
template <> struct DotEntry2<LGP_RBF> {
    static __device__ __forceinline__ float2 k(float2 g, float ls2) {
        const float2 arg = __fadd2_rn(g, make_float2(ls2, ls2));
        return make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
    }
};
template <> struct DotEntry2<LGP_MATERN52> {
    // k = e + e (rh + rh^2 / 3), e = 2^(ls2 - rh log2 e), rh = sqrt|g|; rh^2 / 3 taken as -g / 3, which
    // needs no absolute value (a rounding-positive g near r = 0 only perturbs q by that rounding)
    static __device__ __forceinline__ float2 k(float2 g, float ls2) {
        const float2 rh = make_float2(sqrt_approx(fabsf(g.x)), sqrt_approx(fabsf(g.y)));
        const float2 arg = __ffma2_rn(rh, make_float2(-kLog2e, -kLog2e), make_float2(ls2, ls2));
        const float2 e = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
        const float2 q = __ffma2_rn(g, make_float2(-1.0f / 3.0f, -1.0f / 3.0f), rh);
        return __ffma2_rn(e, q, e);
    }
};
template <> struct DotEntry2<LGP_MATERN32> {
    static __device__ __forceinline__ float2 k(float2 g, float ls2) {
        return tc::Entry2<LGP_MATERN32>::k(make_float2(fabsf(g.x), fabsf(g.y)), make_float2(ls2, ls2));
    }
};
// Matern-1/2 has no dot form (its entries are not smooth in r^2 at 0); this stub is never launched.
template <> struct DotEntry2<LGP_MATERN12> {
    static __device__ __forceinline__ float2 k(float2 g, float ls2) { (void)ls2; return g; }
};

// hi/lo split of two entries for the MMA, lo = k - hi (exact in float32), then both packed.
// float16: hi = k with its float32 significand cut to 11 bits by clearing the low bits, so that
//   |lo| < one unit of hi's last place. Cutting instead of rounding costs one bit of lo's range (hi + lo
//   keeps 21 significant bits, against 22) and takes the split off the FMA pipe: two bitwise ANDs and
//   one subtraction per pair. (Measured against the rounding split below: 1% faster on Matern-5/2, 4%
//   on the RBF product, the same product error.) Entries below float16's normal range keep an absolute
//   error below 2^-40 s^2, as with rounding.
// bfloat16, whose 16-bit budget has no bit to spare: hi = k rounded to 8 bits by Veltkamp's splitting
//   (t = 65537 k, hi = t - (t - k)). Entries stay below 2^16 in magnitude, so t cannot overflow.
template <int FMT>
__device__ __forceinline__ void split_pair(float2 k, uint32_t &h, uint32_t &l) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    float2 hi;
    if constexpr (FMT == kFmtF16) {
        hi = make_float2(__uint_as_float(__float_as_uint(k.x) & 0xFFFFE000u),
                         __uint_as_float(__float_as_uint(k.y) & 0xFFFFE000u));
    } else {
        const float2 t = __fmul2_rn(k, make_float2(65537.0f, 65537.0f));
        const float2 u = __ffma2_rn(k, m1, t);  // t - k
        hi = __ffma2_rn(u, m1, t);              // t - (t - k)
    }
    const float2 lo = __ffma2_rn(hi, m1, k);
    h = tc::pack2<FMT>(hi.x, hi.y);
    l = tc::pack2<FMT>(lo.x, lo.y);
}

// The MMA-issue loops over K steps stay rolled (#pragma unroll 1): unrolled issue code competes for the
// instruction cache with the generation warps (measured: the dot-form product is ~25% faster rolled).
// The issuers and the drain poll their barriers without a back-off sleep: a sleeping drain notices its
// accumulator up to 500 cycles late, which lengthens the accumulator loop by as much.
// DOT selects the dot form of the squared distance (D is then 4 or 8, the padded width DP). BANDED
// selects the banded tile order (tile_walk.cuh); the instance without it walks the single-band
// order in fewer registers.
template <int KIND, int D, int T, int FMT, bool DOT = false, bool BANDED = false>
__global__ void __launch_bounds__(kTcsThreads, 1)
    mv_tcs_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_v,
                  const __grid_constant__ CUtensorMap tm_out, const TcsArgs a) {
    constexpr int DP = D <= 4 ? 4 : 8;
    using L = TcsLayout<T, DP, DOT>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBar);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kBar + 384);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::kBar + 392);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform for the compiler
    const int lane = threadIdx.x & 31;
    using Walk = std::conditional_t<BANDED, TileWalk, RowWalk>;
    const TileOrder ord = tile_order(a.nb, BANDED ? a.band : a.nb, (int)blockIdx.x, (int)gridDim.x);
    const int n_it = (int)Walk::count(ord);

    auto bar = [&](int k) { return smem_u32(&bars[k]); };
    auto bar_full = [&](int s) { return bar(s); };             // V_J slot loaded
    auto bar_ready = [&](int s) { return bar(2 + s); };        // entry buffer written (16 generation warps)
    auto bar_empty = [&](int s) { return bar(4 + s); };        // entry buffer and V_J slot released by both issuers
    // each direction's half of accumulator buffer b, by its issuer and by the 8 drain warps
    auto bar_acc_full = [&](int b) { return bar(6 + b); };
    auto bar_acc_empty = [&](int b) { return bar(8 + b); };
    auto bar_accj_full = [&](int b) { return bar(10 + b); };
    auto bar_accj_empty = [&](int b) { return bar(12 + b); };
    auto bar_vi_full = [&](int b) { return bar(14 + b); };     // V_I slot, released by the out_J issuer
    auto bar_vi_empty = [&](int b) { return bar(16 + b); };
    auto bar_u_full = [&](int b) { return bar(18 + b); };      // U_J / x_J slot, released by the Gram issuer or
    auto bar_u_empty = [&](int b) { return bar(20 + b); };     // by the generation warps
    auto bar_ui_full = [&](int b) { return bar(22 + b); };     // dot form: U_I slot
    auto bar_ui_empty = [&](int b) { return bar(24 + b); };
    auto bar_gram_full = [&](int b) { return bar(26 + b); };   // dot form: Gram buffer b written by the tensor pipe
    auto bar_gram_empty = [&](int b) { return bar(28 + b); };  // and read by the generation warps
    const uint32_t bar_fin = bar(30), bar_fin_j = bar(31), bar_fin_g = bar(32);  // the issuers' final commits

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_full(b), 1);
            mbar_init(bar_ready(b), kGenWarps);
            mbar_init(bar_empty(b), 2);
            mbar_init(bar_acc_full(b), 1);
            mbar_init(bar_acc_empty(b), 8);
            mbar_init(bar_accj_full(b), 1);
            mbar_init(bar_accj_empty(b), 8);
            mbar_init(bar_vi_full(b), 1);
            mbar_init(bar_vi_empty(b), 1);
            mbar_init(bar_u_full(b), 1);
            mbar_init(bar_u_empty(b), DOT ? 1 : kGenWarps);
            mbar_init(bar_ui_full(b), 1);
            mbar_init(bar_ui_empty(b), 1);
            mbar_init(bar_gram_full(b), 1);
            mbar_init(bar_gram_empty(b), kGenWarps);
        }
        mbar_init(bar_fin, 1);
        mbar_init(bar_fin_j, 1);
        mbar_init(bar_fin_g, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(L::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // barriers and tensor memory are being set up; from here on the inputs are needed
    chain_wait();
    chain_next();
    const bool idle = (a.skip && *a.skip) || (a.gate && (__uint_as_float(*a.gate) <= a.gate_lim) != DOT);
    // the per-column epilogue factors (float16 halves), read by the drain from shared memory
    float *col_scale = reinterpret_cast<float *>(smem + L::kBar + 512);
    if (a.col_scale && threadIdx.x < T) col_scale[threadIdx.x] = a.col_scale[threadIdx.x];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_acc = *tmem_slot;
    if (idle) {
        if (warp == kMmaWarp) tmem_free<L::kTmemCols>(tmem_acc);
        return;
    }

    Walk w;
    w.init(ord);

    if (warp == kProducerWarp) {
        // ------------------------------------------------------------ producer
        // lane 0: the V_I slots and the V_J ring, released by the contraction; lane 1: the distance operands
        // (U_I slots and U_J ring, released by the Gram MMA; x_J ring, released by the generation), which
        // therefore run ahead of the contraction, also into the next tile row
        if (lane == 0) {
            int last_v[2] = {-1, -1}, last_vi[2] = {-1, -1};
            int sg = -1;
            for (int it = 0; it < n_it; ++it, w.next(ord)) {
                if (w.starts_segment(it)) {
                    ++sg;
                    const int b = sg % L::kViSlots;
                    if (sg >= L::kViSlots && !mbar_wait(bar_vi_empty(b), ((sg / L::kViSlots) - 1) & 1, a.budget, abort_flag,
                                                        a.err, kErrWaitVi, 64))
                        break;
                    const uint32_t dst = smem_u32(smem + L::kVi + b * 2 * L::kB);
                    mbar_arrive_expect_tx(bar_vi_full(b), (uint32_t)(2 * L::kB));
                    tma_load_2d(dst, &tm_v, 0, (2 * w.I) * 2 * T, bar_vi_full(b));
                    tma_load_2d(dst + L::kB, &tm_v, 0, (2 * w.I + 1) * 2 * T, bar_vi_full(b));
                    last_vi[b] = sg;
                }
                const int s = it & 1;
                if (it >= 2 &&
                    !mbar_wait(bar_empty(s), ((it >> 1) - 1) & 1, a.budget, abort_flag, a.err, kErrWaitEmpty, 64))
                    break;
                const uint32_t vdst = smem_u32(smem + L::kV + s * 2 * L::kB);
                mbar_arrive_expect_tx(bar_full(s), (uint32_t)(2 * L::kB));
                tma_load_2d(vdst, &tm_v, 0, (2 * w.J) * 2 * T, bar_full(s));
                tma_load_2d(vdst + L::kB, &tm_v, 0, (2 * w.J + 1) * 2 * T, bar_full(s));
                last_v[s] = it;
            }
            if (*abort_flag) {
                // drain the copies this thread issued
                volatile int no_abort = 0;
                for (int s = 0; s < 2; ++s) {
                    if (last_v[s] >= 0) mbar_wait(bar_full(s), (last_v[s] >> 1) & 1, kDrainBudget, &no_abort, a.err, 0);
                    if (last_vi[s] >= 0)
                        mbar_wait(bar_vi_full(s), (last_vi[s] / L::kViSlots) & 1, kDrainBudget, &no_abort, a.err, 0);
                }
            }
        } else if (lane == 1) {
            int last_u[2] = {-1, -1}, last_ui[2] = {-1, -1};
            int sg = -1;
            for (int it = 0; it < n_it; ++it, w.next(ord)) {
                const int s = it & 1;
                if (DOT && w.starts_segment(it)) {
                    ++sg;
                    const int b = sg & 1;
                    if (sg >= 2 &&
                        !mbar_wait(bar_ui_empty(b), ((sg >> 1) - 1) & 1, a.budget, abort_flag, a.err, kErrWaitVi, 64))
                        break;
                    mbar_arrive_expect_tx(bar_ui_full(b), (uint32_t)L::kU);
                    bulk_load(smem_u32(smem + L::kUi + b * L::kU), a.ua + (int64_t)w.I * L::kU, (uint32_t)L::kU,
                              bar_ui_full(b));
                    last_ui[b] = sg;
                }
                if (it >= 2 &&
                    !mbar_wait(bar_u_empty(s), ((it >> 1) - 1) & 1, a.budget, abort_flag, a.err, kErrWaitEmpty, 64))
                    break;
                const uint32_t udst = smem_u32(smem + L::kUr + s * L::kU);
                mbar_arrive_expect_tx(bar_u_full(s), (uint32_t)L::kU);
                if constexpr (DOT) {
                    bulk_load(udst, a.ub + (int64_t)w.J * L::kU, (uint32_t)L::kU, bar_u_full(s));
                } else {
                    tma_load_2d(udst, &tm_x, w.J * kTile, 0, bar_u_full(s));
                    tma_load_2d(udst + L::kU / 2, &tm_x, w.J * kTile + 64, 0, bar_u_full(s));
                }
                last_u[s] = it;
            }
            if (*abort_flag) {
                volatile int no_abort = 0;
                for (int s = 0; s < 2; ++s) {
                    if (last_u[s] >= 0) mbar_wait(bar_u_full(s), (last_u[s] >> 1) & 1, kDrainBudget, &no_abort, a.err, 0);
                    if (last_ui[s] >= 0) mbar_wait(bar_ui_full(s), (last_ui[s] >> 1) & 1, kDrainBudget, &no_abort, a.err, 0);
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer (out_I)
        const uint32_t idesc2 = tc::instr_desc<2 * T, FMT>();  // K_hi x [V_hi V_lo]
        const uint32_t idesc1 = tc::instr_desc<T, FMT>();      // K_lo x V_hi, onto the K_hi V_lo block
        bool issued = false;
        for (int it = 0; it < n_it; ++it) {
            const int s = it & 1;  // entry buffer, V_J slot and accumulator buffer
            const uint32_t ph = (uint32_t)((it >> 1) & 1);
            // accumulator half free (a fresh barrier's previous phase counts as complete), V_J, entries
            const uint32_t wb[3] = {bar_acc_empty(s), bar_full(s), bar_ready(s)};
            const uint32_t wp[3] = {ph ^ 1u, ph, ph};
            if (!mbar_wait_all_warp<3>(wb, wp, a.budget, abort_flag, a.err, kErrWaitReady)) break;
            tc_fence_after();
            const uint32_t acc_i = tmem_acc + (uint32_t)(s * L::kAccStride);
            const uint32_t ka = smem_u32(smem + L::kK + s * 2 * L::kA);
            const uint32_t b_vj = smem_u32(smem + L::kV + s * 2 * L::kB);
            // A core matrix (row group rg of i, column group kg of j) at (kg * 16 + rg) * 128 bytes.
            // K-major read (K = j): step ks covers kg = 2ks, 2ks+1: start + ks * 4096, K-group stride
            // 2048, row-group stride 128. MN-major read (M = j, K = i): step ks covers rg = 2ks, 2ks+1:
            // start + ks * 256, K-group (rg) stride 128, M-group (kg) stride 2048.
            // B (V tile, 128 rows): core matrix (column group cg of the stacked 2t, row group kg) at
            // (kg * 2t/8 + cg) * 128 bytes.
#pragma unroll 1
            for (int ks = 0; ks < kTile / 16; ++ks) {
                const uint32_t first = ks == 0 ? 0u : 1u;
                const uint64_t dbv = smem_desc(b_vj + ks * 2 * (2 * T) * 16, 2 * T * 16, 128);
                if (elect_one()) {
                    mma_ss(acc_i, smem_desc(ka + ks * 4096, 2048, 128), dbv, idesc2, first);
                    mma_ss(acc_i + T, smem_desc(ka + L::kA + ks * 4096, 2048, 128), dbv, idesc1, 1u);
                }
            }
            if (elect_one()) {
                mma_commit(bar_empty(s));  // V_J slot and entry buffer s (with the out_J issuer)
                mma_commit(bar_acc_full(s));
            }
            issued = true;
        }
        if (issued) {
            // every MMA this warp issued has completed before the CTA frees tensor memory
            if (elect_one()) mma_commit(bar_fin);
            volatile int no_abort = 0;
            mbar_wait(bar_fin, 0, kDrainBudget, &no_abort, a.err, 0);
        }
    } else if (warp < kGenWarps) {
        if constexpr (DOT) {
            // ------------------------------------------------------------ generation, dot form (warps 0-15)
            // Warp w reads tensor-memory lanes 32 (w % 4) .. +31 (its rows i of the tile) and Gram
            // columns 32 (w / 4) .. +31 (j): 32 entries per thread.
            const int q = warp & 3, cb = warp >> 2;
            const int rloc = 32 * q + lane;
            const uint32_t taddr = tmem_acc + ((uint32_t)(32 * q) << 16) + (uint32_t)(L::kGramCol + 32 * cb);
            const float ls2 = a.log2s2;
            // 16 entries of row rloc, columns j = 32 cb + 16 half .. +15, from Gram values g into the entry
            // buffer [hi | lo] at st: each 8 columns are one 16-byte row of core matrix (rg, kg)
            auto generate = [&](const uint32_t (&g)[16], uint8_t *st, int half) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t h[4], l[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float2 dv = make_float2(__uint_as_float(g[8 * u + 2 * v]), __uint_as_float(g[8 * u + 2 * v + 1]));
                        split_pair<FMT>(DotEntry2<KIND>::k(dv, ls2), h[v], l[v]);
                    }
                    const int off = ((4 * cb + 2 * half + u) * 16 + (rloc >> 3)) * 128 + (rloc & 7) * 16;
                    *reinterpret_cast<uint4 *>(st + off) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4 *>(st + L::kA + off) = make_uint4(l[0], l[1], l[2], l[3]);
                }
            };
            // Two 16-column register buffers, one loaded while the other's entries are computed: the load of
            // each half tile is in flight during the half before it.
            uint32_t ga[16], gb[16];
            bool got = n_it > 0 && mbar_wait_warp(bar_gram_full(0), 0, a.budget, abort_flag, a.err, kErrWaitGram);
            if (got) {
                tc_fence_after();
                tmem_ld<16>(taddr, ga);
            }
            for (int it = 0; it < n_it && got; ++it) {
                const int s = it & 1;
                uint8_t *st = smem + L::kK + s * 2 * L::kA;  // entry buffer s: [hi | lo]
                tmem_wait_ld(ga);
                tmem_ld<16>(taddr + (uint32_t)(s * kTile + 16), gb);
                // entry buffer released by both issuers' products of tile it - 2
                if (!mbar_wait_warp(bar_empty(s), (uint32_t)(((it >> 1) - 1) & 1), a.budget, abort_flag, a.err,
                                    kErrWaitEmpty))
                    break;
                generate(ga, st, 0);
                tmem_wait_ld(gb);
                // the Gram buffer may be rewritten once every generation warp holds its part
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_gram_empty(s));
                if (it + 1 < n_it) {
                    got = mbar_wait_warp(bar_gram_full(s ^ 1), (uint32_t)(((it + 1) >> 1) & 1), a.budget, abort_flag, a.err,
                                         kErrWaitGram);
                    if (!got) break;
                    tc_fence_after();
                    tmem_ld<16>(taddr + (uint32_t)((s ^ 1) * kTile), ga);
                }
                generate(gb, st, 1);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_ready(s));
            }
            tmem_wait_ld();
        } else {
            // ------------------------------------------------------------ generation (warps 0-15)
            const int kg0 = warp & 7;    // column groups kg0 and kg0 + 8 of every tile
            const int half = warp >> 3;  // rows 64*half .. 64*half + 63
            const float2 m1 = make_float2(-1.0f, -1.0f);
            const float2 ls2 = make_float2(a.log2s2, a.log2s2);
            const float2 acc_init = tc::Entry2<KIND>::acc0(ls2);
            float2 xi2[2][D];
            for (int it = 0; it < n_it; ++it, w.next(ord)) {
                if (w.starts_segment(it)) {
                    // this thread's 2 rows of tile row I, each coordinate duplicated into both halves of
                    // a float2 (rows < Np because Np % 128 == 0)
    #pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float *xr = a.Xs + ((int64_t)w.I * kTile + 64 * half + 32 * r + lane) * DP;
    #pragma unroll
                        for (int d = 0; d < D; ++d) xi2[r][d] = make_float2(xr[d], xr[d]);
                    }
                }
                // x_J here, and entry buffer s released by both issuers' products of tile it - 2
                const int s = it & 1;
                const uint32_t ph = (uint32_t)((it >> 1) & 1);
                if (!mbar_wait_warp(bar_empty(s), ph ^ 1u, a.budget, abort_flag, a.err, kErrWaitEmpty)) break;
                if (!mbar_wait_warp(bar_u_full(s), ph, a.budget, abort_flag, a.err, kErrWaitFull)) break;
                uint8_t *st = smem + L::kK + s * 2 * L::kA;
                // the two 64-column passes: unrolled when D is small (short bodies), kept as a loop for
                // larger D (measured faster, smaller code)
                constexpr int kPassUnroll = D <= 4 ? 2 : 1;
    #pragma unroll kPassUnroll
                for (int p = 0; p < 2; ++p) {
                    const int kg = kg0 + 8 * p;
                    const float *xs = reinterpret_cast<const float *>(smem + L::kUr + s * L::kU + p * (L::kU / 2));
                    float k[2][8];
    #pragma unroll
                    for (int jh = 0; jh < 2; ++jh) {
                        // columns j = 8*kg + 4*jh + {0,1} (pair 0) and {2,3} (pair 1): the squared
                        // distances of 2 rows x 4 columns accumulate one coordinate at a time
                        float2 r2[2][2];
    #pragma unroll
                        for (int r = 0; r < 2; ++r) r2[r][0] = r2[r][1] = acc_init;
    #pragma unroll
                        for (int d = 0; d < D; ++d) {
                            const float4 q = *reinterpret_cast<const float4 *>(xs + d * 64 + 8 * kg0 + 4 * jh);
                            const float2 xa = make_float2(q.x, q.y), xb = make_float2(q.z, q.w);
    #pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                const float2 da = __ffma2_rn(xa, m1, xi2[r][d]);
                                const float2 db = __ffma2_rn(xb, m1, xi2[r][d]);
                                r2[r][0] = __ffma2_rn(da, da, r2[r][0]);
                                r2[r][1] = __ffma2_rn(db, db, r2[r][1]);
                            }
                        }
    #pragma unroll
                        for (int r = 0; r < 2; ++r) {
    #pragma unroll
                            for (int jp = 0; jp < 2; ++jp) {
                                const float2 kv = tc::Entry2<KIND>::k(r2[r][jp], ls2);
                                k[r][4 * jh + 2 * jp] = kv.x;
                                k[r][4 * jh + 2 * jp + 1] = kv.y;
                            }
                        }
                    }
                    uint8_t *ahi = st;
                    uint8_t *alo = st + L::kA;
    #pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        uint32_t h[4], l[4];
    #pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            h[u] = tc::pack2<FMT>(k[r][2 * u], k[r][2 * u + 1]);
                            float h0, h1;
                            tc::unpack2<FMT>(h[u], h0, h1);
                            const float2 lo =
                                __ffma2_rn(make_float2(h0, h1), m1, make_float2(k[r][2 * u], k[r][2 * u + 1]));
                            l[u] = tc::pack2<FMT>(lo.x, lo.y);
                        }
                        const int rg = 8 * half + 4 * r + (lane >> 3);
                        const int off = (kg * 16 + rg) * 128 + (lane & 7) * 16;
                        *reinterpret_cast<uint4 *>(ahi + off) = make_uint4(h[0], h[1], h[2], h[3]);
                        *reinterpret_cast<uint4 *>(alo + off) = make_uint4(l[0], l[1], l[2], l[3]);
                    }
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(bar_ready(s));
                    mbar_arrive(bar_u_empty(s));
                }
            }
        }
    } else if (warp == kMmaWarpJ) {
        // ------------------------------------------------------------ MMA issuer (out_J)
        const uint32_t idesc2t = instr_desc_amn<2 * T, FMT>();  // K_hi^T x [V_hi V_lo]
        const uint32_t idesc1t = instr_desc_amn<T, FMT>();      // K_lo^T x V_hi
        bool issued = false;
        int sg = -1;
        for (int it = 0; it < n_it; ++it) {
            const bool seg_first = w.starts_segment(it);
            const bool diag = w.J == w.I;
            const int I = w.I;
            w.next(ord);
            const bool seg_last = it == n_it - 1 || w.segment_changed(I);
            if (seg_first) ++sg;
            const int s = it & 1;
            const int vb = sg % L::kViSlots;
            const uint32_t ph = (uint32_t)((it >> 1) & 1);
            // (V_I stays full for the whole tile row, so its phase can be tested at every tile)
            const uint32_t wb[3] = {bar_accj_empty(s), bar_vi_full(vb), bar_ready(s)};
            const uint32_t wp[3] = {ph ^ 1u, (uint32_t)((sg / L::kViSlots) & 1), ph};
            if (!mbar_wait_all_warp<3>(wb, wp, a.budget, abort_flag, a.err, kErrWaitReady)) break;
            tc_fence_after();
            if (!diag) {
                const uint32_t acc_j = tmem_acc + (uint32_t)(s * L::kAccStride + L::kAccJ);
                const uint32_t ka = smem_u32(smem + L::kK + s * 2 * L::kA);
                const uint32_t b_vi = smem_u32(smem + L::kVi + vb * 2 * L::kB);
#pragma unroll 1
                for (int ks = 0; ks < kTile / 16; ++ks) {
                    const uint32_t first = ks == 0 ? 0u : 1u;
                    const uint64_t dbv = smem_desc(b_vi + ks * 2 * (2 * T) * 16, 2 * T * 16, 128);
                    if (elect_one()) {
                        mma_ss(acc_j, smem_desc(ka + ks * 256, 128, 2048), dbv, idesc2t, first);
                        mma_ss(acc_j + T, smem_desc(ka + L::kA + ks * 256, 128, 2048), dbv, idesc1t, 1u);
                    }
                }
            }
            // (a commit with nothing outstanding arrives at once: diagonal tiles)
            if (elect_one()) {
                mma_commit(bar_empty(s));
                mma_commit(bar_accj_full(s));
                if (seg_last) mma_commit(bar_vi_empty(vb));
            }
            issued = true;
        }
        if (issued) {
            if (elect_one()) mma_commit(bar_fin_j);
            volatile int no_abort = 0;
            mbar_wait(bar_fin_j, 0, kDrainBudget, &no_abort, a.err, 0);
        }
    } else if (warp == kGramWarp) {
        if constexpr (DOT) {
            // -------------------------------------------------------- MMA issuer (Gram tiles), dot form
            // Gram tile k into tensor-memory buffer k & 1 (A = the tile-row operand U_I, B = U_J from
            // the ring) as soon as the generation warps have read Gram tile k - 2 out of that buffer.
            {
                const uint32_t idg = tc::instr_desc<kTile, kFmtF16>();  // M = N = 128, float16
                bool issued = false;
                int sg = -1;
                for (int k = 0; k < n_it; ++k) {
                    const bool seg_first = w.starts_segment(k);
                    const int I = w.I;
                    w.next(ord);
                    const bool seg_last = k == n_it - 1 || w.segment_changed(I);
                    if (seg_first) ++sg;
                    const int b = k & 1;  // Gram buffer and U_J ring slot
                    if (k >= 2 &&
                        !mbar_wait_warp(bar_gram_empty(b), ((k >> 1) - 1) & 1, a.budget, abort_flag, a.err, kErrWaitGram))
                        break;
                    if (!mbar_wait_warp(bar_u_full(b), (k >> 1) & 1, a.budget, abort_flag, a.err, kErrWaitFull)) break;
                    if (seg_first && !mbar_wait_warp(bar_ui_full(sg & 1), (sg >> 1) & 1, a.budget, abort_flag, a.err, kErrWaitVi))
                        break;
                    tc_fence_after();
                    const uint32_t ua = smem_u32(smem + L::kUi + (sg & 1) * L::kU);
                    const uint32_t ub = smem_u32(smem + L::kUr + b * L::kU);
                    const uint32_t dg = tmem_acc + (uint32_t)(L::kGramCol + b * kTile);
#pragma unroll
                    for (int ks = 0; ks < L::kKg / 16; ++ks) {
                        if (elect_one())
                            mma_ss(dg, smem_desc(ua + ks * 4096, 2048, 128), smem_desc(ub + ks * 4096, 2048, 128), idg,
                                   ks == 0 ? 0u : 1u);
                    }
                    if (elect_one()) {
                        mma_commit(bar_u_empty(b));
                        mma_commit(bar_gram_full(b));
                        if (seg_last) mma_commit(bar_ui_empty(sg & 1));
                    }
                    issued = true;
                }
                if (issued) {
                    if (elect_one()) mma_commit(bar_fin_g);
                    volatile int no_abort = 0;
                    mbar_wait(bar_fin_g, 0, kDrainBudget, &no_abort, a.err, 0);
                }
            }
        }
    } else {
        // ------------------------------------------------------------ drain (warps 20-27)
        // Each warp moves its own slab of 32 rows x t/2 columns: tensor memory -> registers -> its part of
        // the staging tile -> its own TMA reduce-add, so the drain warps never wait for one another.
        constexpr int TC = T / 2;
        const int quarter = warp & 3;         // tensor-memory lanes 32*quarter .. +31
        const int col0 = TC * ((warp - kTcsDrainWarp0) >> 2);
        const int row = 32 * quarter + lane;  // this thread's row of the 128-row block
        uint8_t *slab = smem + L::kStaging + (warp - kTcsDrainWarp0) * 32 * TC * 4;
        const uint32_t slab_u32 = smem_u32(slab);
        const bool tma = a.add_mode == kAddTma;
        float sum_i[TC];
        // the epilogue factors of this warp's columns (1 for bfloat16 halves): in registers, because the
        // generation's stores keep the shared-memory queue full and a load behind them is slow
        float scale[TC];
#pragma unroll
        for (int c = 0; c < TC; ++c) {
            sum_i[c] = 0.0f;
            scale[c] = a.col_scale ? col_scale[col0 + c] : 1.0f;
        }
        // hands the staged slab to the TMA unit (rows r0 + 32 quarter .. +31 of out; rows >= N are clipped by
        // the tensor map, and a slab that starts at or after row N holds only padding rows)
        auto flush_staged = [&](int r0) {
            fence_async_smem();
            __syncwarp();
            if (lane == 0 && r0 + 32 * quarter < a.N) {
                tma_reduce_add_2d(&tm_out, col0, r0 + 32 * quarter, slab_u32);
                bulk_commit();
            }
        };
        // the slab may be rewritten once this warp's previous reduce has read it
        auto staging_free = [&]() {
            if (lane == 0) bulk_wait_read_all();
            __syncwarp();
        };
        // an accumulator half is free once every drain warp's tensor-memory reads of it are done
        auto release = [&](uint32_t b) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b);
        };
        for (int it = 0; it < n_it; ++it) {
            const bool diag = w.J == w.I;
            const int I = w.I, J = w.J;
            w.next(ord);
            const bool seg_last = it == n_it - 1 || w.segment_changed(I);
            const int s = it & 1;
            const uint32_t ph = (uint32_t)((it >> 1) & 1);
            if (!mbar_wait_warp(bar_acc_full(s), ph, a.budget, abort_flag, a.err, kErrWaitAcc)) break;
            tc_fence_after();
            const uint32_t base = tmem_acc + (uint32_t)(s * L::kAccStride + col0) + ((uint32_t)(32 * quarter) << 16);
            // blocks of each accumulator half: K_hi V_hi at +0, the two corrections at +t; GW columns of each
            // per round (wider rounds cost the registers that the factors take)
            constexpr int GW = 8;
#pragma unroll
            for (int g = 0; g < TC / GW; ++g) {
                uint32_t v0[GW], v1[GW];
                tmem_ld<GW>(base + (uint32_t)(GW * g), v0);
                tmem_ld<GW>(base + (uint32_t)(T + GW * g), v1);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < GW; ++c) sum_i[GW * g + c] += __uint_as_float(v0[c]) + __uint_as_float(v1[c]);
            }
            release(bar_acc_empty(s));
            if (!mbar_wait_warp(bar_accj_full(s), ph, a.budget, abort_flag, a.err, kErrWaitAcc)) break;
            tc_fence_after();
            if (!diag) {
                if (tma) staging_free();
                const int64_t j = (int64_t)J * kTile + row;
#pragma unroll
                for (int g = 0; g < TC / GW; ++g) {
                    uint32_t v0[GW], v1[GW];
                    tmem_ld<GW>(base + L::kAccJ + (uint32_t)(GW * g), v0);
                    tmem_ld<GW>(base + L::kAccJ + (uint32_t)(T + GW * g), v1);
                    tmem_wait_ld();
                    float sj[GW];
#pragma unroll
                    for (int c = 0; c < GW; ++c)
                        sj[c] = (__uint_as_float(v0[c]) + __uint_as_float(v1[c])) * scale[GW * g + c];
                    if (tma) {
#pragma unroll
                        for (int q = 0; q < GW / 4; ++q)
                            *reinterpret_cast<float4 *>(slab + staging_off<TC>(lane, (GW / 4) * g + q)) =
                                make_float4(sj[4 * q], sj[4 * q + 1], sj[4 * q + 2], sj[4 * q + 3]);
                    } else if (j < a.N) {
                        red_row<GW>(a.out + j * a.ldo + col0 + GW * g, sj, a.add_mode == kAddVec4);
                    }
                }
            }
            release(bar_accj_empty(s));
            if (!diag && tma) flush_staged(J * kTile);
            if (seg_last) {
#pragma unroll
                for (int c = 0; c < TC; ++c) sum_i[c] *= scale[c];
                if (tma) {
                    staging_free();
#pragma unroll
                    for (int c = 0; c < TC / 4; ++c)
                        *reinterpret_cast<float4 *>(slab + staging_off<TC>(lane, c)) =
                            make_float4(sum_i[4 * c], sum_i[4 * c + 1], sum_i[4 * c + 2], sum_i[4 * c + 3]);
                    flush_staged(I * kTile);
                } else {
                    const int64_t i = (int64_t)I * kTile + row;
                    if (i < a.N) red_row<TC>(a.out + i * a.ldo + col0, sum_i, a.add_mode == kAddVec4);
                }
#pragma unroll
                for (int c = 0; c < TC; ++c) sum_i[c] = 0.0f;
            }
        }
        // every reduce this warp issued has completed before the CTA exits
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_free<L::kTmemCols>(tmem_acc);
    }
}

}  // namespace tcs
}  // namespace lgp
