// Instantiation of the split tensor-core product for one 16-bit format (included once per format).
#pragma once

#include "mv_tc.cuh"

namespace lgp {
namespace tc {

template <int KIND, int D, int T, int FMT>
cudaError_t launch_tc_inst(dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv,
                           const TcArgs &a, cudaStream_t st) {
    constexpr int DP = D <= 4 ? 4 : 8;
    constexpr int bytes = TcLayout<T, DP, (D <= 4)>::kBytes;
    static DeviceOnce configured;
    const cudaError_t e = allow_shared(configured, mv_tc_kernel<KIND, D, T, FMT>, bytes);
    if (e != cudaSuccess) return e;
    return launch_chained(mv_tc_kernel<KIND, D, T, FMT>, grid, kThreads, bytes, st, mx, mv, a);
}

template <int KIND, int T, int FMT>
cudaError_t dispatch_d(int D, dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv,
                       const TcArgs &a, cudaStream_t st) {
    switch (D) {
        case 1: return launch_tc_inst<KIND, 1, T, FMT>(grid, mx, mv, a, st);
        case 2: return launch_tc_inst<KIND, 2, T, FMT>(grid, mx, mv, a, st);
        case 3: return launch_tc_inst<KIND, 3, T, FMT>(grid, mx, mv, a, st);
        case 4: return launch_tc_inst<KIND, 4, T, FMT>(grid, mx, mv, a, st);
        case 5: return launch_tc_inst<KIND, 5, T, FMT>(grid, mx, mv, a, st);
        case 6: return launch_tc_inst<KIND, 6, T, FMT>(grid, mx, mv, a, st);
        case 7: return launch_tc_inst<KIND, 7, T, FMT>(grid, mx, mv, a, st);
        case 8: return launch_tc_inst<KIND, 8, T, FMT>(grid, mx, mv, a, st);
    }
    return cudaErrorInvalidValue;
}

// One (format, kind) pair: every D and T. Instantiated in its own translation unit
// (mv_tc_<fmt>_<kind>.cu) so that the instantiations compile in parallel.
template <int FMT, int KIND>
cudaError_t dispatch_kind(int D, int T, dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv, const TcArgs &a,
                          cudaStream_t st) {
    return T == 16 ? dispatch_d<KIND, 16, FMT>(D, grid, mx, mv, a, st) : dispatch_d<KIND, 32, FMT>(D, grid, mx, mv, a, st);
}

#define LGP_TC_KIND_DECL(FMT, KIND)                                                                               \
    extern template cudaError_t dispatch_kind<FMT, KIND>(int, int, dim3, const CUtensorMap &, const CUtensorMap &, \
                                                         const TcArgs &, cudaStream_t);
LGP_TC_KIND_DECL(kFmtBF16, LGP_RBF)
LGP_TC_KIND_DECL(kFmtBF16, LGP_MATERN52)
LGP_TC_KIND_DECL(kFmtBF16, LGP_MATERN12)
LGP_TC_KIND_DECL(kFmtBF16, LGP_MATERN32)
LGP_TC_KIND_DECL(kFmtF16, LGP_RBF)
LGP_TC_KIND_DECL(kFmtF16, LGP_MATERN52)
LGP_TC_KIND_DECL(kFmtF16, LGP_MATERN12)
LGP_TC_KIND_DECL(kFmtF16, LGP_MATERN32)
#undef LGP_TC_KIND_DECL

template <int FMT>
cudaError_t dispatch_fmt(int kind, int D, int T, dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv,
                         const TcArgs &a, cudaStream_t st) {
    switch (kind) {
        case LGP_RBF: return dispatch_kind<FMT, LGP_RBF>(D, T, grid, mx, mv, a, st);
        case LGP_MATERN52: return dispatch_kind<FMT, LGP_MATERN52>(D, T, grid, mx, mv, a, st);
        case LGP_MATERN12: return dispatch_kind<FMT, LGP_MATERN12>(D, T, grid, mx, mv, a, st);
        case LGP_MATERN32: return dispatch_kind<FMT, LGP_MATERN32>(D, T, grid, mx, mv, a, st);
    }
    return cudaErrorInvalidValue;
}

inline cudaError_t dispatch_bf16(int kind, int D, int T, dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv,
                                 const TcArgs &a, cudaStream_t st) {
    return dispatch_fmt<kFmtBF16>(kind, D, T, grid, mx, mv, a, st);
}
inline cudaError_t dispatch_f16(int kind, int D, int T, dim3 grid, const CUtensorMap &mx, const CUtensorMap &mv,
                                const TcArgs &a, cudaStream_t st) {
    return dispatch_fmt<kFmtF16>(kind, D, T, grid, mx, mv, a, st);
}

}  // namespace tc
}  // namespace lgp
