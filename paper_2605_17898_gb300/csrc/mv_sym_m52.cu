#include "mv_sym.cuh"

namespace lgp {
cudaError_t mv_sym_dispatch_m52(int D, int TT, const SymArgs &a, cudaStream_t st) {
    return dispatch_mv_sym<LGP_MATERN52>(D, TT, a, st);
}
}  // namespace lgp
