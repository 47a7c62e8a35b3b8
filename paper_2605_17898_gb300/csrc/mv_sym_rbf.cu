#include "mv_sym.cuh"

namespace lgp {
cudaError_t mv_sym_dispatch_rbf(int D, int TT, const SymArgs &a, cudaStream_t st) {
    return dispatch_mv_sym<LGP_RBF>(D, TT, a, st);
}
}  // namespace lgp
