"""The symmetric float32 product's large blocks and the sizes where it ends: 512 rows with more than 48 KB of shared memory,
1024 rows, and the row kernel where the partial sums would pass 256 MiB.

Sampled rows against the FP64 oracle at the product's gate of 1e-5, and bitwise-equal repeats, as for the smaller blocks. The
product of a large problem has 2^31 and more entries, so the rows at its ends and a few between are sampled.
"""
import numpy as np
import pytest

import workloads as wl
from test_symmetric_fp32_gpu import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,t,D,kind", [
    (37001, 3, 4, wl.RBF), (37001, 4, 4, wl.MATERN52), (37001, 4, 8, wl.RBF),   # 512 rows, 51 and 59 KB
    (94999, 4, 7, wl.MATERN32), (93003, 3, 2, wl.RBF),                            # 1024 rows, four padded columns
    (190001, 1, 8, wl.MATERN52), (140003, 2, 8, wl.MATERN12),                     # 1024 rows, one and two columns
    (100000, 4, 8, wl.MATERN52), (150001, 3, 8, wl.RBF),                          # row kernel: 1024 rows need a whole SM
    (270001, 1, 3, wl.RBF),                                                      # row kernel: beyond the partial sums' bound
])
def test_large_blocks(lgp, N, t, D, kind):
    p = wl.random_problem(N, D, kind, seed=N)
    rows = np.unique(np.concatenate([np.arange(8), np.arange(N - 8, N), np.random.default_rng(2).integers(0, N, 40)]))
    _check(lgp, p, wl.rhs_block(N, t, seed=t), rows)
