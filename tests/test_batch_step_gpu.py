"""The batch's CG step (one cluster or CTA per problem) at the sizes where its loops end: one row, a ragged last block of
four values, one CTA's limit, several passes per CTA; column counts that are a power of two or not.

Gate: componentwise backward error |B - K_y X| / (K_y |X| + |B|) <= 1e-5, the gate of the other float32 solves: CG
stops at a relative residual of 1e-6, and the float32 recurrences add a few units of 2^-24 per iteration to it. A column
of zeros takes no iteration and stays zero, beside a column that is an exact power of two of another and needs exactly as
many iterations; a problem without an active column ends no other problem; max_iter stops every problem on its own count.
"""
import math

import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("t", [1, 2, 3, 4, 5, 8, 13, 16])
@pytest.mark.parametrize("sizes", [[1, 2, 3, 63], [1, 66, 257, 1021], [130, 3001, 7]], ids=["one_cta", "mixed", "cluster"])
def test_batch_step(lgp, sizes, t):
    probs = [wl.random_problem(n, 1 + n % 3, wl.MATERN52, seed=n + t, log_noise=math.log(0.5), log_os=0.0) for n in sizes]
    Bs = [wl.rhs_block(n, t, seed=t + n) for n in sizes]
    Bs[-1][:] = 0.0
    if t > 2:
        for B in Bs:
            B[:, 1] = 0.0
            B[:, t - 1] = 2.0 ** -20 * B[:, 0]
    X = [_dev(p.X) for p in probs]
    sols, iters, rel, s = lgp.lgp_batch_cg_solve(X, probs, [_dev(B) for B in Bs], tol=1e-6, max_iter=4000,
                                                 prec=lgp.LGP_PREC_FP32)
    assert s == lgp.LGP_OK and (rel <= 1e-6).all()
    assert (iters[-1] == 0).all() and not sols[-1].cpu().numpy().any()
    for g, (p, B) in enumerate(zip(probs, Bs)):
        x = sols[g].cpu().numpy().astype(np.float64)
        Ky = go.noisy_kernel_matrix(p.X, go.hyper_of(p))
        denom = Ky @ np.abs(x) + np.abs(B)
        berr = np.abs(B - Ky @ x) / np.where(denom > 0, denom, 1.0)
        assert berr.max() <= 1e-5, (p.N, berr.max())
        if t > 2:
            assert iters[g, 1] == 0 and iters[g, t - 1] == iters[g, 0]
    if max(iters.flat) > 2:
        _, few, _, s = lgp.lgp_batch_cg_solve(X, probs, [_dev(B) for B in Bs], tol=1e-6, max_iter=2, prec=lgp.LGP_PREC_FP32)
        assert s == lgp.LGP_WARN_NOT_CONVERGED and (few == np.minimum(iters, 2)).all()
