"""The CG step's launches (product tail, alpha, beta, the update and split of p) at the sizes where their loops end.

Gate: componentwise backward error |B - K_y X| / (K_y |X| + |B|) <= 1e-5, the gate of the other split and float32 solves:
CG stops at a relative residual of 1e-6, and the float32 recurrences add a few units of 2^-24 per iteration to it.
A column of zeros takes no iteration and stays zero; a column that is an exact multiple of another one needs as many
iterations (both run through every launch beside columns that have stopped).
"""
import math

import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


def _solve(lgp, N, t, prec, ctx, rank=0):
    import torch
    p = wl.random_problem(N, 3, wl.MATERN52, seed=N + t, log_noise=math.log(0.5), log_os=0.0)
    B = wl.rhs_block(N, t, seed=t)
    if t > 2:
        B[:, 1] = 0.0
        B[:, t - 1] = 2.0 ** -20 * B[:, 0]
    x, iters, rel, status = lgp.lgp_cg_solve(torch.as_tensor(p.X, device="cuda"), p, torch.as_tensor(B, device="cuda"), tol=1e-6,
                                             max_iter=4000, prec=prec, ctx=ctx, precond_rank=rank)
    assert status == lgp.LGP_OK and (rel <= 1e-6).all()
    x = x.cpu().numpy().astype(np.float64)
    Ky = go.noisy_kernel_matrix(p.X, go.hyper_of(p))
    denom = Ky @ np.abs(x) + np.abs(B)
    berr = np.abs(B - Ky @ x) / np.where(denom > 0, denom, 1.0)
    print(f"N={N} t={t} prec={prec}: iterations {iters.min()}..{iters.max()}, backward error {berr.max():.2e}")
    assert berr.max() <= 1e-5
    if t > 2:
        assert iters[1] == 0 and np.all(x[:, 1] == 0.0)
    return iters


@pytest.mark.parametrize("t", [1, 2, 3, 4, 5, 8, 13, 33, 64])
@pytest.mark.parametrize("N", [1, 2, 63, 257, 1030, 4099])
def test_float32_step(lgp, N, t):
    iters = _solve(lgp, N, t, lgp.LGP_PREC_FP32, None)
    if t > 2:  # an exact power of two: the same recurrence
        assert iters[t - 1] == iters[0]


@pytest.mark.parametrize("symmetric", ["1", "0"], ids=["symmetric", "row"])
@pytest.mark.parametrize("prec", ["f16", "bf16"])
@pytest.mark.parametrize("t", [16, 32])
@pytest.mark.parametrize("N", [9, 257, 1030, 3001])
def test_split_step(lgp, monkeypatch, N, t, prec, symmetric):
    monkeypatch.setenv("LGP_TC_SYMMETRIC", symmetric)
    ctx = lgp.Context(0)
    try:
        _solve(lgp, N, t, lgp.LGP_PREC_SPLIT_F16 if prec == "f16" else lgp.LGP_PREC_SPLIT_BF16, ctx)
    finally:
        ctx.close()


@pytest.mark.parametrize("t", [1, 5, 16])
def test_preconditioned_step(lgp, t):
    _solve(lgp, 1030, t, lgp.LGP_PREC_AUTO, None, rank=8)
