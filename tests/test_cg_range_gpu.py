"""CG on right-hand sides near the end of float32's range: the recurrence is homogeneous, and 2^60 B needs exactly the iterations of B.

A term p Kp or r r stays below 3e37, and so does a thread's sum; a block's sum of 1000 and more is beyond 3.4e38 and has to be
carried in more range than float32's. Every operation on the scaled vectors is the unscaled one times a power of two, so that the
solutions agree bit for bit where the product sums in a fixed order.
"""
import math

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

SCALE = np.float32(2.0 ** 60)


def _data(N, t):
    p = wl.random_problem(N, 3, wl.MATERN32, seed=N + t, lo=0.01, hi=0.02, log_os=math.log(0.1), log_noise=0.0)
    B = np.where(np.random.default_rng(t).random((N, t)) < 0.5, -1.0, 1.0).astype(np.float32)
    return p, B


@pytest.mark.parametrize("N,t", [(3000, 1), (8000, 1), (4099, 2), (2500, 3), (30000, 2), (60001, 1)])
def test_solve(lgp, N, t):
    import torch
    p, B = _data(N, t)
    X = torch.as_tensor(p.X, device="cuda")
    a = lgp.lgp_cg_solve(X, p, torch.as_tensor(B, device="cuda"), tol=1e-5, max_iter=200)
    b = lgp.lgp_cg_solve(X, p, torch.as_tensor(B * SCALE, device="cuda"), tol=1e-5, max_iter=200)
    assert a[3] == b[3] == lgp.LGP_OK and (a[1] == b[1]).all() and a[1].min() >= 2
    assert torch.equal(a[0] * float(SCALE), b[0])


@pytest.mark.parametrize("t", [1, 3])
def test_batch(lgp, t):
    import torch
    data = [_data(N, t) for N in (4000, 1200, 3100)]
    X = [torch.as_tensor(p.X, device="cuda") for p, _ in data]
    hyp = [p for p, _ in data]
    a = lgp.lgp_batch_cg_solve(X, hyp, [torch.as_tensor(B, device="cuda") for _, B in data], tol=1e-5, max_iter=200, prec=lgp.LGP_PREC_FP32)
    b = lgp.lgp_batch_cg_solve(X, hyp, [torch.as_tensor(B * SCALE, device="cuda") for _, B in data], tol=1e-5, max_iter=200,
                               prec=lgp.LGP_PREC_FP32)
    assert a[3] == b[3] == lgp.LGP_OK and (a[1] == b[1]).all()
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x * float(SCALE), y)
