"""The two passes over a tensor-core product's inputs (maxima, transposed X and box; halves of V and distance operands).

They collect maxima in words that the product's first kernel clears: each product here follows one with much larger values of V
and a much larger box of X on the same context, so that a stale word would cost the halves their low bits or the dot form its
gate. Sizes: one row, the edges of a 256-row block, several blocks with a ragged end. Gate: 1e-5 column error, that of the
other float16 products.
"""
import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("symmetric", ["0", "1"], ids=["row", "symmetric"])
@pytest.mark.parametrize("t", [5, 16, 32])
@pytest.mark.parametrize("N,D", [(1, 8), (255, 3), (257, 8), (1025, 4), (2300, 7)])
def test_products_one_after_another(lgp, monkeypatch, N, D, t, symmetric):
    import torch
    monkeypatch.setenv("LGP_TC_SYMMETRIC", symmetric)
    p = wl.random_problem(N, D, wl.RBF, seed=N + t)
    V = wl.rhs_block(N, t, seed=t)
    ref = go.matvec(p.X, V, go.hyper_of(p)).reshape(N, -1)
    X, Vd = torch.as_tensor(p.X, device="cuda"), torch.as_tensor(V, device="cuda")
    ctx = lgp.Context(0)
    try:
        for scale, spread in ((2.0 ** 30, 1.0), (2.0 ** -30, 1.0), (2.0 ** 30, 100.0), (1.0, 1.0)):
            out = lgp.lgp_kernel_matvec(spread * X, p, scale * Vd, prec=lgp.LGP_PREC_SPLIT_F16, ctx=ctx)
            if spread == 1.0:
                got = out.cpu().numpy().astype(np.float64) / scale
                err = np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)
                assert err.max() <= 1e-5, (scale, err.max())
    finally:
        ctx.close()
