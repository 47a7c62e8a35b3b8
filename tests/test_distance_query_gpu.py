"""lgp_tc_distance_form keeps answering for the last symmetric product when a row-kernel product of the same size follows."""
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("repeat", [1, 3])
@pytest.mark.parametrize("t", [16, 32])
def test_row_product_leaves_the_answer(lgp, monkeypatch, t, repeat):
    import torch
    import numpy as np

    def product(p):
        V = wl.rhs_block(p.N, t, seed=t)
        out = lgp.lgp_kernel_matvec(torch.as_tensor(p.X, device="cuda"), p, torch.as_tensor(V, device="cuda"), ctx=ctx).cpu().numpy()
        ref = go.matvec(p.X, V, go.hyper_of(p))
        assert (np.linalg.norm(out - ref, axis=0) / np.linalg.norm(ref, axis=0)).max() <= 1e-5

    ctx = lgp.Context(0)
    try:
        first, second = wl.random_problem(2000, 6, wl.RBF, seed=1), wl.random_problem(2000, 5, wl.MATERN52, seed=2)
        monkeypatch.setenv("LGP_TC_SYMMETRIC", "1")
        for _ in range(repeat):
            product(first)
        form, norm = ctx.tc_distance_form()
        assert form == lgp.LGP_DIST_DOT and norm > 0.0
        monkeypatch.setenv("LGP_TC_SYMMETRIC", "0")
        for _ in range(repeat):
            product(second)
        assert ctx.tc_kernel_choice(2000, 5, wl.MATERN52, t) == lgp.LGP_TC_ROW
        assert ctx.tc_distance_form() == (form, norm)
        product(first)
        assert ctx.tc_distance_form() == (form, norm)
    finally:
        ctx.close()
