"""The symmetric float32 product (t <= 4) at the edges of its blocks, sweeps and column counts.

Gate: column relative error <= 1e-5, the product's gate (float32 entries carry about 3e-7, and the sums are trees).
"""
import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


def _check(lgp, p, V, rows=None):
    import torch
    out = lgp.lgp_kernel_matvec(torch.as_tensor(p.X, device="cuda"), p, torch.as_tensor(V, device="cuda"), prec=lgp.LGP_PREC_FP32)
    out2 = lgp.lgp_kernel_matvec(torch.as_tensor(p.X, device="cuda"), p, torch.as_tensor(V, device="cuda"), prec=lgp.LGP_PREC_FP32)
    assert torch.equal(out, out2), "the float32 product is reproducible bit for bit"
    out = out.cpu().numpy()
    hyp = go.hyper_of(p)
    ref = go.matvec(p.X, V, hyp) if rows is None else go.matvec_rows(p.X, V, hyp, rows)
    got = out if rows is None else out[rows]
    err = np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)
    print(f"N={p.N} D={p.D} kind={p.kind} t={V.shape[1]}: {err.max():.2e}")
    assert err.max() <= 1e-5


# one block of 64; two with a last row or column alone; the switch to blocks of 128; a ragged size in between
@pytest.mark.parametrize("N", [1, 2, 64, 65, 129, 1027, 4991, 5057])
@pytest.mark.parametrize("t", [1, 2, 3, 4])
def test_blocks(lgp, N, t):
    p = wl.random_problem(N, 3, wl.MATERN52, seed=N)
    _check(lgp, p, wl.rhs_block(N, t, seed=t))


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", wl.KINDS)
@pytest.mark.parametrize("t", [1, 2, 4])
def test_every_instance(lgp, kind, D, t):
    p = wl.random_problem(700, D, kind, seed=10 * D + kind)
    _check(lgp, p, wl.rhs_block(p.N, t, seed=t))


# blocks of 256 and of 512 rows
@pytest.mark.parametrize("N,t", [(17003, 1), (17003, 4), (37001, 1), (37001, 2)])
def test_large_blocks(lgp, N, t):
    p = wl.random_problem(N, 4, wl.RBF, seed=N)
    rows = np.unique(np.concatenate([np.arange(40), np.arange(N - 40, N), np.random.default_rng(1).integers(0, N, 200)]))
    _check(lgp, p, wl.rhs_block(N, t, seed=t), rows)
