"""The float32 row kernel (t > 4, and the cross products of prediction) at the edges of its tiles, rows and column groups.

Gate: column relative error <= 1e-5, the product's gate.
"""
import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu


def _err(lgp, p, t):
    import torch
    V = wl.rhs_block(p.N, t, seed=t)
    out = lgp.lgp_kernel_matvec(torch.as_tensor(p.X, device="cuda"), p, torch.as_tensor(V, device="cuda"),
                                prec=lgp.LGP_PREC_FP32).cpu().numpy()
    ref = go.matvec(p.X, V, go.hyper_of(p))
    return (np.linalg.norm(out - ref, axis=0) / np.linalg.norm(ref, axis=0)).max()


@pytest.mark.parametrize("N", [1, 63, 64, 65, 127, 129, 255, 257, 1100])
@pytest.mark.parametrize("t", [5, 8, 9, 16, 17, 32, 40, 64])
def test_edges(lgp, N, t):
    assert _err(lgp, wl.random_problem(N, 3, wl.MATERN52, seed=N + t), t) <= 1e-5


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", wl.KINDS)
@pytest.mark.parametrize("t", [6, 16, 31])
def test_every_instance(lgp, kind, D, t):
    assert _err(lgp, wl.random_problem(500, D, kind, seed=10 * D + kind), t) <= 1e-5


@pytest.mark.parametrize("t", [1, 3, 8, 16])
def test_batch_items(lgp, t):
    """The batched product's tiles: problems around one and two row blocks of 256, column splits included."""
    import math
    import torch
    probs = [wl.random_problem(N, D, kind, seed=N, log_noise=math.log(0.5), log_os=0.0)
             for N, D, kind in [(1, 1, wl.RBF), (65, 2, wl.MATERN12), (255, 5, wl.MATERN32), (257, 8, wl.MATERN52), (600, 3, wl.RBF)]]
    dev = lambda a: torch.as_tensor(a, device="cuda")
    Bs = [wl.rhs_block(p.N, t, seed=p.N) for p in probs]
    sols, iters, rel, status = lgp.lgp_batch_cg_solve([dev(p.X) for p in probs], probs, [dev(B) for B in Bs], tol=1e-6,
                                                      max_iter=2000, prec=lgp.LGP_PREC_FP32)
    assert status == lgp.LGP_OK and (rel <= 1e-6).all()
    for p, B, x in zip(probs, Bs, sols):
        x = x.cpu().numpy().astype(np.float64)
        Ky = go.noisy_kernel_matrix(p.X, go.hyper_of(p))
        berr = np.abs(B - Ky @ x) / (Ky @ np.abs(x) + np.abs(B))
        assert berr.max() <= 1e-5, (p.N, berr.max())  # the componentwise gate of the other solves
