"""RBF entries of the float32 products at outputscales far from 1.

The points are two clusters whose squared distance is the sum of eight terms of 3.6e-6 in the kernel's base-2 exponent. Near
|log2 s^2| = 99, where float32 numbers are 7.6e-6 apart, a distance accumulated there loses every one of them: the entries between
the clusters come out 2.0e-5 too large, the sums over both clusters 1.0e-5. Formed by itself and scaled afterwards, an entry
carries the exponential's 2^-22, its rounded distance (8 units of 2^-24 of 2.9e-5) and the rounding of s^2.

Gate on a row sum of N = 300 positive terms: 2^-22 + (70 + 6) 2^-24 = 4.8e-6 (chains of at most 64 additions, then trees and at most 5
partial sums; the scalings and the noise term).
"""
import math
from types import SimpleNamespace

import numpy as np
import pytest

from oracle import gp_oracle as go
import workloads as wl

pytestmark = pytest.mark.gpu

GATE = 2.0 ** -22 + 76 * 2.0 ** -24
N, D = 300, 8


def _problem(log_s2):
    step = np.float32(math.sqrt(3.6e-6 / (0.5 * math.log2(math.e))))
    X = np.repeat((np.arange(N) % 2 == 1).astype(np.float32)[:, None] * step, D, axis=1)
    return SimpleNamespace(X=X, kind=wl.RBF, log_lengthscale=np.zeros(D, np.float32), log_outputscale=float(np.float32(log_s2)),
                           log_noise=float(np.float32(log_s2 + math.log(0.5))))


def _cov(p):
    x = p.X.astype(np.float64)
    r2 = ((x[:, None, :] - x[None, :, :]) ** 2).sum(2)
    return math.exp(p.log_outputscale) * np.exp(-0.5 * r2) + math.exp(p.log_noise) * np.eye(N)


@pytest.mark.parametrize("t", [1, 2, 4, 5, 12, 32])  # symmetric kernel up to 4 columns, row kernel above
@pytest.mark.parametrize("log_s2", [-69.0, 0.0, 69.0])
def test_products(lgp, log_s2, t):
    import torch
    p = _problem(log_s2)
    out = lgp.lgp_kernel_matvec(torch.as_tensor(p.X, device="cuda"), p, torch.ones((N, t), device="cuda"), prec=lgp.LGP_PREC_FP32)
    err = np.abs(out.cpu().numpy().astype(np.float64) / _cov(p).sum(1)[:, None] - 1.0).max()
    print(f"log s2 {log_s2} t={t}: {err:.2e}")
    assert err <= GATE


@pytest.mark.parametrize("t", [1, 8])
@pytest.mark.parametrize("log_s2", [-69.0, 69.0])
def test_batch(lgp, log_s2, t):
    """One CG iteration from ones: x = (b^T b / b^T K b) b, so that the solution shows the product's sum."""
    import torch
    p = _problem(log_s2)
    x = lgp.lgp_batch_cg_solve([torch.as_tensor(p.X, device="cuda")], [p], [torch.ones((N, t), device="cuda")], tol=1e-12,
                               max_iter=1)[0][0]
    err = np.abs(x.cpu().numpy().astype(np.float64) * (_cov(p).sum() / N) - 1.0).max()
    print(f"log s2 {log_s2} t={t}: {err:.2e}")
    assert err <= GATE


@pytest.mark.parametrize("log_s2", [-20.0, -3.0, 5.0, 20.0])
def test_ordinary_points(lgp, log_s2):
    """The product's gate of 1e-5 at every outputscale, and the cross products through the predictive mean at the training points.

    The mean K alpha of targets without structure is small beside |K| |alpha| (1 : 4665 here), so its error is gated by what it is
    made of: the solve's residual of 1e-6 |y|, twice for the recurrence's drift, which K K_y^-1 does not enlarge, and 8 units of
    2^-24 of |K| |alpha| for the rounding of alpha, of the entries and of the sums. (Gated at 1e-4 of itself, the mean misses in the
    row kernel with exact scaling too: 4e-5 to 2e-4, with the iterate at which CG stops.)"""
    import torch
    p = wl.random_problem(700, 6, wl.RBF, seed=5, log_noise=float(np.float32(log_s2 + math.log(0.1))), log_os=float(np.float32(log_s2)))
    hyp = go.hyper_of(p)
    X = torch.as_tensor(p.X, device="cuda")
    for t in (1, 3, 7):
        V = wl.rhs_block(p.N, t, seed=t)
        ref = go.matvec(p.X, V, hyp)
        got = lgp.lgp_kernel_matvec(X, p, torch.as_tensor(V, device="cuda"), prec=lgp.LGP_PREC_FP32).cpu().numpy()
        assert (np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)).max() <= 1e-5
    y = p.y.astype(np.float64)
    Ky = go.noisy_kernel_matrix(p.X, hyp)
    alpha = go.cholesky_solve(Ky, y[:, None])[:, 0]
    ref = y - math.exp(p.log_noise) * alpha
    gate = 2e-6 * np.linalg.norm(y) + 8 * 2.0 ** -24 * np.linalg.norm(Ky @ np.abs(alpha))
    mean = lgp.lgp_predict(X, torch.as_tensor(p.y, device="cuda"), p, X, tol=1e-6, max_iter=2000, want_var=False)[0].cpu().numpy()
    print(f"log s2 {log_s2}: mean off by {np.linalg.norm(mean - ref):.2e}, gate {gate:.2e}, mean {np.linalg.norm(ref):.2e}")
    assert gate < 0.01 * np.linalg.norm(ref) and np.linalg.norm(mean - ref) <= gate
