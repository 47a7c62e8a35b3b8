"""Every way to run the CG step, at sizes that reach it, against the gates of the other steps (test_cg_step_gpu)."""
import pytest

from test_cg_step_gpu import _solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,t,prec,ctas", [
    (500, 1, "f32", 1), (900, 4, "f32", 8), (4096, 1, "f32", 8), (300, 64, "f32", 8),
    (1025, 64, "f32", 16), (1400, 64, "f32", 16), (2049, 32, "f32", 16), (3001, 16, "f32", 16),   # Kp stored by the step
    (2049, 32, "f16", 16), (5000, 16, "bf16", 16),                                                # p split by the step
    (8000, 8, "f32", 0), (1030, 5, "f32", 0), (9001, 32, "f16", 0),
])
def test_step_reached(lgp, N, t, prec, ctas):
    modes = {"f32": lgp.LGP_PREC_FP32, "f16": lgp.LGP_PREC_SPLIT_F16, "bf16": lgp.LGP_PREC_SPLIT_BF16}
    ctx = lgp.Context(0)
    try:
        assert ctx.cg_step_ctas() == -1
        iters = _solve(lgp, N, t, modes[prec], ctx)
        assert ctx.cg_step_ctas() == ctas
        if prec == "f32" and t > 2:  # an exact power of two: the same recurrence
            assert iters[t - 1] == iters[0]
    finally:
        ctx.close()
