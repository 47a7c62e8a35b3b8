"""The CG step of a cluster of 16 CTAs (65537 to 262144 vector elements) at the ends of its range, against the gates of the
other steps (test_cg_step_gpu): componentwise backward error <= 1e-5 at a relative residual of 1e-6, zero columns untouched."""
import pytest

from test_cg_step_gpu import _solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,t,prec", [(2049, 32, "f32"), (4096, 64, "f32"), (4097, 16, "f32"), (2049, 32, "f16"), (2061, 32, "bf16"),
                                      (5000, 16, "f16"), (8190, 32, "f16")])
def test_wide_step(lgp, N, t, prec):
    modes = {"f32": lgp.LGP_PREC_FP32, "f16": lgp.LGP_PREC_SPLIT_F16, "bf16": lgp.LGP_PREC_SPLIT_BF16}
    iters = _solve(lgp, N, t, modes[prec], None)
    if prec == "f32":  # an exact power of two: the same recurrence
        assert iters[t - 1] == iters[0]
