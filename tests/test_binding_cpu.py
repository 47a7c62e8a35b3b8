"""The binding's packed hyperparameters hold the same values as the array form, for every way a caller can give them."""
import ctypes

import numpy as np
import pytest

import paper_2605_17898_gb300 as lgp

LS = np.array([-1.25, 0.1, 3.0, -0.7, 1e-30, 2.5, -4.0, 0.3])


def _forms(D):
    import torch
    v = LS[:D]
    ro = v.astype(np.float32)
    ro.setflags(write=False)
    return {"float64": v, "float32": v.astype(np.float32), "read-only": ro, "strided": np.repeat(v, 2)[::2], "list": list(v),
            "tensor": torch.tensor(v), "column": v[:, None]}


@pytest.mark.parametrize("D", [1, 3, 8])
@pytest.mark.parametrize("form", ["float64", "float32", "read-only", "strided", "list", "tensor", "column"])
def test_packed_hyperparameters(D, form):
    p = lgp.Hyper(np.int64(lgp.LGP_MATERN52), _forms(D)[form], np.float32(0.3), -2)
    want, keep = lgp.Hyper.of(p).to_c()
    got = lgp._c_hyper(p)
    assert (got.kind, got.D, got.log_outputscale, got.log_noise) == (want.kind, want.D, want.log_outputscale, want.log_noise)
    assert ctypes.string_at(got.log_lengthscale, 4 * D) == ctypes.string_at(want.log_lengthscale, 4 * D)
    del keep
