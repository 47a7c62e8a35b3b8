"""The CG kernels' sum across a block's threads (csrc/limb_sum.cuh) on the host, against exactly rounded sums.

Bound: each of the 2 n values rounds at most half a unit of the last place 2^(e-59), e the exponent of the largest (|v| < 2^e), and
the total rounds twice to float64. A sum of float32 pairs, 2^-48 per addition, misses it and overflows at 3.4e38.
"""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def limb_sum(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    so = str(tmp_path_factory.mktemp("limb_sum") / "limb_sum_check.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_17898_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "limb_sum_check.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).limb_block_sum
    fn.restype = ctypes.c_double
    ptr = np.ctypeslib.ndpointer(np.float32, flags="C")
    fn.argtypes = [ptr, ptr, ctypes.c_int]
    return lambda hi, lo: fn(hi, lo, len(hi))


def _pairs(kind, n, rng):
    z = rng.standard_normal(n)
    v = {"squares": z * z, "signed": z, "equal": np.full(n, 0.7), "wide": z * np.exp(20 * rng.standard_normal(n)),
         "spike": np.where(np.arange(n) == 3, 1e6, 1.0) * z * z, "cancelling": np.where(np.arange(n) % 2, -1.0, 1.0) * (1 + 1e-6 * z),
         "large": 3e38 * np.abs(np.sin(z)), "small": 1e-36 * z, "denormal": 1e-43 * z, "zero": 0.0 * z}[kind]
    hi = v.astype(np.float32)
    return hi, np.where(np.abs(hi) < 1e37, (v - hi.astype(np.float64)), 0.0).astype(np.float32)


@pytest.mark.parametrize("kind", ["squares", "signed", "equal", "wide", "spike", "cancelling", "large", "small", "denormal", "zero"])
@pytest.mark.parametrize("n", [1, 2, 33, 256, 1024])
def test_sum(limb_sum, kind, n):
    for seed in range(20):
        hi, lo = _pairs(kind, n, np.random.default_rng(1000 * n + seed))
        exact = math.fsum(hi.astype(np.float64).tolist() + lo.astype(np.float64).tolist())
        largest = float(max(np.abs(hi).max(), np.abs(lo).max()))
        e = max(math.frexp(largest)[1], -108)
        assert abs(limb_sum(hi, lo) - exact) <= 2 * n * 2.0 ** (e - 60) + 2.0 ** -52 * abs(exact)


def test_not_finite(limb_sum):
    for bad, want in ((np.inf, math.isinf), (np.nan, math.isnan)):
        hi = np.ones(40, np.float32)
        hi[7] = bad
        assert want(limb_sum(hi, np.zeros(40, np.float32)))
