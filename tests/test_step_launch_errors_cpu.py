"""A launch of the CG step that fails is reported by the launcher, not left for a later call to find.

The failure is the absence of a device: a small program linked against the library calls every form of the step with the GPUs
hidden, so that each launch is refused on the host.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    from paper_2605_17898_gb300 import build as b
    lib = b.build()
    exe = str(tmp_path_factory.mktemp("step_launch") / "step_launch_check")
    subprocess.run([b.nvcc(), "-std=c++17", "-O1", *b.ARCH, "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-I", b.CSRC,
                    os.path.join(ROOT, "tests", "native", "step_launch_check.cu"), lib, "-Xlinker", f"-rpath={os.path.dirname(lib)}",
                    "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert out.returncode == 0, out.stdout + out.stderr
    return dict(line.split() for line in out.stdout.splitlines())


@pytest.mark.parametrize("form", ["one-cta", "cluster-8", "three-vec4", "three-vec4-parts", "three-vec1", "three-split", "split",
                                  "precond", "precond-apply", "tally"])
def test_refused_launch_is_returned(errors, form):
    assert int(errors[form]) != 0
