"""A product's chained launches on the caller's stream and inside a captured graph.

Its kernels are placed before their predecessors end, so each has to wait for the values it reads: here V is written by the
kernel right before the call, the result is read by the one right after it, and the next product overwrites the same
workspace at once. Replays of a captured chain give the bits of the direct calls (at shapes whose sums have a fixed
order; 2e-6 of the column norm, twice what float32 additions in another order change, for the symmetric tensor-core ones).
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,t", [(700, 2, 1), (3000, 8, 3), (4099, 5, 5), (1500, 8, 16), (5000, 3, 16), (9000, 8, 32)])
def test_replay_matches_direct_calls(lgp, N, D, t):
    import torch
    p = wl.random_problem(N, D, wl.MATERN52, seed=N)
    X = torch.as_tensor(p.X, device="cuda")
    W = torch.as_tensor(wl.rhs_block(N, t, seed=t), device="cuda")
    V, out = torch.empty_like(W), [torch.empty_like(W) for _ in range(3)]
    ctx = lgp.Context(0)
    stream = torch.cuda.Stream()

    def chain():
        for k, o in enumerate(out):
            torch.mul(W, 1.0 + k, out=V)
            lgp.lgp_kernel_matvec(X, p, V, out=o, ctx=ctx)
        return out[0] + out[1] - out[2]

    try:
        with torch.cuda.stream(stream):
            chain()
            direct = chain().clone()
            ref = [o.clone() for o in out]
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                zero = chain()
            for o in out:
                o.zero_()
            for _ in range(5):
                graph.replay()
            stream.synchronize()
        scale = ref[0].norm(dim=0)
        tol = 2e-6 if t >= 16 and N >= 4608 else 0.0
        for a, b in zip(out, ref):
            assert ((a - b).norm(dim=0) <= tol * 3.0 * scale).all()
        assert ((zero - direct).norm(dim=0) <= 9.0 * tol * scale).all()
        # K (1 W) + K (2 W) - K (3 W) is zero up to the products' own rounding
        assert (zero.norm(dim=0) <= 1e-5 * 3.0 * scale).all()
        assert ctx.check_device_status() == lgp.LGP_OK
    finally:
        ctx.close()
