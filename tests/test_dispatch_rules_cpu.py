"""Host rules of the float32 products, read from the built library without a GPU: partial sums per row and column."""
import ctypes

import pytest

SMS = 152


@pytest.fixture(scope="module")
def slots():
    from paper_2605_17898_gb300 import build as b
    fn = getattr(ctypes.CDLL(b.build()), "_ZN3lgp22mv_simt_partial_floatsElliii")  # lgp::mv_simt_partial_floats
    fn.restype = ctypes.c_int64
    fn.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int]

    def count(N, t, D):
        Np = -(-N // 256) * 256
        f = fn(N, Np, t, D, SMS)
        assert f % (Np * t) == 0
        return f // (Np * t)
    return count


@pytest.mark.parametrize("D", range(1, 9))
@pytest.mark.parametrize("N,t", [(93000, 4), (100000, 4), (115000, 3), (133000, 2), (187000, 1), (250000, 1)])
def test_blocks_of_1024_rows_need_two_ctas_on_an_sm(slots, N, t, D):
    """Where the partial sums of 512-row blocks pass 256 MiB, 1024-row blocks run only if two CTAs share an SM's 228 KB: at D = 8 and
    four padded columns one CTA of four warps was 1.4 times slower than the row kernel."""
    blocks = -(-N // 1024)
    padded = t if t <= 2 else 4
    rows = 64 if D <= 4 and padded <= 2 else 32
    smem = 4 * (1024 * (D + 5 * padded) + 4 * rows * padded)
    if 2 * (smem + 1024) <= 228 * 1024:
        assert slots(N, t, D) == blocks
    else:
        assert slots(N, t, D) not in (blocks, -(-N // 512))
    assert slots(N, t, D) * N * t * 4 <= 256 << 20


@pytest.fixture(scope="module")
def step():
    from paper_2605_17898_gb300 import build as b
    fn = getattr(ctypes.CDLL(b.build()), "_ZN3lgp12cg_step_ruleEliib")  # lgp::cg_step_rule
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_bool]
    return fn


@pytest.mark.parametrize("N,t,S,ctas", [
    (1024, 1, 16, 1), (500, 8, 8, 1), (8192, 1, 5, 8), (1, 1, 0, 1), (8192, 1, 0, 1), (8193, 1, 0, 8),
    (8000, 2, 63, 8), (4500, 4, 71, 16), (8000, 8, 125, 0),   # 1.0, 1.3 and 8 million partial sums
    (65000, 1, 127, 0), (16000, 4, 63, 16), (9000, 8, 71, 0),
    (65536, 1, 16, 8), (65536, 1, 17, 16), (262144, 1, 16, 16), (262144, 1, 17, 0), (8193, 32, 0, 0),
    (1000, 3, 1, 0), (100, 128, 0, 0),
])
def test_cluster_of_the_cg_step(step, N, t, S, ctas):
    """One cluster runs a CG step only where its SMs can also take the product's S partial sums per element: beyond 2^20 (8 CTAs) and
    2^22 (16) the step had become slower than the launches it replaced."""
    assert step(N, t, S, True) == ctas
    assert step(N, t, S, False) == (0 if ctas == 16 else ctas)


@pytest.mark.parametrize("t,rows", [(16, 256), (32, 128), (64, 64)])
@pytest.mark.parametrize("N", [3000, 4500, 6000, 8000])
def test_row_kernel_splits_of_many_columns(slots, N, t, rows):
    """From 16 columns on the row kernel aims at 8 CTAs per SM while its row blocks (64 columns: two groups of 32 over 128 rows) are fewer
    than half the SMs, and at 16 up to their number: with 32, splits of one column tile, N = 6000 had become 11% to 18% slower."""
    blocks = -(-N // rows)
    assert blocks < SMS
    assert 1 < slots(N, t, 8) and (slots(N, t, 8) - 1) * blocks < (8 if 2 * blocks < SMS else 16) * SMS
