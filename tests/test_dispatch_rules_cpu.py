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
