"""The workspace query against the buffers a call holds: the forms that work on 128-column
blocks alone ask for nothing wider, at any size."""
import pytest


@pytest.fixture(scope="module")
def zb():
    from paper_1806_06204_gb300 import build
    build.build()
    from paper_1806_06204_gb300 import binding
    return binding


def blocks(m, n, r, sb):
    """Bytes of X, X_next, S, M and per shift W, V, the panels' and (super-)blocks' T, V^T V,
    V^T C and T V^T C with super-blocks of sb columns."""
    shift = ((m + n) * n + (m + sb) * n + -(-n // 32) * 1024 + -(-n // sb) * sb * sb + sb * sb + 2 * sb * n)
    return 8 * (3 * m * n + n * n + r * shift)


SLACK = 1 << 16   # partial sums, norms, status, alignment


@pytest.mark.parametrize("m,n,r", [(2047, 2047, 8), (2048, 2048, 8), (4096, 4096, 8), (16384, 4096, 6),
                                   (16384, 16384, 8), (3000, 2500, 1)])
def test_bytes_by_precision(zb, m, n, r):
    f64 = zb.workspace_bytes(m, n, r)
    assert blocks(m, n, r, 128) <= f64 <= blocks(m, n, r, 128) + SLACK
    wide = 512 if n >= 2048 else 128
    assert zb.workspace_bytes(m, n, r, zb.ZOLO_SPLIT_BF16) == zb.workspace_bytes(m, n, r, zb.ZOLO_SPLIT_FP16)
    # the split forms' planes are the same: what is left of their difference is the super-blocks'
    diff = zb.workspace_bytes(m, n, r, zb.ZOLO_SPLIT_BF16) - zb.workspace_bytes(m, n, r, zb.ZOLO_SPLIT_FP8)
    assert abs(diff - (blocks(m, n, r, wide) - blocks(m, n, r, 128))) <= SLACK
