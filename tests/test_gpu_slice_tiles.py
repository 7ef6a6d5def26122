"""The slicing kernel at the edges of its tiles: K ends inside, at and after a tile of 64, a
CTA's tiles all kept in shared memory (up to four of each CTA, eight CTAs) or some read
again, 16 rows per cluster; either storage order of both operands.

Entries are integers of one digit (below 64) times a power of two per row of op(A) and per
column of op(B): every step is exact, so is the result.  The row of 2^-1074 alone is not
normalised: a row of subnormals counts as below 2^-1022, and its products carry the error
of the format at that size, 2 k 2^-48 max|A| max|B|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06204_gb300 import build
    build.build()
    from paper_1806_06204_gb300 import binding as zb
    h = zb.Handle(0)
    yield zb, h
    h.close()


def dev(a):
    import torch
    return torch.from_numpy(np.asfortranarray(a)).cuda()


@pytest.mark.parametrize("prec,S", [(1, 8), (1, 9), (2, 8), (3, 11)])
@pytest.mark.parametrize("k", [1, 63, 64, 65, 255, 257, 2048, 2049, 2113, 4097, 5000])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 1)])
def test_scaled_integer_products_are_exact(handle, prec, S, k, ta, tb):
    zb, h = handle
    m, n = 33, 17
    rng = np.random.default_rng(k + 7 * prec + ta)
    A = rng.integers(-63, 64, (m, k)).astype(np.float64)
    B = rng.integers(-63, 64, (k, n)).astype(np.float64)
    ea = np.concatenate([[-1074, -1060, 900, 0], rng.integers(-300, 300, m - 4)])
    eb = np.concatenate([[90, 0], rng.integers(-40, 40, n - 2)])
    A[5] = 0.0
    As, Bs = np.ldexp(A, ea[:, None]), np.ldexp(B, eb[None, :])
    C = zb.zolo_dgemm(h, dev(As.T if ta else As), dev(Bs.T if tb else Bs), transA=bool(ta), transB=bool(tb),
                      prec=prec, slices=S).cpu().numpy()
    ref = np.ldexp(A @ B, ea[:, None] + eb[None, :])
    assert np.array_equal(C[1:], ref[1:])
    bmax = np.max(np.abs(B), axis=0)
    assert np.all(np.abs(C[0] - ref[0]) <= np.ldexp(2.0 * k * bmax, eb - 48 - 1022))
