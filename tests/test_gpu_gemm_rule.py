"""The built-in FP64 tile and K-split rule through zolo_dgemm: every tile shape
(64 x 64, 32 x 32, 16 x 16, and 64 x 16 in place), unsplit and cut over clusters of
2, 4 and 8, at sizes around the tile edges, against numpy."""
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


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (17, 15, 31), (16, 16, 256), (96, 64, 200),
                                   (33, 97, 1000), (31, 33, 4099), (257, 255, 17), (300, 290, 130),
                                   (1000, 600, 33), (1100, 1030, 70)])
@pytest.mark.parametrize("ta,tb,alpha,beta", [(0, 0, 1.0, 0.0), (1, 0, -1.0, 1.0), (0, 1, 0.5, -2.0),
                                              (1, 1, -3.0, 0.0)])
def test_rule_matches_numpy(handle, m, n, k, ta, tb, alpha, beta):
    zb, h = handle
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    A = rng.standard_normal((k, m) if ta else (m, k))
    B = rng.standard_normal((n, k) if tb else (k, n))
    C0 = rng.standard_normal((m, n))
    C = dev(C0)
    zb.zolo_dgemm(h, dev(A), dev(B), C, alpha=alpha, beta=beta, transA=bool(ta), transB=bool(tb))
    opA, opB = A.T if ta else A, B.T if tb else B
    ref = alpha * (opA @ opB) + beta * C0
    # k + 3 roundings of terms bounded by |alpha| |A| |B|, on both sides
    tol = 2 * (k + 3) * 2.3e-16 * (abs(alpha) * (np.abs(opA) @ np.abs(opB)) + abs(beta) * np.abs(C0))
    assert np.all(np.abs(C.cpu().numpy() - ref) <= tol)


@pytest.mark.parametrize("m,n", [(64, 3000), (64, 40), (50, 300), (20, 500)])
def test_in_place_products_read_before_they_write(handle, m, n):
    zb, h = handle
    rng = np.random.default_rng(m + n)
    A, B0 = rng.standard_normal((m, m)), rng.standard_normal((m, n))
    C = dev(B0)
    zb.zolo_dgemm(h, dev(A), C, C)
    tol = 2 * (m + 3) * 2.3e-16 * (np.abs(A) @ np.abs(B0))
    assert np.all(np.abs(C.cpu().numpy() - A @ B0) <= tol)
