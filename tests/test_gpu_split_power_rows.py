"""Split products of rows whose largest entry is a power of two (reflectors, unit columns):
the power is its own bound, so the leading digit takes its extreme value and the others keep
one more bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06204_gb300 import build
    build.build()
    from paper_1806_06204_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def handle(zb):
    h = zb.Handle(0)
    yield h
    h.close()


def dev(a):
    import torch
    return torch.from_numpy(np.asfortranarray(a)).cuda()


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("k", [64, 193, 5000])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (0, 1)])
def test_powers_of_two_are_exact(zb, handle, prec, k, ta, tb):
    # +-2^j with j within eight of the row's largest: two digits hold them, and the sums are
    # integers of units whose bits FP64 holds; one row of equal signs fills the leading level
    m, n = 130, 70
    rng = np.random.default_rng(k + prec)
    A = np.ldexp(rng.choice([-1.0, 1.0], (m, k)), rng.integers(-8, 1, (m, k)))
    B = np.ldexp(rng.choice([-1.0, 1.0], (k, n)), rng.integers(-8, 1, (k, n)))
    A[0], B[:, 0], A[1], B[:, 1] = 1.0, 1.0, -1.0, -1.0
    A *= np.ldexp(1.0, rng.integers(-300, 300, (m, 1)))
    B *= np.ldexp(1.0, rng.integers(-300, 300, (1, n)))
    C = zb.zolo_dgemm(handle, dev(A.T if ta else A), dev(B.T if tb else B), transA=bool(ta),
                      transB=bool(tb), prec=prec, slices=9 if prec == 1 else 0)
    assert np.array_equal(C.cpu().numpy(), A @ B)


def test_reflector_gram_keeps_the_bit(zb, handle):
    # columns with a 1 and entries below it: with e = 1 an entry is rounded to units u = 2^-55,
    # a product's float part to f = 2^-54, the result to 2^-54 at most; uniform errors of
    # variance unit^2 / 12.  With the bound one power higher u and f are 2 and 4 times that
    # and the error at least 2.5 times the estimate.
    k, n = 700, 96
    rng = np.random.default_rng(5)
    V = rng.uniform(-1, 1, (k, n)) / 20
    V[np.arange(n), np.arange(n)] = 1.0
    C = zb.zolo_dgemm(handle, dev(V), dev(V), transA=True, prec=zb.ZOLO_SPLIT_BF16, slices=9).cpu().numpy()
    L = V.astype(np.longdouble)
    err = (C - L.T @ L).astype(float)
    if np.finfo(np.longdouble).nmant < 80:
        pytest.skip("long double is too short here")
    off = ~np.eye(n, dtype=bool)
    s = (V * V).sum(0)
    want = np.sqrt(((s[:, None] + s[None, :]) * 2.0 ** -110 + 2.0 ** -108 + 2.0 ** -110) / 12)
    assert np.sqrt((err[off] ** 2).mean()) <= 1.25 * np.sqrt((want[off] ** 2).mean())
