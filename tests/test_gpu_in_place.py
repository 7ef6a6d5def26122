"""FP64 zolo_dgemm with an output that shares elements with an operand: C over A, over B,
over a transposed operand, shifted against it, with tiles by the built-in rule and forced
ones with a K split, against numpy.  Where no tile holds all that its outputs cover, the
product is formed beside C and copied."""
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


def tol(A, B, extra=0.0):
    # k + 3 roundings of terms bounded by |A| |B|, on both sides
    return 2 * (A.shape[1] + 3) * 2.3e-16 * (np.abs(A) @ np.abs(B) + extra)


@pytest.mark.parametrize("pad", [0, 3])
@pytest.mark.parametrize("n", [16, 17, 40, 64, 65, 100])
@pytest.mark.parametrize("m", [20, 40, 1000, 20000])
def test_c_over_a(zb, handle, m, n, pad):
    rng = np.random.default_rng(m + n + pad)
    P, B = rng.standard_normal((m + pad, n)), rng.standard_normal((n, n))
    D = dev(P)
    C = D[:m]
    zb.zolo_dgemm(handle, C, dev(B), C, beta=0.5)
    A = P[:m]
    out = D.cpu().numpy()
    assert np.all(np.abs(out[:m] - (A @ B + 0.5 * A)) <= tol(A, B, np.abs(A)))
    assert np.array_equal(out[m:], P[m:])


@pytest.mark.parametrize("m,n", [(64, 3000), (65, 40), (130, 700), (300, 64)])
def test_c_over_b(zb, handle, m, n):
    rng = np.random.default_rng(m + n)
    A, B = rng.standard_normal((m, m)), rng.standard_normal((m, n))
    C = dev(B)
    zb.zolo_dgemm(handle, dev(A), C, C)
    assert np.all(np.abs(C.cpu().numpy() - A @ B) <= tol(A, B))


@pytest.mark.parametrize("n", [17, 64, 65, 200])
@pytest.mark.parametrize("ta,tb", [(1, 0), (0, 1), (0, 0)])
def test_c_over_both_operands(zb, handle, n, ta, tb):
    # C = op(C) op(C), every element read by a whole row and column of tiles
    A = np.random.default_rng(n).standard_normal((n, n))
    C = dev(A)
    zb.zolo_dgemm(handle, C, C, C, transA=bool(ta), transB=bool(tb))
    X, Y = (A.T if ta else A), (A.T if tb else A)
    assert np.all(np.abs(C.cpu().numpy() - X @ Y) <= tol(X, Y))


@pytest.mark.parametrize("first", [1, 30, 63])
def test_c_shifted_against_a(zb, handle, first):
    m, k, n = 500, 64, 64
    rng = np.random.default_rng(first)
    P, B = rng.standard_normal((m, 128)), rng.standard_normal((k, n))
    D = dev(P)
    zb.zolo_dgemm(handle, D[:, :k], dev(B), D[:, first:first + n])
    out = D.cpu().numpy()
    assert np.all(np.abs(out[:, first:first + n] - P[:, :k] @ B) <= tol(P[:, :k], B))
    assert np.array_equal(out[:, :first], P[:, :first])


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("m,n", [(1000, 64), (300, 300), (60, 500)])
def test_split_products_in_place_have_the_bits_of_others(zb, handle, prec, m, n):
    # the split path slices both operands before it writes C
    rng = np.random.default_rng(m + n)
    A, B, L = dev(rng.standard_normal((m, n))), dev(rng.standard_normal((n, n))), dev(rng.standard_normal((m, m)))
    right, left = (zb.zolo_dgemm(handle, A, B, prec=prec).cpu().numpy(), zb.zolo_dgemm(handle, L, A, prec=prec).cpu().numpy())
    C, D = A.t().clone().t(), A.t().clone().t()
    zb.zolo_dgemm(handle, C, B, C, prec=prec)
    zb.zolo_dgemm(handle, L, D, D, prec=prec)
    assert np.array_equal(C.cpu().numpy(), right) and np.array_equal(D.cpu().numpy(), left)


@pytest.mark.parametrize("v", [0, 3, 4])
@pytest.mark.parametrize("m,n", [(1000, 64), (150, 150), (64, 300)])
def test_forced_kernels_in_place(zb, tmp_path, v, m, n):
    # a kept K split (a tuning file's too) serves an in-place product of any shape
    p = str(tmp_path / "t.txt")
    h = zb.Handle(0)
    try:
        zb.tune_save(h, p)
        with open(p, "a") as f:
            f.write(f"g {m} {n} {n} 1 128 0 {v}\ng {m} {n} {m} 1 128 0 {v}\n")
        assert zb.tune_load(h, p) == 0
        rng = np.random.default_rng(m + n + v)
        A, B = rng.standard_normal((m, n)), rng.standard_normal((n, n))
        C = dev(A)
        zb.zolo_dgemm(h, C, dev(B), C)
        assert np.all(np.abs(C.cpu().numpy() - A @ B) <= tol(A, B))
        L = rng.standard_normal((m, m))
        C = dev(A)
        zb.zolo_dgemm(h, dev(L), C, C)
        assert np.all(np.abs(C.cpu().numpy() - L @ A) <= tol(L, A))
    finally:
        h.close()
