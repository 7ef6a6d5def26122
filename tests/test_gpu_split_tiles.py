"""The split product's kernel at the edges of its tiles, chunks and K split.

A tile is 128 x 64 (FP8: 128 x 32); the leading levels are drained every 192 terms
(FP8: 4096); one chunk that holds all of K is finished in integers; few tiles with
a long K share it over a cluster; more tiles than SMs run several to a CTA; M < 128
< N swaps the operands."""
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


@pytest.mark.parametrize("m,n,k", [(128, 64, 64), (129, 65, 191), (128, 33, 192), (300, 200, 193),
                                   (40, 500, 385), (100, 60, 5000), (512, 512, 9000),
                                   (256, 192, 6151), (2100, 1300, 130)])
@pytest.mark.parametrize("prec,S", [(1, 8), (1, 9), (2, 8), (3, 11)])
def test_split_product_at_the_edges(handle, m, n, k, prec, S):
    zb, h = handle
    rng = np.random.default_rng(m + n + k)
    A = rng.standard_normal((k, m)) * 10.0 ** rng.uniform(-4, 0, (1, m))   # rows of op(A) scaled
    B = rng.standard_normal((k, n))
    C0 = rng.standard_normal((m, n))
    C = dev(C0)
    zb.zolo_dgemm(h, dev(A), dev(B), C, alpha=-1.0, beta=0.5, transA=True, prec=prec, slices=S)
    # an extended reference of some rows and columns, the edges of the tiles among them
    i = np.unique(np.r_[0, m - 1, rng.integers(0, m, 14), np.arange(min(m, 130) - 3, min(m, 130))])
    j = np.unique(np.r_[0, n - 1, rng.integers(0, n, 14), np.arange(min(n, 65) - 3, min(n, 65))])
    ref = -(A.T[i].astype(np.longdouble) @ B[:, j].astype(np.longdouble)) + 0.5 * C0[np.ix_(i, j)]
    amax, bmax = np.abs(A).max(0)[i, None], np.abs(B).max(0)[None, j]
    # per term: two operand roundings of 2^-(bits + 1) 2^e with 2^e <= 4 max, and the pairs
    # left out: at the first level left out p products below 2^(2b - 2) 2^-(b (top + 1))
    b, planes, top = {(1, 8): (8, 6, 8), (1, 9): (8, 7, 9), (2, 8): (8, 7, 8), (3, 11): (5, 11, 13)}[prec, S]
    per = 2 * 2.0 ** -(b * planes - 1) + 1.1 * 16 * (2 * planes - top) * 2.0 ** (2 * b - 2 - b * (top + 1))
    # the float part's FP32 rounding lies below the last bit kept; two FP64 roundings at the end
    tol = 1.1 * k * per * amax * bmax + 4 * 2.3e-16 * (np.abs(ref).astype(float) + np.abs(C0[np.ix_(i, j)]))
    got = C.cpu().numpy()
    assert np.all(np.abs(got[np.ix_(i, j)] - ref) <= tol)
    # every entry, within what the FP64 reference itself may be off
    full = -(A.T @ B) + 0.5 * C0
    tol = (1.1 * k * per * np.abs(A).max(0)[:, None] * np.abs(B).max(0)[None, :]
           + 2 * (k + 3) * 2.3e-16 * (np.abs(A).T @ np.abs(B) + np.abs(C0)))
    assert np.all(np.abs(got - full) <= tol)


@pytest.mark.parametrize("prec,S", [(1, 9), (2, 8), (3, 11)])
@pytest.mark.parametrize("expo", [-560, 500, -1060])
def test_split_product_at_the_ends_of_the_range(handle, prec, S, expo):
    # powers of two scale every digit-exact product exactly: results below the normal
    # range, and near its top
    zb, h = handle
    rng = np.random.default_rng(3)
    A = np.ldexp(rng.integers(1, 9, (140, 60)).astype(np.float64), expo)
    B = np.ldexp(rng.integers(1, 9, (60, 70)).astype(np.float64), expo if expo > -1000 else 0)
    C = zb.zolo_dgemm(h, dev(A), dev(B), prec=prec, slices=S).cpu().numpy()
    with np.errstate(under="ignore"):
        ref = np.ldexp(np.ldexp(A, -expo) @ np.ldexp(B, -expo if expo > -1000 else 0),
                       2 * expo if expo > -1000 else expo)
    assert np.array_equal(C, ref)


@pytest.mark.parametrize("m,n", [(2048, 2048), (2300, 2177)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_super_blocks_keep_the_invariants(handle, m, n, prec):
    # from n = 2048 the 16-bit forms apply 512 columns' reflectors together; 2177 = 4 x 512
    # + 129 leaves a super-block of a whole and a one-column block
    import torch
    zb, h = handle
    g = torch.Generator(device="cuda").manual_seed(n + prec)

    def haar(rows, cols):
        return torch.linalg.qr(torch.randn(rows, cols, dtype=torch.float64, device="cuda", generator=g))[0]

    s = torch.logspace(0, -8, n, dtype=torch.float64, device="cuda")
    U, V = haar(m, n), haar(n, n)
    A = (V @ (U * s).t()).t()
    Qp, H, info = zb.zolo_pd(h, A, zb.opts(beta=1e-8, r=2, prec=prec, ns_steps=1))
    assert info.used_qr[0]
    bwd = torch.linalg.matrix_norm(A - Qp @ H) / torch.linalg.matrix_norm(A)
    orth = torch.linalg.matrix_norm(Qp.t() @ Qp - torch.eye(n, dtype=torch.float64, device="cuda")) / n ** 0.5
    assert float(bwd) <= 1e-13 and float(orth) <= 1e-13
    # H = V diag(s) V^T to the grade of the iteration (A's own rounding included)
    assert float(torch.linalg.matrix_norm(H - (V * s) @ V.t()) / torch.linalg.matrix_norm(H)) <= 1e-13
