"""zolo_svd of a matrix times a power of four, with its bounds scaled alike: every step is a
scaling by a power of two, so U, V and the sweep count are the unscaled ones bit for bit and
S is theirs times the factor, down to where the FP32 cosines of an unscaled eigensolver
would have left their range."""
import numpy as np
import pytest

from oracle import zolo_oracle as zo
from paper_1806_06204_gb300 import synth

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


def dev(a):
    import torch
    return torch.from_numpy(np.asfortranarray(a)).cuda()


SPECTRA = {"graded": lambda n: np.geomspace(1.0, 1e-4, n), "equal": np.ones,
           "pairs": lambda n: np.repeat(np.geomspace(1.0, 1e-3, n // 2), 2)}


@pytest.mark.parametrize("spectrum", sorted(SPECTRA))
@pytest.mark.parametrize("n", [96, 520])
def test_svd_follows_the_scale_of_the_matrix(zb, spectrum, n):
    sm = synth.make_matrix(n, n, SPECTRA[spectrum](n), seed=n)
    low = 0.9 * float(sm.sigma[-1])
    h = zb.Handle(0)
    try:
        U, S, V, info = zb.zolo_svd(h, dev(sm.A), zb.opts(alpha=1.0, beta=low))
        S0 = S.cpu().numpy()
        assert np.max(np.abs(S0 - sm.sigma)) <= 1e-12
        Vh = V.cpu().numpy()
        assert np.max(np.abs(Vh.T @ Vh - np.eye(n))) <= 2 * max(8.0, n ** 0.5) * zo.EPS
        for k in (-400, -150, -120, -110, -100, -90, 64, 100, 126, 150, 400):
            c = 2.0 ** k
            Uk, Sk, Vk, ik = zb.zolo_svd(h, dev(sm.A * c), zb.opts(alpha=c, beta=low * c))
            assert ik.eig_sweeps == info.eig_sweeps, k
            assert np.array_equal(Sk.cpu().numpy(), S0 * c), k
            assert np.array_equal(Vk.cpu().numpy(), Vh) and np.array_equal(Uk.cpu().numpy(), U.cpu().numpy()), k
    finally:
        h.close()


def test_svd_of_columns_far_apart(zb):
    # singular values over 40 decades on separate coordinates, a few of them equal
    n = 64
    rng = np.random.default_rng(3)
    sigma = np.sort(np.concatenate([np.geomspace(1.0, 1e-40, n - 8), np.full(8, 1e-25)]))[::-1]
    A = np.zeros((n, n))
    A[np.arange(n), rng.permutation(n)] = sigma
    h = zb.Handle(0)
    try:
        # the bound is far above the smallest values: only those near 1 are made unit, but
        # H and its eigenvectors must come out finite
        U, S, V, info = zb.zolo_svd(h, dev(A), zb.opts(alpha=1.0, beta=1e-16), check=False)
        V = V.cpu().numpy()
        assert info.status in (0, 2, 6) and np.all(np.isfinite(V)) and np.all(np.isfinite(S.cpu().numpy()))
        assert np.max(np.abs(V.T @ V - np.eye(n))) <= 2 * 8.0 * zo.EPS
    finally:
        h.close()
