"""QR panels where the GPU has no room for clusters beyond the portable eight CTAs (or beyond
twelve): the kernels of eight CTAs up to 4128 rows and the global-memory one above."""
import numpy as np
import pytest

from oracle import zolo_oracle as zo
from paper_1806_06204_gb300 import synth

pytestmark = pytest.mark.gpu

N = 37


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
    zb.debug_max_cluster(h, 0)
    h.close()


@pytest.mark.parametrize("most", [8, 12])
@pytest.mark.parametrize("r", [2, 8])
@pytest.mark.parametrize("m", [511, 512, 3072, 3073, 4128, 4129, 9280, 9281])
def test_smaller_clusters(handle, most, r, m):
    import torch
    zb, h = handle
    sm = synth.make_matrix(m, N, synth.geometric_sigma(N, 1e4), seed=m + r)
    zb.debug_max_cluster(h, most)
    A = torch.from_numpy(np.asfortranarray(sm.A)).cuda()
    Qp, H, info = zb.zolo_pd(h, A, zb.opts(beta=1e-4, r=r, force_qr=1))
    assert all(info.used_qr)
    Qp, H = Qp.cpu().numpy(), H.cpu().numpy()
    assert zo.orthogonality(Qp) <= 1e-13 and zo.backward_error_pd(sm.A, Qp, H) <= 1e-13
    s = np.sort(sm.sigma)
    assert np.max(np.abs(Qp - sm.U @ sm.V.T)) <= 200 * zo.EPS / (s[0] + s[1])


def test_argument_checks(handle):
    zb, h = handle
    assert zb.LIB.zolo_debug_max_cluster(None, 8) == -1
    for bad in (-1, 1, 9, 17):
        assert zb.LIB.zolo_debug_max_cluster(h.ptr, bad) == -2
