"""The register panels at the edges of their row ranges: clusters of 16 CTAs (up to seven
shifts), of 12 (eight shifts), and of 1, 2, 4 and 8 for the problems of a batch.

m and m + 1 straddle a range; 37 columns make a whole panel and a ragged one.  The bounds
are those of the other decomposition tests."""
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
    h.close()


def dev(a):
    import torch
    return torch.from_numpy(np.asfortranarray(a)).cuda()


def check(sm, Qp, H):
    Qp, H = Qp.cpu().numpy(), H.cpu().numpy()
    assert zo.orthogonality(Qp) <= 1e-13 and zo.backward_error_pd(sm.A, Qp, H) <= 1e-13
    s = np.sort(sm.sigma)
    assert np.max(np.abs(Qp - sm.U @ sm.V.T)) <= 200 * zo.EPS / (s[0] + s[1])


@pytest.mark.parametrize("r,m", [(8, 1600), (8, 3136), (8, 4672), (8, 6208), (8, 9280), (8, 12384),
                                 (7, 2144), (7, 4192), (7, 6240), (7, 8288), (7, 12384)])
@pytest.mark.parametrize("over", [0, 1])
def test_single_calls(handle, r, m, over):
    zb, h = handle
    sm = synth.make_matrix(m + over, N, synth.geometric_sigma(N, 1e4), seed=m + over)
    Qp, H, info = zb.zolo_pd(h, dev(sm.A), zb.opts(beta=1e-4, r=r, force_qr=1))
    assert all(info.used_qr)
    check(sm, Qp, H)


@pytest.mark.parametrize("r", [3, 8])
@pytest.mark.parametrize("prec", [0, 1])
def test_batches(handle, r, prec):
    zb, h = handle
    ms = [511, 512, 1056, 1057, 2080, 2081, 3072, 3073, 4128, 4129]
    mats = [synth.make_matrix(m, N, synth.geometric_sigma(N, 1e4), seed=m) for m in ms]
    os_ = [zb.opts(beta=1e-4, r=r, force_qr=1, prec=prec) for _ in ms]
    Qps, Hs, infos, st = zb.zolo_pd_batched(h, [dev(sm.A) for sm in mats], os_)
    assert st == 0
    for sm, Qp, H in zip(mats, Qps, Hs):
        check(sm, Qp, H)
