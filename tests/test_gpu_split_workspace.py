"""The slice planes a call reserves hold every product of its QR form: with one shift there
is no room but one entry's, and a fresh handle has no larger call's planes to lean on."""
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


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("n", [33, 65, 100, 128, 129, 200])
@pytest.mark.parametrize("m", [1024, 2048, 4096])
def test_one_shift_on_a_fresh_handle(zb, m, n, prec):
    import torch
    sm = synth.make_matrix(m, n, synth.geometric_sigma(n, 1e3), seed=m + n)
    h = zb.Handle(0)
    try:
        A = torch.from_numpy(np.asfortranarray(sm.A)).cuda()
        Qp, H, info = zb.zolo_pd(h, A, zb.opts(beta=1e-3, r=1, force_qr=1, prec=prec))
        Qp, H = Qp.cpu().numpy(), H.cpu().numpy()
        assert zo.orthogonality(Qp) <= 1e-13 and zo.backward_error_pd(sm.A, Qp, H) <= 1e-13
    finally:
        h.close()


def test_one_shift_of_the_super_block_width(zb):
    import torch
    m, n = 2304, 2048
    g = torch.Generator(device="cuda").manual_seed(5)
    q = torch.linalg.qr(torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g))[0]
    A = (q * torch.logspace(0, -3, n, dtype=torch.float64, device="cuda")).t().contiguous().t()
    for prec in (1, 2):
        h = zb.Handle(0)
        try:
            Qp, H, info = zb.zolo_pd(h, A, zb.opts(beta=1e-3, r=1, force_qr=1, prec=prec, estimate=True))
            assert info.status == 0 and info.bwd_est <= 1e-13 and info.orth_est <= 1e-13
        finally:
            h.close()
