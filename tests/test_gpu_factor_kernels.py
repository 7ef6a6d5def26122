"""The QR panel kernels and the Cholesky diagonal block at the edges of their ranges.

The panel form changes with the number of rows and shifts (registers of 8 or 16 CTAs
with 17 to 97 rows a thread, then global memory); the Cholesky block is 64 wide, in
steps of 8 columns, with ragged ends."""
import numpy as np
import pytest

from oracle import zolo_oracle as zo
from paper_1806_06204_gb300 import synth

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


@pytest.mark.parametrize("r", [2, 8])
@pytest.mark.parametrize("m", [37, 256, 511, 512, 1024, 1025, 1056, 1057, 2080, 2081, 4128, 4129, 6176, 6177,
                               8256, 8257, 12352, 12353])
def test_qr_form_at_every_panel_kernel(handle, m, r):
    # n = 37: a whole panel and a ragged one of five columns, both with rows below the top
    zb, h = handle
    n = 37
    sm = synth.make_matrix(m, n, synth.geometric_sigma(n, 1e4), seed=m + r)
    Qp, H, info = zb.zolo_pd(h, dev(sm.A), zb.opts(beta=1e-4, r=r, force_qr=1))
    assert all(info.used_qr)
    Qp, H = Qp.cpu().numpy(), H.cpu().numpy()
    assert zo.orthogonality(Qp) <= 1e-13 and zo.backward_error_pd(sm.A, Qp, H) <= 1e-13
    # the polar factor's sensitivity is 1 / (sigma_{n-1} + sigma_n)
    s = np.sort(sm.sigma)
    assert np.max(np.abs(Qp - sm.U @ sm.V.T)) <= 200 * zo.EPS / (s[0] + s[1])


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 33, 63, 64, 65, 71, 120, 129])
@pytest.mark.parametrize("form", [1, 2])
def test_cholesky_form_at_ragged_blocks(handle, n, form):
    zb, h = handle
    sm = synth.make_matrix(n + 40, n, synth.geometric_sigma(n, 20.0) if n > 1 else np.ones(1), seed=n)
    o = zb.opts(beta=1.0 / 20.0, r=3, max_iter=1, force_qr=0, chol_form=form)
    X1, _, info = zb.zolo_pd(h, dev(sm.A), o)
    ref = zo.zolo_step_chol(sm.A, zo.zolotarev_coeffs(1.0 / 20.0, 3))
    assert info.chol_fallbacks == 0
    assert np.linalg.norm(X1.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [1e-150, 1e-120, 1e120])
def test_scales_beyond_the_fast_roots(handle, scale):
    # squared norms outside [1e-280, 1e280] take the library's square root and division
    zb, h = handle
    sm = synth.make_matrix(90, 50, synth.geometric_sigma(50, 1e3), seed=8)
    # alpha = 1 leaves X_0 = A / alpha tiny or huge: R of the beta estimate, any l
    Qp, H, info = zb.zolo_pd(h, dev(sm.A * scale), zb.opts(beta=0.0, alpha=scale if scale < 1 else 2 * scale, r=4))
    Qp, H = Qp.cpu().numpy(), H.cpu().numpy() / scale
    assert zo.orthogonality(Qp) <= 1e-13 and zo.backward_error_pd(sm.A, Qp, H) <= 1e-13


def test_zero_columns_leave_identity_reflectors(handle):
    # a column of zeros in the top block: its reflector comes from the shift's entry alone
    zb, h = handle
    A = np.zeros((60, 40))
    A[:, :20] = synth.make_matrix(60, 20, synth.geometric_sigma(20, 10.0), seed=4).A
    Qp, H, info = zb.zolo_pd(h, dev(A), zb.opts(beta=1e-3, r=3, force_qr=1), check=False)
    ref, _, _ = zo.zolo_pd(A, 1.0, 1e-3, r=3)
    assert np.max(np.abs(Qp.cpu().numpy() - ref)) <= 1e-12
