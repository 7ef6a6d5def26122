"""The Cholesky form's outer blocks of 256 rows on the split forms: n ends inside, at and
after an outer block or one of its panels.

One iteration from a matrix of condition 20 against the oracle's step, to the tolerance of
the FP64 products' test: the split products are of the same grade."""
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


@pytest.mark.parametrize("n", [192, 193, 255, 256, 257, 320, 321, 511, 513, 577])
@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("form", [1, 2])
def test_one_step_matches_the_oracle(handle, n, prec, form):
    import torch
    zb, h = handle
    sm = synth.make_matrix(n, n, synth.geometric_sigma(n, 20.0), seed=n)
    o = zb.opts(beta=1.0 / 20.0, r=3, max_iter=1, force_qr=0, chol_form=form, prec=prec)
    X1, _, info = zb.zolo_pd(h, torch.from_numpy(np.asfortranarray(sm.A)).cuda(), o)
    ref = zo.zolo_step_chol(sm.A, zo.zolotarev_coeffs(1.0 / 20.0, 3))
    assert info.chol_fallbacks == 0
    assert np.linalg.norm(X1.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
