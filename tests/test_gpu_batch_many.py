"""An FP64 batch of sixteen matrices and more: those of 512 rows and more take the tiles that
cost the FP64 units least.  Each result meets the invariants and agrees with the single
call's, bit for bit below 512 rows and to rounding (scaled by the polar factor's
conditioning) from there."""
import numpy as np
import pytest

from oracle import zolo_oracle as zo
from paper_1806_06204_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [15, 16, 33])
def test_fp64_batch_equals_single_calls(count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06204_gb300 import build
    build.build()
    from paper_1806_06204_gb300 import binding as zb
    h = zb.Handle(0)
    try:
        ms = [511, 512, 513, 575, 640, 700, 128, 257]
        shapes = [(ms[i % 8], 33 + 13 * (i % 7)) for i in range(count)]
        kappas = [10.0 ** (1 + i % 9) for i in range(count)]
        mats = [synth.make_matrix(m, n, synth.geometric_sigma(n, k), seed=900 + i)
                for i, ((m, n), k) in enumerate(zip(shapes, kappas))]
        As = [torch.from_numpy(np.asfortranarray(sm.A)).cuda() for sm in mats]
        os_ = [zb.opts(beta=1.0 / k, chol_form=1 + i % 2) for i, k in enumerate(kappas)]
        Qps, Hs, infos, st = zb.zolo_pd_batched(h, As, os_)
        assert st == 0
        for sm, a, o, q, hh in zip(mats, As, os_, Qps, Hs):
            q1, h1, _ = zb.zolo_pd(h, a, o)
            Q, H = q.cpu().numpy(), hh.cpu().numpy()
            assert zo.orthogonality(Q) <= 1e-13 and zo.backward_error_pd(sm.A, Q, H) <= 1e-13
            if sm.A.shape[0] < 512:
                assert np.array_equal(Q, q1.cpu().numpy()) and np.array_equal(H, h1.cpu().numpy())
            else:
                s = np.sort(sm.sigma)
                assert np.max(np.abs(Q - q1.cpu().numpy())) <= 200 * zo.EPS / ((s[0] + s[1]) / s[-1])
                assert np.max(np.abs(H - h1.cpu().numpy())) <= 1e-13 * s[-1]
    finally:
        h.close()
