"""Kernel choices of products that pair two inner ones (a 128-column block's 32-wide Gram
blocks) are kept, saved and loaded apart from those of the single product of the same sizes."""
import numpy as np
import pytest

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


def test_paired_and_single_products_have_their_own_choices(zb, tmp_path):
    import torch
    r = 3
    p, q = str(tmp_path / "a.txt"), str(tmp_path / "b.txt")
    h, h2 = zb.Handle(0), zb.Handle(0)
    try:
        zb.autotune(h, True)
        # 320 x 128: V^T V over 448 rows, its two 32-wide pairs in one launch; 376 x 72: the
        # first pair of its only block alone, over 448 rows too
        for m, n in ((320, 128), (376, 72)):
            sm = synth.make_matrix(m, n, synth.geometric_sigma(n, 1e3), seed=m)
            zb.zolo_pd(h, torch.from_numpy(np.asfortranarray(sm.A)).cuda(),
                       zb.opts(beta=1e-3, r=r, force_qr=1, max_iter=1))
        zb.tune_save(h, p)
        lines = open(p).read().splitlines()
        assert any(l.startswith(f"gi 32 32 448 {r} 1 0 2 ") for l in lines)
        assert any(l.startswith(f"g 32 32 448 {r} 1 0 ") for l in lines)
        assert zb.tune_load(h2, p) == 0
        zb.tune_save(h2, q)
        assert sorted(open(q).read().splitlines()) == sorted(lines)
        for bad in ("gi 32 32 448 3 1 0 1 0", "gi 32 32 448 3 1 0 0", "gi 32 32 448 3 1 0 2 8", "gi 32 32"):
            with open(q, "w") as f:
                f.write(lines[0] + "\n" + bad + "\n")
            assert zb.tune_load(h2, q) == 9, bad
    finally:
        h.close()
        h2.close()
