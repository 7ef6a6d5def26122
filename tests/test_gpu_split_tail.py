"""Split products whose last wave of tiles is shared by pairs of CTAs: one tile, half the SMs
and one more than that beyond the whole waves (152 SMs, tiles of 128 x 64, FP8 128 x 32), K
from the shortest that is shared.

Integers below 64 of one digit: the product and the addend are exact in every form."""
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


@pytest.mark.parametrize("mt,nt", [(9, 17), (12, 19), (13, 18), (8, 25), (19, 24)])
@pytest.mark.parametrize("k", [192, 193, 256, 449, 700])
@pytest.mark.parametrize("prec,S", [(1, 8), (1, 9), (2, 8), (3, 11)])
def test_shared_last_wave_is_exact(handle, mt, nt, k, prec, S):
    import torch
    zb, h = handle
    m, n = 128 * mt - 3, (32 if prec == 3 else 64) * nt - 5
    k = 2 * k if prec == 3 else k          # the same number of K blocks
    g = torch.Generator(device="cuda").manual_seed(mt * 100 + nt + k)
    A, B, C0 = (torch.randint(-63, 64, s, device="cuda", generator=g).to(torch.float64)
                for s in ((k, m), (n, k), (n, m)))
    C = C0.clone()
    zb.zolo_dgemm(h, A.t(), B.t(), C.t(), alpha=-1.0, beta=1.0, prec=prec, slices=S)
    assert torch.equal(C, C0 - B @ A)
