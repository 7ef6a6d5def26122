"""The Jacobi sweeps of zolo_svd at the edges of their kernels' ranges.

FP64 sweep: columns held in registers up to 256, 512 and 1024 rows, read again beyond;
an odd n has a padding column.  FP32 sweep: blocks of 16 columns (an odd number of
blocks is padded), clusters of 1 to 8 CTAs sharing the rows in chunks of 128 (256 from n
= 2048), 16-byte loads only when n is a multiple of 4.

A sweep ends the iteration when no pair's cosine is above max(8, sqrt(n)) eps; rotations
after that move a cosine by rounding only, hence the factor of 2 on V^T V's entries.
"""
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


@pytest.mark.parametrize("n", [1, 2, 3, 16, 17, 33, 127, 128, 130, 255, 256, 257, 511, 512, 513, 1023,
                               1024, 1025, 2047, 2048])
def test_svd_at_the_sweep_kernels_edges(zb, n):
    import torch
    h = zb.Handle(0)
    try:
        kappa = 1e6
        if n <= 513:
            sm = synth.make_matrix(n, n, synth.geometric_sigma(n, kappa), seed=4400 + n)
            A, sigma = torch.from_numpy(np.asfortranarray(sm.A)).cuda(), torch.from_numpy(np.sort(sm.sigma)[::-1].copy()).cuda()
        else:   # the same kind of matrix, built on the device
            g = torch.Generator(device="cuda").manual_seed(4400 + n)
            q = [torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g))[0]
                 for _ in range(2)]
            sigma = torch.logspace(0, -6, n, dtype=torch.float64, device="cuda")
            A = (q[1] @ (q[0] * sigma).t()).t()
        U, S, V, info = zb.zolo_svd(h, A, zb.opts(beta=float(sigma[-1])))
        eye = torch.eye(n, dtype=torch.float64, device="cuda")
        off = (V.t() @ V - eye).abs().max()
        assert float(off) <= 2 * max(8.0, n ** 0.5) * zo.EPS
        norm = torch.linalg.matrix_norm(A)
        assert float(torch.linalg.matrix_norm(A - (U * S) @ V.t()) / norm) <= 1e-13
        assert float(torch.linalg.matrix_norm(U.t() @ U - eye)) / n ** 0.5 <= 1e-13
        assert float((S - sigma).abs().max()) <= 1e-12
        # the same input gives the same bits: no sum depends on the order blocks run in
        U2, S2, V2, _ = zb.zolo_svd(h, A, zb.opts(beta=float(sigma[-1])))
        assert torch.equal(V, V2) and torch.equal(S, S2)
    finally:
        h.close()
