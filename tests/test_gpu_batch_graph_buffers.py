"""A recorded batch graph is replayed only while every buffer its kernels hold is the
handle's: the split path's slice planes and exponents grow apart from the workspace, and a
graph recorded before they moved is recorded anew."""
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


class Batch:
    def __init__(self, zb, n, count, prec, seed):
        import torch
        self.mats = [synth.make_matrix(n, n, synth.geometric_sigma(n, 1e3), seed=seed + i) for i in range(count)]
        self.As = [torch.from_numpy(np.asfortranarray(sm.A)).cuda() for sm in self.mats]
        self.os = [zb.opts(beta=1e-3, prec=prec, r=4) for _ in self.mats]
        self.Qs = [zb.empty_colmajor(n, n) for _ in self.mats]
        self.Hs = [zb.empty_colmajor(n, n) for _ in self.mats]

    def run(self, zb, h):
        for q, x in zip(self.Qs, self.Hs):
            q.zero_()
            x.zero_()
        _, _, _, st = zb.zolo_pd_batched(h, self.As, self.os, Qps=self.Qs, Hs=self.Hs)
        assert st == 0
        for sm, q, x in zip(self.mats, self.Qs, self.Hs):
            q, x = q.cpu().numpy(), x.cpu().numpy()
            assert zo.orthogonality(q) <= 1e-13 and zo.backward_error_pd(sm.A, q, x) <= 1e-13


@pytest.mark.parametrize("prec", [1, 2, 3])
def test_graph_recorded_anew_after_the_split_buffers_grew(zb, prec):
    h = zb.Handle(0)
    try:
        large = Batch(zb, 320, 3, zb.ZOLO_FP64, 10)    # sizes the lanes' workspaces
        small = Batch(zb, 96, 3, prec, 20)
        middle = Batch(zb, 256, 3, prec, 30)           # fits them, but not the small one's planes
        large.run(zb, h)
        small.run(zb, h)
        small.run(zb, h)
        assert zb.batch_graphs_recorded(h) == 2        # the second run replays
        middle.run(zb, h)
        small.run(zb, h)
        assert zb.batch_graphs_recorded(h) == 4        # small's graph held the freed planes
        small.run(zb, h)
        middle.run(zb, h)
        large.run(zb, h)                               # plain FP64: holds no split buffer
        assert zb.batch_graphs_recorded(h) == 4
    finally:
        h.close()


def test_graph_recorded_with_the_stall_hook_on_is_not_replayed_with_it_off(zb):
    h = zb.Handle(0)
    try:
        b = Batch(zb, 96, 2, zb.ZOLO_SPLIT_BF16, 40)
        zb.debug_stall(h, zb.ZOLO_STALL_SPLIT_GEMM, 100_000)
        _, _, infos, st = zb.zolo_pd_batched(h, b.As, b.os, Qps=b.Qs, Hs=b.Hs, check=False)
        assert st == 7 and all(i.status == 7 for i in infos)   # ZOLO_ETIMEOUT
        zb.debug_stall(h, 0, 0)
        b.run(zb, h)
    finally:
        h.close()
