"""Batches of few and of many, small and large images, which run on clusters
of 16 CTAs down to one: every image equals the call made for it alone, and
some of them the oracle's run (Sections 2.1-2.2)."""
import numpy as np
import pytest

import oracle as O
from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,lo,hi", [(2, 60, 70), (9, 40, 50), (30, 24, 44), (90, 20, 24), (200, 9, 40), (330, 8, 20)])
def test_each_cluster_size(n, lo, hi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    ctx = ibip.Context(0)
    kinds = [S.mixed_image(i, 900 + n, lo, hi) for i in range(12)]
    imgs = [np.ascontiguousarray(kinds[i % 12][: max(4, kinds[i % 12].shape[0] - i % 5)]) for i in range(n)]
    dev = [torch.from_numpy(a).cuda() for a in imgs]
    out = ctx.invade_batched(dev, 3, 2)
    for i, (a, d, r) in enumerate(zip(imgs, dev, out)):
        seq, r2, cen, K, st = ctx.invade(d, inlet=3)
        tr, so = ctx.trapping(seq, 2)
        assert r["status"] == 0 and r["K"] == K and torch.equal(r["seq"], seq) and torch.equal(r["seq_out"], so)
        assert torch.equal(r["step_r2"], r2) and torch.equal(r["step_centre"], cen) and torch.equal(r["trapped"], tr)
        if i % 31 == 0:
            assert np.array_equal(r["seq"].cpu().numpy(), O.invade(a, O.edt(a), inlet=3)[0])
