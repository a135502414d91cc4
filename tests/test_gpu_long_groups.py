"""Sphere packs of narrow pores whose last phases have a group of thousands
of steps: the value phases take them whole, on the whole GPU and on one
cluster, alone and in a batch; against the oracle's run (Section 2.1)."""
import numpy as np
import pytest

import oracle as O
from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ibip():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip as m
    return m


@pytest.mark.parametrize("edge,porosity,seed", [(130, 0.36, 4), (140, 0.40, 0)])
def test_taken_whole(ibip, edge, porosity, seed):
    img = S.sphere_pack((edge,) * 3, 4, porosity, np.random.default_rng(seed))
    d = O.edt(img)
    rseq, rr2, rcen, _, K = O.invade(img, d, inlet=0)
    dev, dt = torch.from_numpy(img).cuda(), torch.from_numpy(d).cuda()
    ctx = ibip.Context(0)
    for shared in (False, True):
        ctx.set_shared_device(shared)
        seq, r2, cen, k, _ = ctx.invade(dev, dt)
        assert ctx.invade_stats()["items"] == 0   # nothing was left to the one-CTA loop
        assert k == K and np.array_equal(seq.cpu().numpy(), rseq)
        assert np.array_equal(r2.cpu().numpy(), rr2) and np.array_equal(cen.cpu().numpy(), rcen)
    out = ctx.invade_batched([dev, dev[:40].contiguous()], 0, trapping=False, curve=False)[0]
    assert out["K"] == K and np.array_equal(out["seq"].cpu().numpy(), rseq)


def test_small_packs_taken_whole(ibip):
    """Groups of a few hundred steps in 32^3 packs."""
    ctx = ibip.Context(0)
    for seed in range(16):
        img = S.sphere_pack((32,) * 3, 4, 0.42, np.random.default_rng(seed))
        d = O.edt(img)
        if 0.45 * (d == 1).sum() < 100.0 * float(d.max()) ** 0.8:
            continue   # few steps: the loop's by rule
        seq = ctx.invade(torch.from_numpy(img).cuda(), torch.from_numpy(d).cuda())[0]
        assert ctx.invade_stats()["items"] == 0
        assert np.array_equal(seq.cpu().numpy(), O.invade(img, d, inlet=0)[0])
