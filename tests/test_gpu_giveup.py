"""Invasions whose value phases give up part of the way (a burst of more steps
than a group may take): the one-CTA loop goes on from the phases done.  Step
limits on either side of the change-over, inlet masks, resumed runs and
batches, against the oracle's run (Section 2.1)."""
import numpy as np
import pytest

import oracle as O
from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    return ibip.context()


def image(kind):
    """Noise of single-voxel pores, one long chain; "cavity": with a wide
    pore at the inlet whose phases come first."""
    rng = np.random.default_rng(5)
    img = S.random_image((64, 62, 66), 0.7, rng)
    if kind == "cavity":
        g = np.indices(img.shape)
        img[((g - np.array([8, 30, 32])[:, None, None, None]) ** 2).sum(0) < 150] = 1
    return img


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("kind", ["noise", "cavity"])
def test_give_up(ctx, kind):
    img = image(kind)
    d = O.edt(img)
    rseq, rr2, rcen, _, K = O.invade(img, d, inlet=0)
    dev = cuda(img)
    seq, r2, cen, k, _ = ctx.invade(dev, inlet=0)
    assert ctx.invade_stats()["items"] > 0 and K > 4096   # the loop took part
    assert k == K and np.array_equal(seq.cpu().numpy(), rseq)
    assert np.array_equal(r2.cpu().numpy(), rr2) and np.array_equal(cen.cpu().numpy(), rcen)
    for limit in (1, 40, K // 3, K - 1, K):
        s, a, _, kl, _ = ctx.invade(dev, inlet=0, max_steps=limit)
        want = np.where(rseq > limit, -1, rseq)
        assert kl == limit and np.array_equal(s.cpu().numpy(), want) and np.array_equal(a.cpu().numpy(), rr2[:limit])
    out = ctx.invade_batched([dev, dev[:40].contiguous()], 0, 1)
    assert np.array_equal(out[0]["seq"].cpu().numpy(), rseq) and out[0]["K"] == K
    part = np.ascontiguousarray(img[:40])
    assert np.array_equal(out[1]["seq"].cpu().numpy(), O.invade(part, O.edt(part), inlet=0)[0])


@pytest.mark.parametrize("first", [3, 500])
def test_give_up_resumed(ctx, first):
    img = image("cavity")
    mask = np.zeros_like(img)
    mask[20:24, 10:50, 10:50] = 1
    d = O.edt(img)
    rseq, rr2, rcen, _, K = O.invade(img, d, mask=mask)
    dev, m = cuda(img), cuda(mask)
    part = ctx.invade_ex(dev, inlet_mask=m, max_steps=first)
    seq, r2, cen, k, _ = ctx.invade_ex(dev, inlet_mask=m, resume_from=part[:3])
    assert k == K and np.array_equal(seq.cpu().numpy(), rseq) and np.array_equal(r2.cpu().numpy(), rr2)
