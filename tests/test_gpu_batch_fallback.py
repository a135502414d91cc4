"""Batches in which some images are left to the one-CTA loop (runs that the
value phases give up, images without solid) while the trapping and the curves
of the others are under way on the second stream: every output of every image
equals the calls made for it alone (Sections 2.1-2.2)."""
import time

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


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def chain(seed, shape=(64, 62, 66)):
    """Noise of single-voxel pores with a wide pore in it: one long chain the
    phases give up after the wide pore's, and enough distinct values that the
    loop's rank sort scans in scratch."""
    rng = np.random.default_rng(seed)
    img = S.random_image(shape, 0.7, rng)
    g = np.indices(shape)
    img[((g - np.array([8, 30, 32])[:, None, None, None]) ** 2).sum(0) < 150] = 1
    return img


def alone(ctx, img, inlet=0, outlet=1):
    seq, r2, cen, K, st = ctx.invade(img, inlet=inlet)
    tr, so = ctx.trapping(seq, outlet)
    sat, pc, _ = ctx.pc_curve(so, r2)
    return dict(seq=seq.clone(), step_r2=r2.clone(), step_centre=cen.clone(), trapped=tr.clone(), seq_out=so.clone(),
                S=sat.clone(), Pc=pc.clone(), K=K, status=st)


def same(got, want):
    assert got["status"] == want["status"] and got["K"] == want["K"]
    for k in ("seq", "step_r2", "step_centre", "trapped", "seq_out", "S", "Pc"):
        assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("odd", [1, 5])
def test_equal_images_some_on_the_loop(ibip, odd):
    """Forty samples of one size, which end together; `odd` of them go to the
    loop, the last of those without solid."""
    rng = np.random.default_rng(31)
    imgs = [S.sphere_pack((64, 62, 66), 5, 0.45, rng) for _ in range(6)] * 7
    imgs = imgs[:40 - odd]
    for i in range(odd):
        imgs.insert(3 + 7 * i, np.ones((64, 62, 66), np.uint8) if odd > 1 and i == odd - 1 else chain(40 + i))
    dev = [cuda(a) for a in imgs]
    ctx = ibip.Context(0)
    want = [alone(ctx, d) for d in dev]
    dref = O.edt(imgs[3])
    rseq, _, _, _, K = O.invade(imgs[3], dref, inlet=0)
    assert want[3]["K"] == K > 4096 and np.array_equal(want[3]["seq"].cpu().numpy(), rseq)
    assert np.array_equal(want[3]["trapped"].cpu().numpy(), O.trapping(rseq, 1)[0])
    for _ in range(4):
        for got, w in zip(ctx.invade_batched(dev, 0, 1), want):
            same(got, w)


def test_mixed_sizes_some_on_the_loop(ibip):
    imgs = [S.mixed_image(i, 4100, 24, 72) for i in range(12)]
    imgs[2:2] = [chain(51), np.ones((30, 31, 29), np.uint8)]
    imgs += [chain(52, (90, 60, 61)), np.zeros((9, 8, 7), np.uint8)]
    dev = [cuda(a) for a in imgs]
    ctx = ibip.Context(0)
    want = [alone(ctx, d, 2, 3) for d in dev]
    for got, w in zip(ctx.invade_batched(dev, 2, 3), want):
        same(got, w)


def test_cancel_covers_every_image_on_the_loop(ibip):
    """A request made before the call stops the images of the phases and all
    of those left to the loop, and is served once."""
    rng = np.random.default_rng(12)
    imgs = [np.ones((20, 22, 18), np.uint8), S.blobs((23, 22, 18), 2.0, 0.6, rng), np.ones((9, 30, 33), np.uint8),
            np.ones((12, 12, 40), np.uint8)]
    dev = [cuda(a) for a in imgs]
    ctx = ibip.Context(0)
    ctx.cancel(True)
    res = ctx.invade_batched(dev, 0, trapping=False, curve=False, check=False)
    assert all(r["status"] == ibip.ERR_CANCELLED and r["K"] == 0 for r in res)
    res = ctx.invade_batched(dev, 0, trapping=False, curve=False)
    for a, r in zip(imgs, res):
        assert r["status"] == ibip.OK
        assert np.array_equal(r["seq"].cpu().numpy(), O.invade(a, O.edt(a), inlet=0)[0])


def test_images_on_the_loop_run_side_by_side(ibip):
    """Sixteen chains in a batch take far less than sixteen times one."""
    ctx = ibip.Context(0)
    dev = [cuda(chain(60 + i)) for i in range(16)]

    def seconds(imgs):
        ctx.invade_batched(imgs, 0, trapping=False, curve=False)
        torch.cuda.synchronize()
        t = time.perf_counter()
        ctx.invade_batched(imgs, 0, trapping=False, curve=False)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    assert seconds(dev) < 0.5 * 16 * seconds(dev[:1])
