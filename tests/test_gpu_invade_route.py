"""Which schedule an invasion takes (one-CTA loop or value phases) and that
both give the oracle's run (Section 2.1): open images on either side of the
line, balls of r2 >= 1024 on the phases, short continuations."""
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


def open_image(shape, n, seed):
    img = np.ones(shape, np.uint8)
    img.reshape(-1)[np.random.default_rng(seed).choice(img.size, n, replace=False)] = 0
    return img


def expected_on_the_loop(img, d):
    """The rule: few steps (0.48 of the voxels of value 1) on few large balls."""
    m = float(d.max())
    return 0.48 * (d == 1).sum() < 100.0 * m ** 0.8 and img.sum() < 70.0 * m ** 1.5


def same(got, ref):
    seq, r2, cen, K, st = got
    assert K == ref[4] and np.array_equal(seq.cpu().numpy(), ref[0])
    assert np.array_equal(r2.cpu().numpy(), ref[1]) and np.array_equal(cen.cpu().numpy(), ref[2])


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("img,loop", [
    (open_image((60, 70, 65), 40, 4), True),
    (open_image((100, 101, 99), 100, 5), True),
    (S.blobs((14, 12, 13), 3.0, 0.6, np.random.default_rng(1)), True),
    (S.blobs((24, 25, 23), 2.0, 0.6, np.random.default_rng(2)), True),
    (S.blobs((50, 48, 51), 7.0, 0.65, np.random.default_rng(3)), True),
    (S.sphere_pack((47, 57, 50), 6, 0.49, np.random.default_rng(4)), False),
    (S.blobs((32, 33, 31), 1.5, 0.6, np.random.default_rng(2)), False),
    (open_image((64, 64, 64), 1000, 6), False),
    (open_image((200, 190, 201), 1000, 7), False),   # r2 >= 1024 on the phases
])
def test_route_and_result(ibip, img, loop, shared):
    d = O.edt(img)
    assert expected_on_the_loop(img, d) == loop
    ref = O.invade(img, d, inlet=1)
    ctx = ibip.Context(0)
    ctx.set_shared_device(shared)
    got = ctx.invade(cuda(img), cuda(d), inlet=1)
    assert (ctx.invade_stats()["items"] > 0) == loop
    same(got, (ref[0], ref[1], ref[2], None, ref[4]))


def test_open_images_of_a_batch(ibip):
    """A batch keeps them on the phases, one cluster each."""
    imgs = [open_image((60, 70, 65), 40, 4), open_image((90, 80, 85), 60, 8), open_image((20, 31, 22), 5, 9)]
    ctx = ibip.Context(0)
    out = ctx.invade_batched([cuda(a) for a in imgs], 1, trapping=False, curve=False)
    for a, r in zip(imgs, out):
        ref = O.invade(a, O.edt(a), inlet=1)
        same((r["seq"], r["step_r2"], r["step_centre"], r["K"], r["status"]), ref[:3] + (None, ref[4]))


@pytest.mark.parametrize("step", [700, 4096, 4097])
def test_continued_in_short_runs(ibip, step):
    img = S.sphere_pack((70, 66, 72), 5, 0.42, np.random.default_rng(3))
    d = O.edt(img)
    ref = O.invade(img, d, inlet=0)
    dev, dt = cuda(img), cuda(d)
    ctx = ibip.Context(0)
    got = ctx.invade_ex(dev, dt, max_steps=step)
    while got[4] == ibip.ERR_STEP_LIMIT:
        assert got[3] < ref[4]
        got = ctx.invade_ex(dev, dt, resume_from=got[:3], max_steps=step)
        if step <= 4096:   # the loop: its two parts count their steps
            st = ctx.invade_stats()
            assert st["items"] + st["tiny_steps"] > 0
    same(got, ref[:3] + (None, ref[4]))
