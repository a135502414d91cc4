"""Paper-literal invasion (Section 2.1): steps whose points are more than the
entries of a list that the walk keeps in shared memory (16, 8 from values of
1,536, 4 from 3,072) and no more than one warp takes (21), queued together by
one warp or by many.  Against the oracle, repeated."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    return ibip.Context(0)


def duct(shape, loose=0, seed=0):
    """Pore with a solid plane at the far end of x (values of whole
    cross-sections are equal) and `loose` solid voxels."""
    img = np.ones(shape, np.uint8)
    img[-1] = 0
    rng = np.random.default_rng(seed)
    for _ in range(loose):
        img[tuple(int(rng.integers(0, n)) for n in shape)] = 0
    return img


CASES = [((64, 4, 5), 0), ((63, 3, 7), 0), ((60, 2, 3), 0), ((45, 4, 4), 0), ((44, 3, 3), 0), ((30, 4, 5), 0), ((25, 3, 7), 0),
         ((64, 26, 27), 2), ((62, 40, 40), 6), ((50, 30, 31), 4), ((40, 40, 40), 60), ((34, 60, 60), 200)]


@pytest.mark.parametrize("shape,loose", CASES)
def test_steps_larger_than_the_ring(ctx, shape, loose):
    img = duct(shape, loose, 7)
    d = O.edt(img)
    seq, cstep, r2, cnt, st, K = O.invade_literal(img, d, 0)
    kept = 16 if d.max() < 1536 else 8 if d.max() < 3072 else 4
    assert ((cnt > kept) & (cnt <= 21)).sum() >= 10
    dev, dt = torch.from_numpy(img).cuda(), torch.from_numpy(d).cuda()
    for _ in range(12):
        gseq, gcst, gr2, gcnt, gK, gst = ctx.invade_literal(dev, dt, inlet=0)
        assert gK == K and gst == st
        assert np.array_equal(gcst.cpu().numpy(), cstep) and np.array_equal(gseq.cpu().numpy(), seq)
        assert np.array_equal(gr2.cpu().numpy(), r2) and np.array_equal(gcnt.cpu().numpy(), cnt)
