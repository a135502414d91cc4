"""The dilations of the opening on bit planes (csrc/opening.cu) where their
parts change over: tiles and words with remainders, the radii where the
window widens (16 voxels) and the EDT passes take over (32), levels beyond
one launch, dilation bounds that rise again.  Whole numbers, equal to the
oracle's opening (Section 2.4.1)."""
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


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def cavity(shape, n, seed):
    """An open image with n solid voxels: radii of half the edge."""
    rng = np.random.default_rng(seed)
    img = np.ones(shape, np.uint8)
    img.reshape(-1)[rng.choice(img.size, n, replace=False)] = 0
    return img


def blobs(shape, seed):
    return S.blobs(shape, (3.0, 5.0, 3.0), 0.6, np.random.default_rng(seed))


def check(ctx, img, d, T, inlet, Td=None):
    lev, cnt = ctx.morph_drainage(cuda(img), cuda(d), T, inlet=inlet, dilate_levels=Td)
    rlev, rcnt = O.morph_drainage(img, d, T, inlet=inlet, dilate_levels=Td)
    assert np.array_equal(lev.cpu().numpy(), rlev) and cnt == rcnt.tolist()


@pytest.mark.parametrize("shape", [(16, 32, 32), (17, 33, 33), (15, 31, 16), (40, 41, 15), (49, 63, 95), (1, 70, 130),
                                   (70, 1, 65), (5, 6, 200)])
def test_tiles(ctx, shape):
    """Tiles and words with remainders; 15 voxels along z: the EDT passes."""
    img = blobs(shape, sum(shape))
    d = O.edt(img)
    for inlet in (0, 3, 5):
        check(ctx, img, d, list(range(max(int(d.max()), 1), 0, -1))[:60], inlet)


@pytest.mark.parametrize("top", [1100, 1024, 300, 289])
def test_reaches(ctx, top):
    """Radii around the largest of either window and of the tables, few
    centres (stamped rows) and many (whole tiles)."""
    img = cavity((90, 80, 84), 9, top)
    d = O.edt(img)
    assert d.max() >= top
    check(ctx, img, d, [top + 1, top, top - 1, top - 2, 286, 120, 7, 2, 1], 1)
    check(ctx, img, d, [top - 1], 4)


@pytest.mark.parametrize("seed", range(4))
def test_rising_bounds(ctx, seed):
    """Dilation bounds in any order, across both windows and the EDT passes."""
    rng = np.random.default_rng(seed)
    img = blobs((50, 67, 71), 20 + seed)
    d = O.edt(img)
    T = sorted({int(t) for t in rng.integers(1, int(d.max()) + 2, 40)}, reverse=True)
    Td = [int(t) for t in rng.choice([1, 2, 3, 9, 40, 100, 288, 289, 290, 900, 1024, 1025, 2000], len(T))]
    check(ctx, img, d, T, seed, Td)


def test_many_levels(ctx):
    """Levels beyond one launch, and beyond 254 with EDT levels among them."""
    img = cavity((80, 70, 75), 6, 3)
    d = O.edt(img)
    top = int(d.max())
    assert top > 1100
    check(ctx, img, d, list(range(top, top - 8, -1)) + list(range(600, 250, -1)), 2)
    check(ctx, img, d, list(range(1000, 900, -1)), 2)
