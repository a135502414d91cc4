"""The widest path by maximum spanning forest (csrc/maximin.cu) on fields
without structure, where most neighbour pairs join two basins and the edges
outgrow their list (every pair is then scanned again each round).  Whole
numbers, equal to the oracle's trapping and opening (Sections 2.2.3 and
2.4.1)."""
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
    return ibip.context()


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("shape", [(33, 40, 47), (1, 90, 100), (100, 1, 1), (64, 64, 64)])
@pytest.mark.parametrize("outlet", range(6))
def test_widest_path_noise(ctx, shape, outlet):
    rng = np.random.default_rng(outlet + shape[0])
    N = int(np.prod(shape))
    seq = (rng.permutation(N) + 1).reshape(shape).astype(np.int32)
    u = rng.random(shape)
    seq[u < 0.15] = -1
    seq[u > 0.9] = 0
    trapped, out = ctx.trapping(cuda(seq), outlet)
    rt, ro = O.trapping(seq, outlet)
    assert np.array_equal(trapped.cpu().numpy(), rt) and np.array_equal(out.cpu().numpy(), ro)
    img = (seq != 0).astype(np.uint8)
    d = np.where(img, rng.integers(1, 40, shape), 0).astype(np.int32)
    T = [38, 30, 22, 14, 9, 4, 1]
    lev, cnt = ctx.morph_drainage(cuda(img), cuda(d), T, inlet=outlet)
    rlev, rcnt = O.morph_drainage(img, d, T, inlet=outlet)
    assert np.array_equal(lev.cpu().numpy(), rlev) and cnt == rcnt.tolist()
