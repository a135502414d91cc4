"""The invasion by value phases (csrc/flood.cu) at the sizes where its parts
change over: whole GPU and one cluster, groups on lanes, warps, CTAs and bit
planes, balls stamped by the whole team, images it gives up or does not take
(long chains, no solid, values beyond the 15-bit state), step limits inside
a phase, resumed runs.  Everything is a whole number and equals the oracle's
run (Section 2.1) bit for bit."""
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


def few_solids(shape, n, seed):
    """An open image: n solid voxels, so balls are large and groups long."""
    rng = np.random.default_rng(seed)
    img = np.ones(shape, np.uint8)
    img.reshape(-1)[rng.choice(img.size, n, replace=False)] = 0
    return img


def slabs(shape, gap):
    """Parallel plates `gap` apart: sheets of equal values."""
    img = np.zeros(shape, np.uint8)
    for y in range(0, shape[1], gap + 1):
        img[:, y:y + gap, :] = 1
    img[shape[0] // 2] = 1
    return img


CASES = {
    "grid blobs": lambda: S.blobs((131, 127, 137), (3.0, 5.0, 3.0), 0.6, np.random.default_rng(1)),
    "grid pack": lambda: S.sphere_pack((129, 128, 130), 7, 0.42, np.random.default_rng(2)),
    "cluster pack": lambda: S.sphere_pack((90, 61, 77), 6, 0.45, np.random.default_rng(3)),
    "open": lambda: few_solids((60, 70, 65), 40, 4),           # r2 >= 1024: stamped by the whole team
    "open grid": lambda: few_solids((140, 130, 129), 30, 5),
    "noise": lambda: S.random_image((40, 41, 43), 0.7, np.random.default_rng(6)),     # a chain: given up
    "noise grid": lambda: S.random_image((130, 129, 131), 0.62, np.random.default_rng(7)),
    "slab 1": lambda: slabs((33, 40, 64), 1),                  # sheets of dt2 = 1
    "slab 3": lambda: slabs((33, 40, 64), 3),
    "flat": lambda: S.blobs((1, 190, 211), 3.0, 0.6, np.random.default_rng(8)),
    "line": lambda: S.random_image((1, 1, 300), 0.97, np.random.default_rng(9)),
    "column": lambda: S.blobs((170, 9, 1), 2.0, 0.6, np.random.default_rng(10)),
    "no solid": lambda: np.ones((9, 10, 11), np.uint8),
    "one solid": lambda: few_solids((30, 31, 29), 1, 11),
    "beyond 15 bits": lambda: few_solids((400, 9, 9), 1, 12),  # dt2 above 32767
}


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_equals_the_oracle(ibip, name, shared):
    img = CASES[name]()
    ctx = ibip.Context(0)
    ctx.set_shared_device(shared)   # shared: one cluster whatever the size
    d = O.edt(img)
    for inlet in ((0, 5) if img.size < 100000 else (2,)):
        rseq, rr2, rcen, rst, rK = O.invade(img, d, inlet=inlet)
        seq, r2, cen, K, st = ctx.invade(cuda(img), cuda(d), inlet=inlet)
        assert K == rK and st == rst
        assert np.array_equal(seq.cpu().numpy(), rseq)
        assert np.array_equal(r2.cpu().numpy(), rr2) and np.array_equal(cen.cpu().numpy(), rcen)


@pytest.mark.parametrize("frac", [0.0, 0.01, 0.2, 0.5, 0.999, 1.0])
def test_step_limits_and_resuming(ibip, frac):
    img = S.blobs((64, 66, 59), (2.0, 3.0, 2.0), 0.62, np.random.default_rng(21))
    d = O.edt(img)
    rseq, rr2, rcen, rst, rK = O.invade(img, d, inlet=0)
    ctx = ibip.Context(0)
    k = int(round(frac * rK))
    seq, r2, cen, K, st = ctx.invade(cuda(img), cuda(d), max_steps=k)
    cut = rseq.copy()
    cut[cut > k] = -1
    assert K == k and st == (ibip.OK if k == rK else ibip.ERR_STEP_LIMIT)
    assert np.array_equal(seq.cpu().numpy(), cut)
    assert np.array_equal(r2.cpu().numpy(), rr2[:k]) and np.array_equal(cen.cpu().numpy(), rcen[:k])
    seq, r2, cen, K, st = ctx.invade_ex(cuda(img), cuda(d), resume_from=(seq, r2, cen))
    assert K == rK and st == ibip.OK
    assert np.array_equal(seq.cpu().numpy(), rseq)
    assert np.array_equal(r2.cpu().numpy(), rr2) and np.array_equal(cen.cpu().numpy(), rcen)


def test_short_step_arrays_and_unaligned_buffers(ibip):
    """Step arrays shorter than the run, and a sequence image and distances
    that start 4 bytes off a 16-byte boundary."""
    img = S.blobs((50, 47, 53), 2.0, 0.6, np.random.default_rng(22))
    d = O.edt(img)
    rseq, rr2, rcen, rst, rK = O.invade(img, d, inlet=0)
    ctx = ibip.Context(0)
    n = img.size
    sbuf = torch.empty(n + 8, dtype=torch.int32, device="cuda")
    dbuf = torch.empty(n + 8, dtype=torch.int32, device="cuda")
    seq, dd = sbuf[1:n + 1].view(img.shape), dbuf[3:n + 3].view(img.shape)
    dd.copy_(cuda(d))
    cap = rK // 3
    out = ctx.invade(cuda(img), dd, capacity=cap, seq=seq, check=False)
    assert out[3] == rK and out[4] == ibip.ERR_ARG
    assert np.array_equal(seq.cpu().numpy(), rseq) and np.array_equal(out[1].cpu().numpy(), rr2[:cap])
