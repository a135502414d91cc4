"""A server of more slots than clusters of 16 CTAs fit the GPU: small jobs
take smaller clusters, and every result equals the calls made for it alone."""
import numpy as np
import pytest

from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("slots", [20, 48])
def test_many_slots(slots):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    ctx = ibip.Context(0)
    kinds = [torch.from_numpy(S.mixed_image(i, 7100, 14, 52)).cuda() for i in range(14)]
    kinds.append(torch.from_numpy(S.blobs((104, 103, 101), 3.0, 0.6, np.random.default_rng(1))).cuda())   # a full cluster
    want = []
    for d in kinds:
        seq, r2, cen, K, st = ctx.invade(d)
        tr, so = ctx.trapping(seq, 1)
        want.append((seq, r2, cen, tr, so))
    jobs = [i % len(kinds) for i in range(60)]
    srv = ibip.Server(ctx, 1 << 31, slots)
    try:
        tickets = [srv.submit(kinds[i], 0, 1) for i in jobs]
        res = [srv.wait(t, timeout=600) for t in tickets]
    finally:
        srv.close()
    for i, r in zip(jobs, res):
        assert r["status"] == 0
        for k, w in zip(("seq", "step_r2", "step_centre", "trapped", "seq_out"), want[i]):
            assert torch.equal(r[k], w), k
