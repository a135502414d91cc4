"""A cancel request while a value phase runs a group of thousands of steps:
the call returns soon after it, with a valid invasion of the phases done
that continues to the uninterrupted result (ibip_cancel)."""
import threading
import time

import numpy as np
import pytest

from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_request_in_a_long_group():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    img = torch.from_numpy(S.sphere_pack((200, 200, 200), 4, 0.36, np.random.default_rng(0))).cuda()
    ctx = ibip.Context(0)
    d = ctx.edt(img)

    def run(out):
        torch.cuda.synchronize()
        out["t0"] = time.perf_counter()
        out["r"] = ctx.invade(img, d, check=False)
        out["t1"] = time.perf_counter()

    full = {}
    run(full)
    run(full)
    seq_f, r2_f, cen_f, K_f, _ = full["r"]
    whole = full["t1"] - full["t0"]
    assert ctx.invade_stats()["items"] == 0 and whole > 0.05
    for _ in range(3):
        out = {}
        t = threading.Thread(target=run, args=(out,))
        t.start()
        time.sleep(0.5 * whole)
        asked = time.perf_counter()
        ctx.cancel(True)
        t.join(timeout=60)
        assert not t.is_alive()
        seq, r2, cen, K, st = out["r"]
        assert st == ibip.ERR_CANCELLED and K < K_f
        assert out["t1"] - asked < 0.15 * whole
        assert torch.equal(seq, torch.where(seq_f > K, -1, seq_f))
        assert torch.equal(r2, r2_f[:K]) and torch.equal(cen, cen_f[:K])
    seq, r2, cen, K, st = ctx.invade_ex(img, d, resume_from=(seq, r2, cen))
    assert st == ibip.OK and K == K_f and torch.equal(seq, seq_f) and torch.equal(r2, r2_f) and torch.equal(cen, cen_f)
