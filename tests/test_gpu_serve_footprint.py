"""Jobs that take most of what ibip_job_footprint reserves: dense and sparse
noise (chains left to the one-CTA loop, as many basins as voxels of pore),
open images, sizes whose tables fall on the ends of the arena's pieces.  Each
runs in a server of exactly its footprint and equals the calls made alone."""
import numpy as np
import pytest

from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def checkerboard(shape):
    g = np.indices(shape).sum(0)
    return (g % 2).astype(np.uint8)


def near_solid(shape):
    """Pore everywhere but on a sparse lattice: every value small."""
    img = np.ones(shape, np.uint8)
    img[::2, ::2, ::2] = 0
    return img


RNG = np.random.default_rng(3)
CASES = {
    "checkerboard": checkerboard((64, 64, 64)), "lattice": near_solid((64, 66, 62)),
    "noise 0.1": S.random_image((96, 96, 96), 0.1, RNG), "noise 0.5": S.random_image((64, 64, 64), 0.5, RNG),
    "noise 0.7": S.random_image((64, 64, 64), 0.7, RNG), "noise 0.86": S.random_image((80, 64, 64), 0.86, RNG),
    "noise 0.97": S.random_image((128, 128, 96), 0.97, RNG), "open": S.random_image((128, 128, 128), 0.99999, RNG),
    "line": S.random_image((1, 1, 4000), 0.9, RNG), "blobs": S.blobs((100, 120, 90), 3.0, 0.6, RNG),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fits_its_footprint(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    ctx = ibip.Context(0)
    img = torch.from_numpy(CASES[name]).cuda()
    seq, r2, cen, K, st = ctx.invade(img)
    tr, so = ctx.trapping(seq, 1)
    sat, pc, _ = ctx.pc_curve(so, r2)
    srv = ibip.Server(ctx, ibip.job_footprint(img.shape), 1)
    try:
        for _ in range(2):
            r = srv.wait(srv.submit(img, 0, 1), timeout=600)
            assert r["status"] == 0 and r["K"] == K and r["mem_used"] <= r["mem_reserved"]
            for k, w in (("seq", seq), ("step_r2", r2), ("step_centre", cen), ("trapped", tr), ("seq_out", so), ("S", sat),
                         ("Pc", pc)):
                assert torch.equal(r[k], w), k
    finally:
        srv.close()
