"""The squared EDT at lines whose staged columns cross the 48 KB that a
launch may use without asking (384 entries are 48 KB to the byte), in both
column passes and with rows on and off 16-byte boundaries."""
import numpy as np
import pytest

import oracle as O
from paper_2101_03240_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [255, 256, 257, 383, 384, 385])
@pytest.mark.parametrize("nz", [5, 8, 36])
@pytest.mark.parametrize("axis", [0, 1])
def test_column_sizes(n, nz, axis):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2101_03240_gb300 import ibip
    shape = (n, 4, nz) if axis == 0 else (4, n, nz)
    img = S.blobs(shape, 2.0, 0.6, np.random.default_rng(n + nz))
    d = ibip.context().edt(torch.from_numpy(img).cuda())
    assert np.array_equal(d.cpu().numpy(), O.edt(img))
