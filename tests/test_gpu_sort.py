"""The radix sort at the edges of its tiles (1,024 keys, 3,072 from 2^18 sites
on): a site that a pass loses, doubles or misplaces changes neighbour lists,
which must equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 3073, 262_143, 262_144, 262_145])
def test_sizes_around_the_tiles(n):
    from paper_2605_06408_gb300 import vd

    x = W.uniform(n, n)
    res = vd.Context(0).build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    cells = np.arange(n) if n < 4000 else np.unique(W.rng_for(n).integers(0, n, 400))
    ref = oracle.cells(x, cells=cells)
    off, nb = res.offsets.cpu().numpy(), res.neighbors.cpu().numpy()
    for q, i in enumerate(cells):
        assert np.array_equal(nb[off[i]:off[i + 1]], ref["nbrs"][q]), f"cell {i}"
    vol = res.volume.double().cpu().numpy()
    assert np.all(np.abs(vol[cells] - ref["vol"]) <= 1e-5 * ref["vol"])
    # every cell once: FP32 volumes of the box's parts, each within 1e-5 of its own
    assert abs(vol.sum() - 1.0) <= 1e-5
