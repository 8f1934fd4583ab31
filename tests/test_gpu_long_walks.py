"""Cells that see a whole empty box: their walks end in the large-cell pass."""
import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,side", [(20_000, 1e-3), (60_000, 1e-3), (60_000, 1e-2), (200_000, 1e-3)])
def test_a_tight_cluster_in_a_large_box(n, side):
    from paper_2605_06408_gb300 import vd

    x = (0.5 + side * (W.uniform(n, 6) - 0.5)).astype(np.float32)
    x = np.unique(x, axis=0)
    ctx = vd.Context(0)
    res = ctx.build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    if n >= 60_000:
        assert ctx.status()["overflow_cells"] > 0
    cells = torch.argsort(res.volume, descending=True)[:100].cpu().numpy()
    ref = oracle.cells(x, cells=cells)
    off, nb = res.offsets.cpu().numpy(), res.neighbors.cpu().numpy()
    for q, i in enumerate(cells):
        assert np.array_equal(nb[off[i]:off[i + 1]], ref["nbrs"][q]), f"cell {i}"
    vol, cen = res.volume.double().cpu().numpy()[cells], res.centroid.double().cpu().numpy()[cells]
    assert np.all(np.abs(vol - ref["vol"]) <= 1e-5 * ref["vol"])
    assert np.all(np.linalg.norm(cen - ref["cen"], axis=1) <= 1e-5 * np.linalg.norm(ref["cen"], axis=1))
