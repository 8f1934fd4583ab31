"""The radix sort at the edges that its kernels have: 2,048 keys in one block,
tiles of 1,024 keys above that and of 3,072 from 2^18 on (86 of them hold
264,192). A site that a pass loses has no row, one that it doubles or misplaces
breaks the symmetry of the lists."""
import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2047, 2048, 2049, 3071, 3072, 3073, 264_191, 264_192, 264_193])
def test_every_site_once(n):
    from paper_2605_06408_gb300 import vd

    x = W.uniform(n, n)
    res = vd.Context(0).build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    off, nb = res.offsets.cpu().numpy().astype(np.int64), res.neighbors.cpu().numpy().astype(np.int64)
    src = np.repeat(np.arange(n), np.diff(off))
    assert np.diff(off).min() >= 1
    assert np.array_equal(np.sort(src * n + nb), np.sort(nb * n + src))
    vol = res.volume.double().cpu().numpy()
    assert vol.min() > 0 and abs(vol.sum() - 1.0) <= 1e-5
    # the sites that sort last (the upper corner of the box), and a sample
    cells = np.unique(np.concatenate([np.argsort(x.min(1))[-64:], W.rng_for(n).integers(0, n, 200)]))
    ref = oracle.cells(x, cells=cells)
    for q, i in enumerate(cells):
        assert np.array_equal(nb[off[i]:off[i + 1]], ref["nbrs"][q]), f"cell {i}"
    assert np.all(np.abs(vol[cells] - ref["vol"]) <= 1e-5 * ref["vol"])
