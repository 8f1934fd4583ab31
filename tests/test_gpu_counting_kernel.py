"""The warp-per-cell kernel of the ablation modes, the event counters and plain
FP32 in each of its capacities, starts and leaf sizes. With counters = 1 it
builds the same cells as the kernels of the default modes."""
import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def inputs():
    x = W.mixture(4000, 51)
    return x, [(w, oracle.cells(x, w, max_nbrs=8192)) for w in (None, W.power_weights(x, 52))]


CAPACITIES = [{"verts_per_lane": v, "queue_per_lane": q} for v in (2, 4) for q in (1, 2, 4, 8)]
OTHERS = [{"warm_start": 1}, {"warm_start": 2}, {"warm_start": 1, "verts_per_lane": 4, "queue_per_lane": 1}, {"leaf_size": 1},
          {"leaf_size": 32}, {"leaf_size": 8, "warm_start": 2}, {"warps_per_block": 8, "blocks_per_sm": 2}]


@pytest.mark.parametrize("cfg", CAPACITIES + OTHERS)
def test_knobs_match_the_oracle(inputs, cfg):
    from paper_2605_06408_gb300 import vd

    x, refs = inputs
    ctx = vd.Context(0, dict(cfg, counters=1))
    for w, ref in refs:
        res = ctx.build(torch.from_numpy(x).cuda(), None if w is None else torch.from_numpy(w).cuda(), W.UNIT_BOX)
        off, nb = res.offsets.cpu().numpy(), res.neighbors.cpu().numpy()
        for i in range(len(x)):
            assert np.array_equal(nb[off[i]:off[i + 1]], ref["nbrs"][i]), f"cell {i}"
        vol, cen = res.volume.double().cpu().numpy(), res.centroid.double().cpu().numpy()
        assert np.all(np.abs(vol - ref["vol"]) <= 1e-5 * ref["vol"] + 1e-30)
        assert np.all(np.linalg.norm(cen - ref["cen"], axis=1) <= 1e-5 * np.linalg.norm(ref["cen"], axis=1))
        st = ctx.status()
        assert st["error"] == 0 and st["failed_cells"] == 0 and st["clips"] > 0
