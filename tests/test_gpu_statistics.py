"""vd_status counts each cell's events once: in the build that makes the cell,
by the kernel that finishes it."""
import numpy as np
import pytest

from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EVENTS = ("fp64_fallbacks", "fp64_ambiguous", "refined_vertices", "refined_volumes", "empty_cells", "overflow_cells",
          "ambiguous_cells")


def build(x, w=None, part=None):
    from paper_2605_06408_gb300 import vd

    ctx = vd.Context(0)
    if part:
        ctx.set_partition(*part)
    ctx.build(torch.from_numpy(x).cuda(), None if w is None else torch.from_numpy(w).cuda(), W.UNIT_BOX)
    return ctx


@pytest.mark.parametrize("n", [3001, 60_002])
@pytest.mark.parametrize("weighted", [False, True])
def test_parts_add_up_to_the_whole(n, weighted):
    """Four consecutive cells share a warp from 192 sites per SM on, also where
    two parts meet between them."""
    x = W.mixture(n, 31)
    w = W.power_weights(x, 32) if weighted else None
    whole = build(x, w).status()
    assert whole["refined_vertices"] > 0 and whole["fp64_fallbacks"] > 0
    parts = [build(x, w, (p, 13)).status() for p in range(13)]
    for k in EVENTS:
        assert sum(s[k] for s in parts) == whole[k], k


@pytest.mark.parametrize("seed", [1, 3])
def test_an_ambiguous_cell_is_listed_once(seed):
    """Heavy-tailed weights: cells that outgrow both kernels, some of whose FP64
    signs stay inside their bound."""
    x = W.mixture(1_000_000, seed)
    ctx = build(x, W.power_weights(x, seed + 1))
    st = ctx.status()
    assert st["overflow_cells"] > 0 and st["fp64_ambiguous"] >= st["ambiguous_cells"]
    assert st["ambiguous_cells"] == len(ctx.ambiguous_cells())
