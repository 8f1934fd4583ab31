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


@pytest.mark.parametrize("norm2,faces", [(26, 72), (101, 168)])
@pytest.mark.parametrize("n", [3000, 60_000])
def test_an_ambiguous_cell_is_listed_once(n, norm2, faces):
    """A site with sites on all integer points at one distance around it: many
    planes through one vertex, exactly. 72 faces outgrow the four-per-warp
    kernel, 168 the one-per-warp kernel too."""
    g = np.arange(-10, 11)
    p = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    p = p[(p * p).sum(1) == norm2]
    assert len(p) == faces
    bg = W.uniform(n, 4)
    bg = bg[np.linalg.norm(bg - 0.5, axis=1) > 0.3]
    x = np.concatenate([[[0.5, 0.5, 0.5]], 0.5 + p / 64.0, bg]).astype(np.float32)
    ctx = build(x)
    cells = ctx.ambiguous_cells()
    assert 0 in cells
    assert ctx.status()["ambiguous_cells"] == len(np.unique(cells))
