"""Plane slots taken again: a cell that more planes cut than the one-per-warp
kernel holds (128), though it has few faces at any time."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [9024, 16384])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_nearer_planes_one_after_another(n, seed):
    """vd_cells_noalloc reads the sites in index order after the nearest of
    each residue modulo 32. Here the sites of residue 0 close in on site 0 in
    index order (each cuts a ball that the planes before it leave whole, but
    for those on the side of the nearest one), and the others stay far away."""
    from paper_2605_06408_gb300 import vd

    rng = W.rng_for(seed)
    x = rng.random((4 * n, 3))
    x = x[np.linalg.norm(x - 0.5, axis=1) > 0.45][:n]
    assert len(x) == n
    near = np.arange(32, n, 32)
    u = rng.standard_normal((len(near), 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x[near] = 0.5 + u * np.linspace(0.4, 0.1, len(near))[:, None]
    x[0] = 0.5
    x = x.astype(np.float32)
    assert len(near) // 2 > 128 - 6
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    xs = torch.from_numpy(x).cuda()
    counts, status = (torch.full((m,), -7, dtype=torch.int32, device="cuda") for m in (n, 1))
    nbrs = torch.full((n, 64), -7, dtype=torch.int32, device="cuda")
    vol, cen = torch.empty(n, device="cuda"), torch.empty(n, 3, device="cuda")
    rc = vd.load_library().vd_cells_noalloc(p(xs), None, n, vd._box(W.UNIT_BOX), p(counts), p(nbrs), p(vol), p(cen),
                                            p(status), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == vd.VD_OK
    ref = oracle.cells(x, cells=np.array([0]))
    c = int(counts[0])
    assert np.array_equal(nbrs[0, :c].cpu().numpy(), ref["nbrs"][0])
    assert abs(float(vol[0]) - ref["vol"][0]) <= 1e-5 * ref["vol"][0]
