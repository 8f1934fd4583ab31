"""The kernels that walk the 8-wide tree, four cells per warp (from 192 sites
per SM on) and one, against the oracle where they can go wrong: the last
sites of a warp, sets that meet inside one, lists longer than a row, cells at
and past the capacities, cells that reach far."""
import numpy as np
import pytest

import oracle
from paper_2605_06408_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vdmod():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_06408_gb300 import vd

    return vd


def threshold():
    return 192 * torch.cuda.get_device_properties(0).multi_processor_count


def check(res, ref, cells, first=0):
    off, nb = res.offsets.cpu().numpy(), res.neighbors.cpu().numpy()
    vol, cen = res.volume.double().cpu().numpy(), res.centroid.double().cpu().numpy()
    for q, i in enumerate(cells):
        assert np.array_equal(nb[off[first + i]:off[first + i + 1]], ref["nbrs"][q]), f"cell {first + i}"
    idx = first + np.asarray(cells)
    assert np.all(np.abs(vol[idx] - ref["vol"]) <= 1e-5 * ref["vol"] + 1e-30)
    assert np.all(np.linalg.norm(cen[idx] - ref["cen"], axis=1) <= 1e-5 * np.linalg.norm(ref["cen"], axis=1))


@pytest.mark.parametrize("extra", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("weighted", [False, True])
def test_last_sites_of_a_warp(vdmod, extra, weighted):
    n = threshold() + extra
    x = W.mixture(n, 5 + extra)
    w = W.gaussian_weights(x, 6) if weighted else None
    res = vdmod.Context(0).build(torch.from_numpy(x).cuda(), None if w is None else torch.from_numpy(w).cuda(), W.UNIT_BOX)
    # a sample, and the sites that sort last (the upper corner of the box)
    cells = np.unique(np.concatenate([W.rng_for(7).integers(0, n, 300), np.argsort(x.min(1))[-8:]]))
    check(res, oracle.cells(x, w, cells=cells), cells)


@pytest.mark.parametrize("warm", [0, 2])
def test_sets_that_meet_inside_a_warp(vdmod, warm):
    rng = W.rng_for(11)
    sizes = np.concatenate([rng.integers(1, 60, 1000), [threshold() // 3, 1, 2, 17]])
    assert sizes.sum() >= threshold()
    offsets = np.concatenate([[0], np.cumsum(sizes)])
    xs, ws, flags, boxes = [], [], [], []
    for s, m in enumerate(sizes):
        lo = rng.uniform(-1, 1, 3).astype(np.float32)
        hi = (lo + rng.uniform(0.5, 2, 3)).astype(np.float32)
        xs.append((lo + (hi - lo) * W.uniform(int(m), 100 + s)).astype(np.float32))
        d = float(np.cbrt(1.0 / m))
        ws.append((0.1 * d * d * rng.standard_normal(int(m))).astype(np.float32))
        flags.append(s % 2)
        boxes.append((lo, hi))
    res = vdmod.Context(0, {"warm_start": warm}).build_batched(
        torch.from_numpy(np.concatenate(xs)).cuda(), torch.from_numpy(np.concatenate(ws)).cuda(), offsets, boxes, flags)
    for s in np.concatenate([rng.integers(0, 1000, 250), np.arange(1000, len(sizes))]):
        m = int(sizes[s])
        cells = np.arange(m) if m < 100 else rng.integers(0, m, 100)
        ref = oracle.cells(xs[s], ws[s] if flags[s] else None, boxes[s], cells=cells)
        check(res, ref, cells, int(offsets[s]))


@pytest.mark.parametrize("faces", [60, 70, 110, 126, 180])
@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("tape", [0, 1])
def test_cells_of_many_faces(vdmod, faces, large, tape):
    """A site inside a sphere of others: up to and past a row of 64 and the
    one-per-warp kernel's 128 planes and 192 vertices."""
    i = np.arange(faces) + 0.5
    phi, th = np.arccos(1 - 2 * i / faces), np.pi * (1 + 5 ** 0.5) * i
    s = np.stack([np.cos(th) * np.sin(phi), np.sin(th) * np.sin(phi), np.cos(phi)], 1)
    s = s * (0.2 + 0.002 * W.rng_for(3).random((faces, 1)))
    bg = W.uniform(threshold() + 4000 if large else 2000, 4)
    bg = bg[np.linalg.norm(bg - 0.5, axis=1) > 0.3]
    x = np.concatenate([[[0.5, 0.5, 0.5]], 0.5 + s, bg]).astype(np.float32)
    ctx = vdmod.Context(0, {"tape": tape})
    res = ctx.build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    cells = np.arange(faces + 200)
    ref = oracle.cells(x, cells=cells)
    assert ref["counts"][0] >= 0.9 * faces
    check(res, ref, cells)
    # the adjoint of a loss on those cells alone, from the tape or re-clipped: as large a tolerance as the
    # adjoint's own tests take (1e-4 of the largest component)
    c, d = W.loss_coefficients(len(x), 2)
    c[len(cells):] = 0
    d[len(cells):] = 0
    gp, _ = ctx.backward(torch.from_numpy(c).float().cuda(), torch.from_numpy(d).float().cuda(), want_weights=False)
    gr, _ = ctx.backward(torch.from_numpy(c).float().cuda(), torch.from_numpy(d).float().cuda(), want_weights=False,
                         recompute=True)
    assert float((gp - gr).abs().max()) <= 1e-4 * float(gr.abs().max())


@pytest.mark.parametrize("n", [20_000, 60_000])
def test_cells_that_reach_far(vdmod, n):
    """Tight clusters: the cells at their edges extend across the empty box,
    past the walk limits of both kernels."""
    x = W.clustered(n, 3, 9)
    res = vdmod.Context(0).build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    cells = torch.argsort(res.volume, descending=True)[:200].cpu().numpy()
    check(res, oracle.cells(x, cells=cells), cells)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 97, 4097, 16384])
def test_without_a_tree(vdmod, n):
    """vd_cells_noalloc reads the sites 64 a step, after the nearest of every 32nd."""
    import ctypes

    x = W.uniform(n, 90 + n)
    w = W.gaussian_weights(x, 3) if n > 2 else None
    p = lambda t: None if t is None else ctypes.c_void_p(t.data_ptr())
    xs, ws = torch.from_numpy(x).cuda(), None if w is None else torch.from_numpy(w).cuda()
    counts, status = (torch.full((m,), -7, dtype=torch.int32, device="cuda") for m in (n, 1))
    nbrs = torch.full((n, 64), -7, dtype=torch.int32, device="cuda")
    vol, cen = torch.empty(n, device="cuda"), torch.empty(n, 3, device="cuda")
    rc = vdmod.load_library().vd_cells_noalloc(p(xs), p(ws), n, vdmod._box(W.UNIT_BOX), p(counts), p(nbrs), p(vol), p(cen),
                                               p(status), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == vdmod.VD_OK and int(status.item()) == vdmod.VD_OK
    cells = np.arange(n) if n < 200 else np.unique(W.rng_for(n).integers(0, n, 300))
    ref = oracle.cells(x, w, cells=cells)
    counts, nbrs, vol = counts.cpu().numpy(), nbrs.cpu().numpy(), vol.double().cpu().numpy()
    for q, i in enumerate(cells):
        assert np.array_equal(nbrs[i, :counts[i]], ref["nbrs"][q]), f"cell {i}"
        assert np.all(nbrs[i, counts[i]:] == -7), f"cell {i}: written past its row"
    assert np.all(np.abs(vol[cells] - ref["vol"]) <= 1e-5 * ref["vol"] + 1e-30)


@pytest.mark.parametrize("n", [3_000, 60_000])
@pytest.mark.parametrize("what", ["nan", "inf", "equal", "few"])
def test_inputs_that_cull_nothing(vdmod, n, what):
    """Sites without a finite position are reported, and copies of one position
    leave one cell, without walks of the whole tree for each of them."""
    x = W.uniform(n, 3)
    if what in ("nan", "inf"):
        x[::2] = np.nan if what == "nan" else np.inf
        with pytest.raises(vdmod.VdError) as e:
            vdmod.Context(0).build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
        assert e.value.code == vdmod.VD_ERR_INVALID_ARG
        return
    distinct = 1 if what == "equal" else 20
    x = x[np.arange(n) % distinct]
    res = vdmod.Context(0).build(torch.from_numpy(x).cuda(), None, W.UNIT_BOX)
    vol = res.volume.double().cpu().numpy()
    assert np.all(vol[distinct:] == 0) and abs(vol[:distinct].sum() - 1.0) <= 1e-5
    if distinct > 1:
        check(res, oracle.cells(x[:distinct]), np.arange(distinct))
