"""What is timed: builds of 3D Voronoi and power diagrams through the public entry points.

Each case is one call that a program makes again and again on new sites: a
forward build (`vd.Context.build`, `build_batched`), a training step
(`vd.cells` or `vd.mesh_cells` with the gradients of a loss), or the
allocation-free entry point `vd_cells_noalloc`. Inputs are made on the GPU
from the seed alone, shaped like the generators of
`paper_2605_06408_gb300/workloads.py`; the context a program keeps is made
beforehand. Weights, where a case has them, are the power weights of its sites.

Case fields: kind (forward, batched, train, mesh, noalloc), dist (uniform,
gradient, mixture, clustered, surfaces), weights (none, gauss, lognormal), n, and for
contexts leaf and warm (vd_config.leaf_size, warm_start); batched: nsets, lo, hi.
"""
import ctypes
import math
import random

import torch

from paper_2605_06408_gb300 import vd

BOX = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
DEV = "cuda:0"


def _c(name, kind, dist, weights, n, leaf=16, warm=0, **more):
    return dict(name=name, kind=kind, dist=dist, weights=weights, n=n, leaf=leaf, warm=warm, **more)


def listed():
    return [
        # a handful of seeds, rebuilt after every edit of an interactive program: launches and latency
        _c("few_sites", "forward", "uniform", "none", 500),
        # the small benchmark configuration (white noise), default settings
        _c("uniform_10k", "forward", "uniform", "none", 10_000),
        # a power diagram with mild weights (packing, material microstructure), odd size
        _c("gauss_weights_37k", "forward", "uniform", "gauss", 37_451),
        # a scan-like set: clusters of very different shapes and densities, default settings
        _c("mixture_200k", "forward", "mixture", "none", 200_003),
        # the same at the million-site configuration of the benchmark, with the KNN start that the tuner picks
        _c("mixture_1M", "forward", "mixture", "none", 1_000_000, leaf=32, warm=2),
        # heavy-tailed weights: most of the time goes to a few very large cells and half of the cells are empty
        _c("power_1M", "forward", "mixture", "lognormal", 1_000_000, leaf=32, warm=1),
        # the largest diagram of the benchmark: samples of surfaces, as a radiance-field scene has them
        _c("surfaces_20M", "forward", "surfaces", "none", 20_000_000, leaf=32, warm=2),
        # many independent sets of ragged sizes in one call, half of them with weights
        _c("batched_64", "batched", "mixture", "lognormal", 0, leaf=32, warm=2, nsets=64, lo=1_000, hi=200_000),
        # a step of site optimisation (equal volumes, centroidal sites): forward, loss and gradients
        _c("train_voronoi_300k", "train", "gradient", "none", 300_000),
        # the same on a small weighted diagram, weights optimised too
        _c("train_power_10k", "train", "uniform", "gauss", 10_007),
        # a step whose loss also sees the cell vertices (mesh extraction and rendering)
        _c("mesh_train_12k", "mesh", "gradient", "none", 12_000),
        # the entry point for callers that must not allocate
        _c("noalloc_4k", "noalloc", "uniform", "none", 4_001),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "forward", "batched", "train", "train", "mesh", "noalloc"])
    dist = rng.choice(["uniform", "gradient", "mixture", "clustered", "surfaces"])
    weights = rng.choice(["none", "none", "gauss", "lognormal"])
    leaf, warm = rng.choice([(16, 0), (16, 0), (32, 2), (32, 1), (32, 0), (8, 2)])
    if kind == "batched":
        lo = _size(rng, 200, 5_000)
        return dict(kind=kind, dist=dist, weights=weights, n=0, leaf=leaf, warm=warm,
                    nsets=rng.randint(3, 200), lo=lo, hi=_size(rng, 2 * lo, 50_000))
    if kind == "noalloc":
        return dict(kind=kind, dist="uniform", weights=rng.choice(["none", "gauss"]), n=_size(rng, 200, 16_384), leaf=16, warm=0)
    hi = {"forward": 3_000_000, "train": 1_000_000, "mesh": 200_000}[kind]
    if weights == "lognormal":
        hi = min(hi, 1_000_000)
    return dict(kind=kind, dist=dist, weights=weights, n=_size(rng, 300, hi), leaf=leaf, warm=warm)


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _truncated(point_of, m):
    """m points of point_of(indices), those outside the box drawn again."""
    p = point_of(torch.arange(m, device=DEV))
    while True:
        bad = (~((p >= 0.0) & (p <= 1.0)).all(1)).nonzero()[:, 0]
        if bad.numel() == 0:
            return p
        p[bad] = point_of(bad)


def _gaussians(g, n, clusters, lo, hi, background):
    """Points around `clusters` centres (per-axis sigma 10^U(lo, hi)) and a uniform background; and their mean spacing."""
    centre = _rand(g, clusters, 3)
    sigma = 10.0 ** (lo + (hi - lo) * _rand(g, clusters, 3))
    m = n - int(round(background * n))
    lab = torch.arange(m, device=DEV) % clusters
    p = _truncated(lambda i: centre[lab[i]] + sigma[lab[i]] * _randn(g, i.numel(), 3), m)
    p = torch.cat([p, _rand(g, n - m, 3)])
    rho = torch.full((n,), float(max(n - m, 1)), device=DEV, dtype=torch.float64)
    for k in range(clusters):
        q = ((p - centre[k]) / sigma[k]).square().sum(1)
        rho += (m / clusters) * torch.exp(-0.5 * q) / ((2.0 * math.pi) ** 1.5 * sigma[k].prod())
    return p, rho


def _surfaces(g, n):
    """Nested Gaussian shells (sigma 1e-2 .. 1e-5) around spheres, tori and height fields, and 1% background."""
    host = random.Random(int(torch.randint(1 << 30, (1,), generator=g, device=DEV)))
    nsurf, n_bg = 32, int(round(0.01 * n))
    parts, left = [_rand(g, n_bg, 3)], n - n_bg
    for s in range(nsurf):
        m = left // (nsurf - s)
        left -= m
        sig = 10.0 ** (-2.0 - (torch.arange(m, device=DEV) % 4).double())
        kind = s % 3
        if kind == 0:
            c = torch.tensor([host.uniform(0.2, 0.8) for _ in range(3)], device=DEV, dtype=torch.float64)
            r = host.uniform(0.05, 0.3)

            def point(i):
                u = _randn(g, i.numel(), 3)
                u /= u.norm(dim=1, keepdim=True)
                return c + u * (r + sig[i] * _randn(g, i.numel()))[:, None]
        elif kind == 1:
            c = torch.tensor([host.uniform(0.3, 0.7) for _ in range(3)], device=DEV, dtype=torch.float64)
            big = host.uniform(0.1, 0.25)
            small = big * host.uniform(0.15, 0.5)
            rot = torch.linalg.qr(_randn(g, 3, 3))[0]

            def point(i):
                a, b = 2.0 * math.pi * _rand(g, i.numel()), 2.0 * math.pi * _rand(g, i.numel())
                t = small + sig[i] * _randn(g, i.numel())
                q = torch.stack([(big + t * b.cos()) * a.cos(), (big + t * b.cos()) * a.sin(), t * b.sin()], 1)
                return c + q @ rot.T
        else:
            z0, ax = host.uniform(0.3, 0.7), host.randrange(3)
            amp = [host.uniform(0.01, 0.05) for _ in range(4)]
            freq = [(host.choice((-1, 1)) * host.uniform(2, 12), host.choice((-1, 1)) * host.uniform(2, 12)) for _ in range(4)]
            phase = [host.uniform(0, 2 * math.pi) for _ in range(4)]

            def point(i):
                u, v = _rand(g, i.numel()), _rand(g, i.numel())
                h, hu, hv = torch.full_like(u, z0), torch.zeros_like(u), torch.zeros_like(u)
                for a, (fu, fv), ph in zip(amp, freq, phase):
                    t = fu * u + fv * v + ph
                    h += a * t.sin()
                    hu += a * fu * t.cos()
                    hv += a * fv * t.cos()
                nrm = torch.stack([-hu, -hv, torch.ones_like(u)], 1)
                q = torch.stack([u, v, h], 1) + nrm * (sig[i] * _randn(g, i.numel()) / nrm.norm(dim=1))[:, None]
                return q.roll(ax, 1)
        parts.append(_truncated(point, m))
    return torch.cat(parts)


def _sites(g, dist, weights, n):
    """(sites float32 [n, 3], weights float32 [n] or None) of one set."""
    rho = None
    if dist == "uniform":
        p = _rand(g, n, 3)
    elif dist == "gradient":
        p = _rand(g, n, 3)
        p[:, 0] = p[:, 0].sqrt()
    elif dist == "mixture":
        p, rho = _gaussians(g, n, 64, -3.0, -1.0, 0.10)
    elif dist == "clustered":
        p, rho = _gaussians(g, n, 10, math.log10(0.005), math.log10(0.005), 0.0)
    else:
        p = _surfaces(g, n)
    order = torch.randperm(n, generator=g, device=DEV)
    x = p[order].float().contiguous()
    if weights == "none":
        return x, None
    rho = torch.full((n,), float(n), device=DEV, dtype=torch.float64) if rho is None else rho[order]
    if weights == "gauss":  # w ~ N(0, (d^2 / 3)^2), d the median nearest-neighbour distance
        d = ((math.log(2.0) * 0.75 / math.pi) / rho.median()) ** (1.0 / 3.0)
        return x, (_randn(g, n) * (d * d / 3.0)).float()
    # w = r^2, r = 0.2 nn exp(N(0, 1)), nn distributed as the nearest-neighbour distance at the local density
    nn = (-_rand(g, n).clamp_min(1e-300).log() * (0.75 / math.pi) / rho) ** (1.0 / 3.0)
    return x, (0.2 * nn * _randn(g, n).exp()).square().float()


def _set_sizes(case):
    k, lo, hi = case["nsets"], case["lo"], case["hi"]
    return [int(round(lo * (hi / lo) ** ((s + 0.5) / k))) for s in range(k)]


def prepare(case, seed):
    g = _gen(seed)
    n = case["n"]
    state = {"case": dict(case)}
    if case["kind"] == "batched":
        sizes = _set_sizes(case)
        random.Random(int(seed)).shuffle(sizes)
        flags, xs, ws = [], [], []
        for s, m in enumerate(sizes):
            weighted = case["weights"] != "none" and s % 2 == 1
            x, w = _sites(g, case["dist"] if s % 4 < 2 else "uniform", case["weights"] if weighted else "none", m)
            xs.append(x)
            ws.append(torch.zeros(m, device=DEV) if w is None else w)
            flags.append(1 if weighted else 0)
        state["x"], n = torch.cat(xs), sum(sizes)
        state["w"] = torch.cat(ws) if any(flags) else None
        state["offsets"] = [sum(sizes[:s]) for s in range(len(sizes) + 1)]
        state["flags"], state["boxes"] = flags, [BOX] * len(sizes)
    else:
        state["x"], state["w"] = _sites(g, case["dist"], case["weights"], n)
    if case["kind"] == "noalloc":
        state["out"] = {"counts": torch.zeros(n, dtype=torch.int32, device=DEV),
                        "neighbors": torch.zeros(n, 64, dtype=torch.int32, device=DEV),
                        "volume": torch.zeros(n, device=DEV), "centroid": torch.zeros(n, 3, device=DEV),
                        "status": torch.zeros(1, dtype=torch.int32, device=DEV)}
        state["lib"] = vd.load_library()
        return state
    state["rows"] = torch.zeros(24 * n + 64, dtype=torch.int32, device=DEV)
    grad = case["kind"] in ("train", "mesh")
    state["ctx"] = vd.Context(0, {"leaf_size": case["leaf"], "warm_start": case["warm"], "tape": int(grad)})
    state["ctx"].reserve(n, case["weights"] != "none")
    if grad:
        state["x"].requires_grad_(True)
        if state["w"] is not None:
            state["w"].requires_grad_(True)
    return state


# ---------------------------------------------------------------- one pass

def _loss(vol, cen, x, verts=None):
    """Equal volumes and sites at their cells' centroids; with a mesh, vertices near the box centre too."""
    n = x.shape[0]
    loss = (vol * n - 1.0).square().mean() + n ** (2.0 / 3.0) * (vol * (cen - x).square().sum(1)).sum()
    if verts is not None:
        loss = loss + 0.1 * (verts - 0.5).square().sum() / n
    return loss


def _keep(rows, neighbors):
    """The neighbour lists in the program's own buffer (whose size does not hang on how many there are)."""
    rows[:neighbors.shape[0]] = neighbors
    return rows


def run(state):
    case, x, w = state["case"], state["x"], state["w"]
    kind = case["kind"]
    if kind == "forward":
        r = state["ctx"].build(x, w, BOX)
        return {"offsets": r.offsets, "neighbors": _keep(state["rows"], r.neighbors), "volume": r.volume, "centroid": r.centroid}
    if kind == "batched":
        r = state["ctx"].build_batched(x, w, state["offsets"], state["boxes"], state["flags"] if w is not None else None)
        return {"offsets": r.offsets, "neighbors": _keep(state["rows"], r.neighbors), "volume": r.volume, "centroid": r.centroid}
    if kind == "noalloc":
        o, p = state["out"], lambda t: ctypes.c_void_p(t.data_ptr())
        box = vd.VdBox((ctypes.c_float * 3)(*BOX[0]), (ctypes.c_float * 3)(*BOX[1]))
        rc = state["lib"].vd_cells_noalloc(p(x), None if w is None else p(w), x.shape[0], box, p(o["counts"]), p(o["neighbors"]),
                                           p(o["volume"]), p(o["centroid"]), p(o["status"]),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != vd.VD_OK:
            raise vd.VdError(rc, "vd_cells_noalloc")
        return dict(o)
    wrt = [x] if w is None else [x, w]
    if kind == "train":
        vol, cen, off, nb = vd.cells(x, w, BOX, state["ctx"])
        grads = torch.autograd.grad(_loss(vol, cen, x), wrt)
        out = {"offsets": off, "neighbors": _keep(state["rows"], nb)}
    else:  # the rows of a cell's vertices come in the library's own order: the gradients and row offsets stand for them
        vol, cen, verts, off, nb, voff, _ = vd.mesh_cells(x, w, BOX, state["ctx"])
        grads = torch.autograd.grad(_loss(vol, cen, x, verts), wrt)
        out = {"offsets": off, "neighbors": _keep(state["rows"], nb), "vertex_offsets": voff}
    out.update(volume=vol.detach(), centroid=cen.detach(), grad_sites=grads[0])
    if w is not None:
        out["grad_weights"] = grads[1]
    return out


def work(case):
    """Bytes: sites and weights in, rows, volumes and centroids (and gradients) out. Flops per cell with 15.5 faces and 27
    vertices: each vertex solved (51) and checked against each face's plane (6), the planes (30 each), 81 volume tetrahedra (60
    each); a gradient adds 81 face triangles (150 each)."""
    n = sum(_set_sizes(case)) if case["kind"] == "batched" else case["n"]
    w = case["weights"] != "none"
    nnz = (8.0 if case["weights"] == "lognormal" else 15.5) * n
    cells = 0.5 * n if case["weights"] == "lognormal" else n
    b = n * (12 + (4 if w else 0)) + 4 * (n + 1) + 4 * nnz + 16 * n
    f = cells * (27 * 51 + 15.5 * 27 * 6 + 15.5 * 30 + 81 * 60)
    if case["kind"] in ("train", "mesh"):
        b += n * (16 + 12 + (4 if w else 0))
        f += cells * 81 * 150
    if case["kind"] == "mesh":
        b += 27 * n * 36
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- 64 bits

def _planes(x, w, cell, ident):
    """Normal and offset (n.v <= b, v from the cell's site) of plane `ident` (a site, or n + box face) of each cell."""
    n = x.shape[0]
    face = (ident - n).clamp_min(0)
    axis, low = face // 2, face % 2 == 1
    j = ident.clamp_max(n - 1)
    p = x[cell]
    d = x[j] - p
    fn = torch.nn.functional.one_hot(axis, 3).double() * torch.where(low, -1.0, 1.0).unsqueeze(-1).double()
    at = p.gather(-1, axis.unsqueeze(-1)).squeeze(-1)
    site = ident < n
    return (torch.where(site.unsqueeze(-1), d, fn),
            torch.where(site, 0.5 * (d.square().sum(-1) + w[cell] - w[j]), torch.where(low, at, 1.0 - at)))


def _vertices(x, w, cell, tri):
    """The point of three planes of each cell, from its site."""
    (a, ba), (b, bb), (c, bc) = (_planes(x, w, cell, tri[:, k]) for k in range(3))
    num = ba[:, None] * torch.linalg.cross(b, c) + bb[:, None] * torch.linalg.cross(c, a) + bc[:, None] * torch.linalg.cross(a, b)
    return num / (a * torch.linalg.cross(b, c)).sum(1, keepdim=True)


def _combinatorics(x, w, room=96, chunk=256):
    """(cell, planes) of every vertex of every cell: each cell is the box, cut by the site most violated at any of its vertices
    until none is."""
    n = x.shape[0]
    half = 0.5 * (x.square().sum(1) - w)
    corner = torch.tensor([[a, 2 + b, 4 + c] if (a + b + c) % 2 == 0 else [a, 4 + c, 2 + b]
                           for c in (0, 1) for b in (0, 1) for a in (0, 1)], device=DEV) + n
    found = []
    for lo in range(0, n, chunk):
        ids = torch.arange(lo, min(n, lo + chunk), device=DEV)
        tri = torch.zeros(ids.numel(), room, 3, dtype=torch.long, device=DEV)
        tri[:, :8] = corner
        live = torch.zeros(ids.numel(), room, dtype=torch.bool, device=DEV)
        live[:, :8] = True
        pos = torch.zeros(ids.numel(), room, 3, dtype=torch.float64, device=DEV)
        pos[:, :8] = _vertices(x, w, ids.repeat_interleave(8), corner.repeat(ids.numel(), 1)).view(-1, 8, 3)
        while ids.numel():
            y = pos + x[ids][:, None]
            least, at = (half - y.reshape(-1, 3) @ x.T).min(1)
            own = half[ids][:, None] - (y * x[ids][:, None]).sum(2)
            worst, v = torch.where(live, own - least.view(own.shape), -math.inf).max(1)
            cut = worst > 1e-15
            done = ~cut
            c, r = live[done].nonzero(as_tuple=True)
            found.append((ids[done][c], tri[done][c, r]))
            ids, tri, live, pos, h = ids[cut], tri[cut], live[cut], pos[cut], at.view(own.shape)[cut].gather(1, v[cut][:, None])[:, 0]
            if ids.numel() == 0:
                break
            nh, bh = _planes(x, w, ids, h)
            out = live & ((pos * nh[:, None]).sum(2) > bh[:, None])
            out.scatter_(1, v[cut][:, None], True)
            # edges between an outside and a kept vertex: directed pairs of outside vertices without their reverse
            a, b = tri, tri.roll(-1, 2)
            key = torch.where(out[:, :, None], a * (n + 6) + b, -1).flatten(1)
            rev = (b * (n + 6) + a).flatten(1)
            new = (key >= 0) & ~(rev[:, :, None] == key[:, None, :]).any(2)
            c, e = new.nonzero(as_tuple=True)
            t = torch.stack([a.flatten(1)[c, e], b.flatten(1)[c, e], h[c]], 1)
            slot = (torch.cumsum(new, 1) - 1)[c, e]
            live = live & ~out
            tri, pos = torch.cat([tri, torch.zeros_like(tri)], 1), torch.cat([pos, torch.zeros_like(pos)], 1)
            live = torch.cat([live, torch.zeros_like(live)], 1)
            tri[c, room + slot], pos[c, room + slot], live[c, room + slot] = t, _vertices(x, w, ids[c], t), True
            order = torch.argsort(live, dim=1, descending=True, stable=True)
            if int(live.sum(1).max()) > room:
                return None
            live = live.gather(1, order)[:, :room]
            tri = tri.gather(1, order[:, :, None].expand(-1, -1, 3))[:, :room]
            pos = pos.gather(1, order[:, :, None].expand(-1, -1, 3))[:, :room]
    return torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])


def exact(case, seed):
    """Volumes, centroids and gradients in 64 bits (Cramer's rule, signed tetrahedra from each site, autograd)."""
    if case["kind"] == "batched" or case["weights"] == "lognormal" or case["n"] > 13_000 or case["dist"] in ("surfaces", "clustered"):
        return None
    state = prepare(dict(case, kind="noalloc"), seed)
    x = state["x"].detach().double().requires_grad_(True)
    w = (torch.zeros(x.shape[0], device=DEV) if state["w"] is None else state["w"].detach()).double().requires_grad_(True)
    n = x.shape[0]
    with torch.no_grad():
        topology = _combinatorics(x, w)
    if topology is None:
        return None
    cell, tri = topology
    v = _vertices(x, w, cell, tri)
    # every directed edge of a face: from vertex t to the vertex of its cell that holds the reverse plane pair
    a, b = tri, tri.roll(-1, 1)
    local = torch.unique(torch.cat([cell * (n + 6) + tri[:, k] for k in range(3)]), return_inverse=True)[1].view(3, -1).T
    m = int(local.max()) + 1
    key, rev = (local * m + local.roll(-1, 1)).flatten(), (local.roll(-1, 1) * m + local).flatten()
    order = torch.argsort(key)
    hit = torch.searchsorted(key[order], rev).clamp_max(key.numel() - 1)
    u = order[hit]
    ok = key[u] == rev
    t = torch.arange(cell.numel(), device=DEV).repeat_interleave(3)
    t, u, face = t[ok], u[ok] // 3, b.flatten()[ok]
    nf, bf = _planes(x, w, cell[t], face)
    foot = nf * (bf / nf.square().sum(1))[:, None]
    det = (foot * torch.linalg.cross(v[t], v[u])).sum(1)
    vol = torch.zeros(n, device=DEV, dtype=torch.float64).index_add(0, cell[t], det / 6.0)
    mom = torch.zeros(n, 3, device=DEV, dtype=torch.float64).index_add(0, cell[t], det[:, None] * (foot + v[t] + v[u]) / 24.0)
    full = vol > 0
    cen = torch.where(full[:, None], x + mom / torch.where(full, vol, 1.0)[:, None], x)
    out = {"volume": vol.detach(), "centroid": cen.detach()}
    if case["kind"] in ("train", "mesh"):
        loss = _loss(vol, cen, x.detach(), x[cell] + v if case["kind"] == "mesh" else None)
        # the library's gradients are those of a loss on (volume, centroid, vertices), plus the loss's own on the sites
        gx, gw = torch.autograd.grad(loss, [x, w])
        gx = gx + torch.autograd.grad(_loss(vol.detach(), cen.detach(), x), x)[0]
        out["grad_sites"] = gx
        if state["w"] is not None:
            out["grad_weights"] = gw
    return out
