"""The work a program gives this library, as cases for timing and comparing outputs.

One case is one deposit as a user's program calls it (``paper_1612_09491_gb300``): particles of a
Lagrangian lattice (or explicit tetrahedra) onto a uniform grid or onto an octree built from
them.  Inputs are synthetic and made on the GPU from the seed: Zel'dovich-displaced lattices
(P(k) ~ k^index, the rms displacement in lattice spacings), optionally with collapsed regions,
and random explicit tetrahedra.

``listed`` names the cases; ``draw`` gives more of the same ranges; ``prepare`` makes a case's
inputs; ``run`` is one pass; ``work`` is what a pass cannot do without; ``exact`` evaluates the
same deposit in float64 with plain torch (its own clip and its own tree).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1612_09491_gb300 as pse


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def _uniform(name, n, g, index=-2.0, rms=1.0, precision=1, periodic=True, reuse=False, slab_of=0):
    c = {"kind": "uniform", "n0": n[0], "n1": n[1], "n2": n[2], "g0": g[0], "g1": g[1], "g2": g[2],
         "index": index, "rms": rms, "precision": precision, "periodic": periodic, "reuse": reuse,
         "slab_of": slab_of}
    return dict(c, name=name) if name else c


def _octree(name, n, bc, max_level, index=-2.0, rms=1.5, halos=0, slab=0):
    c = {"kind": "octree", "n0": n[0], "n1": n[1], "n2": n[2], "bc": bc, "max_level": max_level, "index": index,
         "rms": rms, "halos": halos, "slab": slab}
    return dict(c, name=name) if name else c


def _tets(name, count, g, lo, hi, slivers):
    c = {"kind": "tets", "count": count, "g": g, "size_lo": lo, "size_hi": hi, "slivers": slivers}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest calls (a test box, one region of a survey of many): latency and launches count
        _uniform("uniform-16c-grid32", (16,) * 3, (32,) * 3, rms=0.5),
        # the plain workload, in a loop over snapshots that keeps its output and workspace
        _uniform("uniform-32c-grid64", (32,) * 3, (64,) * 3, rms=0.5, reuse=True),
        # the ordinary call: two cells per lattice spacing, some shell crossing, default options
        _uniform("uniform-128c-grid256", (128,) * 3, (256,) * 3, rms=2.0, reuse=True),
        # odd sizes on every axis, an open (zoom-in) lattice, compensated FP32 accumulation
        _uniform("ragged-open-comp", (90, 65, 77), (181, 130, 93), rms=1.5, precision=2, periodic=False),
        # few particles on a fine grid (images of a low-resolution run): large tetrahedra,
        # mostly cells inside them
        _uniform("fine-48c-grid384", (48,) * 3, (384,) * 3, rms=1.0, reuse=True),
        # many particles on a coarse grid (power spectra, quick looks): most tetrahedra meet a
        # few cells only
        _uniform("coarse-256c-grid128", (256,) * 3, (128,) * 3, rms=1.5, reuse=True),
        # the adaptive path, tree built from the tetrahedra's sizes and then the deposit, at the
        # headline workload's geometry (two finest cells per spacing)
        _octree("octree-256c-bc32", (256,) * 3, 32, 4, rms=1.5),
        # the same field with collapsed regions: a tree with leaves on several levels
        _octree("halos-256c-bc64", (256,) * 3, 64, 4, rms=1.5, halos=8),
        # strongly shell-crossed (a late snapshot): slivers, a quarter of the clips in FP64
        _octree("crossed-128c-bc16", (128,) * 3, 16, 3, index=-1.5, rms=3.4),
        # positions in pinned host memory, streamed in z-slabs
        _octree("streamed-192c-bc32", (192,) * 3, 32, 4, rms=1.3, slab=32),
        # explicit tetrahedra of widely spread sizes
        _tets("tets-60k-grid128", 60000, 128, 0.05, 12.0, 0.02),
        # every step in FP64 (reference runs)
        _uniform("fp64-48c-grid96", (48,) * 3, (96,) * 3, rms=1.0, precision=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _axes(rng, n):
    return tuple(max(4, int(round(n * rng.uniform(0.88, 1.12)))) for _ in range(3))


def _pairs_per_tet(r):
    """Cells a tetrahedron of a lattice with r cells per spacing meets: Kuhn tetrahedra have
    volume r^3/6, projections r^2/2 and widths r along each axis."""
    return r ** 3 / 6 + 1.5 * r ** 2 + 3 * r + 1


def draw(rng):
    kind = rng.choice(["uniform"] * 5 + ["crossed", "octree", "octree", "streamed", "tets", "fp64"])
    if kind in ("uniform", "crossed", "fp64"):
        while True:
            n = _axes(rng, _log(rng, 14, 56 if kind == "fp64" else 150))
            r = _log(rng, 0.5, 3.0 if kind == "fp64" else 8.0)
            g = tuple(max(4, int(round(a * r))) for a in n)
            m = (n[0] * n[1] * n[2]) ** (1 / 3)
            pairs = 6 * n[0] * n[1] * n[2] * _pairs_per_tet(r)
            if g[0] * g[1] * g[2] <= 1 << 27 and pairs <= {"uniform": 6e8, "crossed": 6e7, "fp64": 1e7}[kind]:
                break
        if kind == "crossed":
            return _uniform("", n, g, index=-1.5, rms=round(_log(rng, 0.3, 1.0) * m ** 0.25, 3),
                            precision=rng.choice([1, 1, 2]), reuse=rng.random() < 0.5)
        rms = round(_log(rng, 0.05, 0.2) * m ** 0.5, 3)
        if kind == "fp64":
            return _uniform("", n, g, rms=rms, precision=0, periodic=rng.random() < 0.8)
        return _uniform("", n, g, rms=rms, precision=rng.choice([1, 1, 1, 2]), periodic=rng.random() < 0.75,
                        reuse=rng.random() < 0.5, slab_of=rng.choice([0, 0, 0, 4]))
    if kind in ("octree", "streamed"):
        # with collapsed regions: a finer tree, whose field stops refining at level 3
        halos = rng.choice([0, 0, 4, 8])
        while True:
            n = _axes(rng, _log(rng, 40, 110 if halos else 176))
            m = (n[0] * n[1] * n[2]) ** (1 / 3)
            bc = rng.choice([8, 16, 24, 32])
            level = min(4, max(1, int(round(math.log2(_log(rng, 1.0, 3.0) * m / bc)))))
            if halos:
                level = 4
            # mean edges in cells, level by level, away from the size rule's threshold (the bin
            # edge at 2.37 cells), so that a case has one tree whatever its seed
            edge = [1.26 * bc * 2 ** a / m for a in range(level)]
            if all(e < 1.9 or e > 2.9 for e in edge) and (not halos or edge[2] < 1.9 and 2.9 < edge[3] < 5.0):
                break
        return _octree("", n, bc, level, rms=round(_log(rng, 0.05, 0.12) * m ** 0.5, 3), halos=halos,
                       slab=rng.randint(5, 48) if kind == "streamed" else 0)
    return _tets("", int(_log(rng, 1000, 80000)), rng.randint(24, 160), 0.05, round(_log(rng, 1.0, 12.0), 2),
                 rng.choice([0.0, 0.02, 0.1]))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _positions(case, seed):
    """float32 [n2*n1*n0, 3] positions, x fastest (particle i + n0 (j + n1 k)): wrapped into [0, 1)
    on periodic lattices, as displaced on open ones (some lie outside the grid)."""
    n = (case["n0"], case["n1"], case["n2"])
    dev, f64 = "cuda", torch.float64
    gen = _generator(seed)
    wk = torch.fft.rfftn(torch.randn((n[2], n[1], n[0]), generator=gen, device=dev, dtype=f64))
    k = [torch.fft.rfftfreq(n[0], d=1.0 / n[0], device=dev, dtype=f64).view(1, 1, -1),
         torch.fft.fftfreq(n[1], d=1.0 / n[1], device=dev, dtype=f64).view(1, -1, 1),
         torch.fft.fftfreq(n[2], d=1.0 / n[2], device=dev, dtype=f64).view(-1, 1, 1)]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    wk *= k2 ** (0.25 * case["index"])
    wk[0, 0, 0] = 0.0
    for a in range(3):
        if n[a] % 2 == 0:
            wk *= (k[a].abs() != n[a] // 2).to(f64)
    psi = [torch.fft.irfftn(wk * (1j * k[a] / k2), s=(n[2], n[1], n[0])) for a in range(3)]
    rms = math.sqrt(sum(float((p * p).mean()) for p in psi))
    scale = case["rms"] / (n[0] * n[1] * n[2]) ** (1 / 3) / max(rms, 1e-300)
    x = torch.empty((n[2], n[1], n[0], 3), device=dev, dtype=f64)
    for a in range(3):
        shape = [1, 1, 1]
        shape[2 - a] = n[a]
        x[..., a] = psi[a] * scale + (torch.arange(n[a], device=dev, dtype=f64) / n[a]).view(shape)
    x = x.view(-1, 3)
    for h in range(case.get("halos", 0)):
        # a collapsed region: offsets scaled by 0.35 inside radius 0.1, back to 1 at 0.16.  Eight
        # places half a box apart, each in the middle of a level-3 node
        c = torch.tensor([(3 + 8 * ((h >> a) & 1)) / 16 for a in range(3)], device=dev, dtype=f64)
        d = x - c
        d -= torch.round(d)
        r = d.norm(dim=1, keepdim=True).clamp_min(1e-12)
        s = torch.where(r < 0.1, torch.full_like(r, 0.35), (0.035 + (r - 0.1) * (0.125 / 0.06)) / r)
        x = x + d * torch.where(r < 0.16, s - 1.0, torch.zeros_like(r))
    if not case.get("periodic", True):
        return x.float().contiguous()
    pos = torch.remainder(x, 1.0).float()
    pos[pos >= 1.0] = 0.0
    return pos.contiguous()


def _explicit(case, seed):
    """float32 [T, 4, 3] vertices (box units) and float64 [T] masses: random shapes, sizes spread
    evenly in the logarithm, a share of them flattened to slivers."""
    gen, dev, f64 = _generator(seed), "cuda", torch.float64
    t, g = case["count"], case["g"]
    lo, hi = math.log(case["size_lo"]), math.log(case["size_hi"])
    size = torch.exp(lo + (hi - lo) * torch.rand((t, 1, 1), generator=gen, device=dev, dtype=f64))
    shape = torch.rand((t, 4, 3), generator=gen, device=dev, dtype=f64) - 0.5
    thin = torch.rand((t, 1, 1), generator=gen, device=dev, dtype=f64) < case["slivers"]
    flat = torch.tensor([1.0, 1.0, 1e-3], device=dev, dtype=f64)
    shape = torch.where(thin, shape * flat, shape)
    centre = torch.rand((t, 1, 3), generator=gen, device=dev, dtype=f64)
    verts = (centre + shape * size / g).float().contiguous()
    mass = 0.5 + torch.rand(t, generator=gen, device=dev, dtype=f64)
    return verts, mass


def _cube_ids(case):
    """The cube layers of the second of `slab_of` ranks that share the lattice."""
    from paper_1612_09491_gb300 import shard
    nc = [case["n%d" % a] - (0 if case["periodic"] else 1) for a in range(3)]
    k0, k1 = shard.slab_bounds(nc[2], case["slab_of"], 1)
    return shard.slab_cube_ids(nc, k0, k1)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "tets":
        s["verts"], s["mass"] = _explicit(case, seed)
        return s
    s["n"] = (case["n0"], case["n1"], case["n2"])
    pos = _positions(case, seed)
    if case["kind"] == "octree" and case["slab"]:
        s["pos"] = torch.empty(pos.shape, dtype=pos.dtype, pin_memory=True)
        s["pos"].copy_(pos)
        return s
    s["pos"] = pos
    if case["kind"] == "uniform":
        s["grid"] = (case["g0"], case["g1"], case["g2"])
        if case["slab_of"]:
            s["ids"] = torch.from_numpy(_cube_ids(case)).cuda()
        if case["reuse"]:
            s["out"] = torch.empty(s["grid"][::-1], dtype=torch.float64, device="cuda")
            s["ws"] = torch.empty(pse.workspace_size(), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "tets":
        return pse.deposit_tets(state["verts"], state["mass"], case["g"])
    if case["kind"] == "octree":
        n, bc, level = state["n"], case["bc"], case["max_level"]
        if case["slab"]:
            tree = pse.build_octree_streamed(state["pos"], n, bc, level, case["slab"])
            mass = pse.deposit_octree_streamed(state["pos"], n, tree, case["slab"])
        else:
            tree = pse.build_octree_from_tet_sizes(state["pos"], n, bc, level)
            mass = pse.deposit_octree(state["pos"], n, tree)
        return {"leaves": tree.leaves(), "mass": mass}
    schedule = pse.PSE_THREAD_PER_TET if case["precision"] == pse.PSE_FP64_PLAIN else pse.PSE_WARP_COOPERATIVE
    return pse.deposit_uniform(state["pos"], state["n"], state["grid"], periodic=case["periodic"],
                               precision=case["precision"], schedule=schedule, cube_ids=state.get("ids"),
                               out=state.get("out"), workspace=state.get("ws"))


def work(case):
    """Bytes: the inputs read once and the masses written once.  Operations: 200 per tetrahedron
    (volume, planes, bounds) and 1000 per (tetrahedron, cell) pair that overlaps (four faces cut
    by the cell's planes and integrated), the pairs from the undisplaced lattice's geometry."""
    if case["kind"] == "tets":
        lo, hi, t = case["size_lo"], case["size_hi"], case["count"]
        span = math.log(hi / lo)
        # E[s^k] of sizes even in the logarithm; a random tetrahedron in a unit cube has volume
        # 1/72, projections 1/9 and widths 3/5 on average
        m = [(hi ** k - lo ** k) / (k * span) for k in (1, 2, 3)]
        pairs = t * (m[2] / 72 + 3 * m[1] / 9 + 3 * m[0] * 0.6 + 1)
        return {"bytes": t * 56.0 + 8.0 * case["g"] ** 3, "flops": 200.0 * t + 1000.0 * pairs}
    n = [case["n%d" % a] for a in range(3)]
    m = (n[0] * n[1] * n[2]) ** (1 / 3)
    tets = 6.0 * n[0] * n[1] * n[2]
    if case["kind"] == "uniform":
        cells = float(case["g0"] * case["g1"] * case["g2"])
        r = cells ** (1 / 3) / m
        if case["slab_of"]:
            tets /= case["slab_of"]
    else:
        # a node is refined while the mean edge (1.26 spacings) is below two of its cells
        level = 0
        while level < case["max_level"] and 1.26 * case["bc"] * 2 ** level / m < 2.0:
            level += 1
        r = case["bc"] * 2 ** level / m
        cells = float((case["bc"] * 2 ** level) ** 3)
    return {"bytes": 12.0 * n[0] * n[1] * n[2] + 8.0 * cells, "flops": tets * (200.0 + 1000.0 * _pairs_per_tet(r))}


# ---------------------------------------------------------------------------------------------
# the same deposit in float64, plain torch
# ---------------------------------------------------------------------------------------------
_PATHS = torch.tensor([[1, 3], [1, 5], [2, 3], [2, 6], [4, 5], [4, 6]])  # corners visited between 000 and 111


def _lattice_tets(case, seed):
    """float64 [T, 4, 3] unwrapped vertices (box units) of every tetrahedron."""
    n = (case["n0"], case["n1"], case["n2"])
    periodic = case.get("periodic", True)
    x = _positions(case, seed).double().view(n[2], n[1], n[0], 3)
    nc = n if periodic else tuple(a - 1 for a in n)
    corner = []
    for c in range(8):
        y = torch.roll(x, shifts=(-(c >> 2), -((c >> 1) & 1), -(c & 1)), dims=(0, 1, 2))
        y = y[:nc[2], :nc[1], :nc[0]].reshape(-1, 3)
        if c and periodic:
            d = y - corner[0]
            y = y - (d >= 0.5).double() + (d < -0.5).double()
        corner.append(y)
    corner = torch.stack(corner, 1)
    paths = _PATHS.to(x.device)
    idx = torch.cat([torch.zeros_like(paths[:, :1]), paths, torch.full_like(paths[:, :1], 7)], 1)
    t = corner[:, idx.reshape(-1)].view(-1, 6, 4, 3)
    if case.get("slab_of"):
        t = t[torch.from_numpy(_cube_ids(case)).to(t.device)]
    return t.reshape(-1, 4, 3)


def _cut(a, b, axis, plane, keep_above):
    """Cut closed chains of segments a -> b (float64 [..., E, 3]) by a coordinate plane; the
    closing segment is appended, dropped segments become points on the plane."""
    s = (1.0 if keep_above else -1.0)
    ca, cb = (a[..., axis] - plane) * s, (b[..., axis] - plane) * s
    ia, ib = ca >= 0, cb >= 0
    den = ca - cb
    t = (ca / torch.where(den == 0, torch.ones_like(den), den)).clamp(0.0, 1.0)
    p = a + t[..., None] * (b - a)
    p[..., axis] = plane
    out, ent = (ia & ~ib), (~ia & ib)
    first = (p * out[..., None]).sum(-2, keepdim=True)
    second = (p * ent[..., None]).sum(-2, keepdim=True)
    na = torch.where(ia[..., None], a, p)
    nb = torch.where(ib[..., None], b, p)
    return torch.cat([na, first], -2), torch.cat([nb, second], -2)


def _above(a, b, o, level):
    """Integral of max(z - level, 0) over the xy projection of closed chains (signed): fans from
    o, a point of each chain's plane."""
    a, b = _cut(a, b, 2, level, True)
    u, v = a - o, b - o
    cr = u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]
    return (0.5 * cr * ((a[..., 2] + b[..., 2] + o[..., 2]) / 3.0 - level)).sum(-1)


def _overlap(v):
    """Volume of positively oriented tetrahedra v (float64 [N, 4, 3]) inside the unit cell [0,1)^3."""
    faces = torch.tensor([[1, 2, 3], [0, 3, 2], [0, 1, 3], [0, 2, 1]], device=v.device)
    tri = v[:, faces]  # [N, 4, 3, 3]
    a, b = tri, torch.roll(tri, -1, dims=2)
    for axis in (0, 1):
        a, b = _cut(a, b, axis, 0.0, True)
        a, b = _cut(a, b, axis, 1.0, False)
    o = tri[:, :, :1]
    return (_above(a, b, o, 0.0) - _above(a, b, o, 1.0)).sum(-1)


_CHUNK = 1 << 20
_MOST_PAIRS = 1.2e8


def _deposit64(verts, mass, g, periodic):
    """Cell masses [g2 * g1 * g0] of tetrahedra given in box units, or None if too many pairs."""
    dev = verts.device
    scale = torch.tensor([float(a) for a in g], device=dev, dtype=torch.float64)
    gi = torch.tensor(list(g), device=dev)
    v = verts * scale
    e = v[:, 1:] - v[:, :1]
    det = torch.linalg.det(e) if len(v) < 1000 else (e[:, 0] * torch.linalg.cross(e[:, 1], e[:, 2])).sum(-1)
    flip = det < 0
    v[flip] = v[flip][:, [0, 2, 1, 3]]
    lo = v.amin(1).floor().long()
    dim = v.amax(1).floor().long() - lo + 1
    lo[det == 0] = v[det == 0].mean(1).floor().long()
    dim[det == 0] = 1
    count = dim.prod(1)
    if float(count.sum()) > _MOST_PAIRS:
        return None
    out = torch.zeros(g[0] * g[1] * g[2], device=dev, dtype=torch.float64)
    rho = torch.where(det == 0, torch.zeros_like(det), 6.0 * mass / det.abs().clamp_min(1e-300))
    ends = count.cumsum(0)
    total = int(ends[-1])
    for p0 in range(0, total, _CHUNK):
        p = torch.arange(p0, min(total, p0 + _CHUNK), device=dev)
        t = torch.searchsorted(ends, p, right=True)
        r = p - (ends[t] - count[t])
        d = dim[t]
        cell = lo[t] + torch.stack([r % d[:, 0], (r // d[:, 0]) % d[:, 1], r // (d[:, 0] * d[:, 1])], 1)
        m = rho[t] * _overlap(v[t] - cell[:, None].double())
        m = torch.where(count[t] == 1, mass[t], m)
        if periodic:
            cell = torch.remainder(cell, gi)
        else:
            m = m * ((cell >= 0) & (cell < gi)).all(1)
            cell = torch.minimum(cell.clamp_min(0), gi - 1)
        out.index_add_(0, cell[:, 0] + g[0] * (cell[:, 1] + g[1] * cell[:, 2]), m)
    return out


def _tree64(verts, bc, max_level, threshold=2.0):
    """Leaves (level, x, y, z), depth first: a node is refined while the lower median of its
    tetrahedra's mean edge (64 bins of log10 over [-3, 3) cells) is below the threshold."""
    i, j = torch.triu_indices(4, 4, 1, device=verts.device)
    edge = (verts[:, i] - verts[:, j]).norm(dim=-1).mean(1)
    cen = torch.remainder(verts.mean(1), 1.0)
    refine = []
    for level in range(max_level):
        nn = 1 << level
        c = (cen * nn).long().clamp(0, nn - 1)
        node = c[:, 0] + nn * (c[:, 1] + nn * c[:, 2])
        b = ((torch.log10(edge * bc * nn) + 3.0) * (64.0 / 6.0)).floor().long().clamp(0, 63)
        h = torch.bincount(node * 64 + b, minlength=64 * nn ** 3).view(-1, 64)
        cum = h.cumsum(1)
        k = (cum[:, -1:] - 1).div(2, rounding_mode="floor")
        med = (cum <= k).sum(1).clamp_max(63)
        low = 10.0 ** (-3.0 + 6.0 * med.double() / 64.0)
        refine.append(((cum[:, -1] > 0) & (low < threshold)).cpu().numpy())
    leaves = []

    def visit(level, x, y, z):
        if level == max_level or not refine[level][x + (y + (z << level) << level)]:
            leaves.append((level, x, y, z))
            return
        for c in range(8):
            visit(level + 1, 2 * x + (c & 1), 2 * y + ((c >> 1) & 1), 2 * z + (c >> 2))

    visit(0, 0, 0, 0)
    return np.array(leaves, dtype=np.int64)


def exact(case, seed):
    if case["kind"] == "tets":
        verts, mass = _explicit(case, seed)
        m = _deposit64(verts.double(), mass, (case["g"],) * 3, True)
        return None if m is None else m.view((case["g"],) * 3)
    tets = 6.0 * case["n0"] * case["n1"] * case["n2"]
    if tets > 6e6:
        return None
    verts = _lattice_tets(case, seed)
    mass = torch.full((len(verts),), 1.0 / tets, device=verts.device, dtype=torch.float64)
    if case["kind"] == "uniform":
        g = (case["g0"], case["g1"], case["g2"])
        m = _deposit64(verts, mass, g, case["periodic"])
        return None if m is None else m.view(g[::-1])
    leaves, bc = _tree64(verts, case["bc"], case["max_level"]), case["bc"]
    out = torch.empty((len(leaves), bc, bc, bc), device=verts.device, dtype=torch.float64)
    for level in sorted(set(leaves[:, 0].tolist())):
        g = bc << level
        m = _deposit64(verts, mass, (g,) * 3, True)
        if m is None:
            return None
        m = m.view(g, g, g)
        for i in np.nonzero(leaves[:, 0] == level)[0]:
            x, y, z = (int(a) * bc for a in leaves[i, 1:])
            out[i] = m[z:z + bc, y:y + bc, x:x + bc]
    return {"leaves": None, "mass": out}
