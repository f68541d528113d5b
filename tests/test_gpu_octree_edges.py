"""Octree deposits of tetrahedra as small as the rounding of their float32 coordinates, at leaf
and cell planes: every tetrahedron is deposited once, into a cell of the leaf array.

The lattices are 2 x 2 x 2 particles in one tight cluster, so that all 48 tetrahedra of the
periodic tessellation lie in the cluster.  Expected cells and masses follow from the positions."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1612_09491_gb300 as pse  # noqa: E402

pytestmark = pytest.mark.gpu

WARP = [pse.PSE_FP32_FP64ACC, pse.PSE_FP32_COMPENSATED]
# (precision, schedule, guard_list_cap)
PATHS = [(p, pse.PSE_WARP_COOPERATIVE, cap) for p in WARP for cap in (0, -1)] + \
    [(p, pse.PSE_THREAD_PER_TET, 0) for p in (pse.PSE_FP32_FP64ACC, pse.PSE_FP64_PLAIN)]
EIGHTHS = [(1, c & 1, (c >> 1) & 1, c >> 2) for c in range(8)]
GUARD = 4096  # cells kept around the leaf array to see writes outside it


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


def deposit(pos, tree, bc, box, **kw):
    """Leaf masses of a cluster of total mass 1, with sentinels on both sides of the leaf array."""
    n_cells = tree.n_leaves * bc ** 3
    big = torch.full((n_cells + 2 * GUARD,), 7.0, dtype=torch.float64, device="cuda")
    out = big[GUARD:GUARD + n_cells].view(tree.n_leaves, bc, bc, bc)
    p = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float32)).cuda()
    r = pse.deposit_octree(p, 2, tree, box=box, particle_mass=0.125, out=out, mass_fixup=False, **kw)
    assert bool((big[:GUARD] == 7.0).all()) and bool((big[-GUARD:] == 7.0).all())
    return (out.cpu().numpy(), r[1]) if isinstance(r, tuple) else out.cpu().numpy()


@pytest.mark.parametrize("prec,sched,cap", PATHS)
def test_single_cell_just_below_the_box(prec, sched, cap):
    """z a few 1e-20 below the box: float64 names the last leaf (of the image below), float32
    rounds the cell to the one after it."""
    rng = np.random.default_rng(2)
    pos = np.empty((8, 3))
    pos[:, :2] = 0.97 + rng.uniform(0, 0.01, (8, 2))
    pos[:, 2] = -1e-20 * rng.permutation(np.arange(1, 9))
    bc = 4
    tree = pse.octree_from_leaves(np.array(EIGHTHS, np.int32), bc, 1)
    got, st = deposit(pos, tree, bc, 1.0, precision=prec, schedule=sched, stats=True, tuning={"guard_list_cap": cap})
    want = np.zeros_like(got)
    want[7, 3, 3, 3] = 1.0
    # (compensated sums hold a cell to 2^-48 of each addend)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-12)
    assert st["single_cell_tets"] + st["degenerate_tets"] == 48 == st["overlapped_cells"]


@pytest.mark.parametrize("prec,sched,cap", PATHS)
def test_single_cell_across_a_leaf_plane(prec, sched, cap):
    """Cells per box that float32 rounds up: a vertex below a leaf plane lands on it or above, so
    float64 names two leaves and float32 one cell.  Deposited once, beside the plane."""
    box, bc = 33.3, 32
    sd = 8 * bc / box
    sf = np.float32(sd)
    assert float(sf) > sd
    below = None
    for node in range(1, 8):
        x = np.float32(box * node / 8)
        while float(x) * sd >= node * bc:
            x = np.nextafter(x, np.float32(0))
        base = np.floor(float(x) * sd)
        assert base == node * bc - 1
        if np.float32(float(x) * float(sf) - base) >= 1.0:  # (the product and the sum are exact in float64)
            below = (node, x)
            break
    assert below is not None
    node, x = below
    rng = np.random.default_rng(3)
    cell = box / (8 * bc)
    pos = np.empty((8, 3))
    pos[:, 0] = float(x) + cell * rng.uniform(0.05, 0.4, 8)
    pos[:, 1:] = cell * (5 + rng.uniform(0.2, 0.8, (8, 2)))
    pos[0, 0] = x
    nodes = [(3, c & 7, (c >> 3) & 7, c >> 6) for c in range(512)]
    tree = pse.octree_from_leaves(np.array(nodes, np.int32), bc, 3, box)
    got = deposit(pos, tree, bc, box, precision=prec, schedule=sched, tuning={"guard_list_cap": cap})
    # beside the plane: the last cell of the leaf below it, the first one of the leaf above
    assert got[node - 1, 5, 5, bc - 1] + got[node, 5, 5, 0] == pytest.approx(1.0, abs=1e-12)
    assert float(got.sum()) == pytest.approx(1.0, abs=1e-12)


# cells a side over a box whose ratio float32 has to round, so that a plane of float32 positions is no
# plane any more in cells (box 100 with 24 and 192 cells, 75 with 100, 1 with 100 and 384); 1 and 256: exact
COPLANAR = [(100.0, 24, 0), (100.0, 24, 3), (75.0, 100, 0), (1.0, 100, 0), (1.0, 24, 4), (1.0, 32, 3)]


def coplanar_cluster(box, cells, rng, across=False):
    """Eight particles of an oblique plane, a few to a few dozen float32 steps wide, on a cell plane
    (across: on the box boundary, half of them in the image on the other side)."""
    cell = box / cells
    while True:
        c = np.float32(cell * (rng.integers(1, cells, 3) + rng.uniform(0.1, 0.9, 3))).astype(np.float64)
        ax = rng.integers(3)
        c[ax] = 0.0 if across else np.float64(np.float32(cell * rng.integers(1, cells)))
        step = np.array([np.spacing(np.float32(v)) for v in c], np.float64)
        if across:
            step[:] = np.spacing(np.float32(box * (1 - 1e-6)))
            c = np.round(c / step) * step
        w = int(rng.integers(1, 20))
        a, b = rng.integers(-w, w + 1, 3), rng.integers(-w, w + 1, 3)
        m, n = rng.integers(-2, 3, 2)
        d = a * m + b * n
        p = np.array([c + step * (a * i + b * j + d * k) for k in (0, 1) for j in (0, 1) for i in (0, 1)])
        p = np.where(p < 0, p + box, p)
        if np.array_equal(p.astype(np.float32).astype(np.float64), p) and np.linalg.matrix_rank(np.array([a, b])) == 2:
            return p


@pytest.mark.parametrize("across", [False, True])
@pytest.mark.parametrize("box,bc,level", COPLANAR)
def test_coplanar_clusters(box, bc, level, across):
    """Exactly coplanar tetrahedra go whole to their centroid's cell, as in the thread kernel, also
    where float32 rounding gives them a volume."""
    rng = np.random.default_rng(7)
    nn = 1 << level
    leaves = [(level, x, y, z) for z in range(nn) for y in range(nn) for x in range(nn)]
    tree = pse.octree_from_leaves(np.array(leaves, np.int32), bc, level, box)
    big = bc ** 3 * nn ** 3 > 1 << 23
    for _ in range(4 if big else 25):
        pos = torch.from_numpy(coplanar_cluster(box, bc * nn, rng, across).astype(np.float32)).cuda()
        kw = {"box": box, "particle_mass": 0.125, "mass_fixup": False}
        ref = pse.deposit_octree(pos, 2, tree, schedule=pse.PSE_THREAD_PER_TET, precision=pse.PSE_FP64_PLAIN, **kw)
        assert float(ref.sum()) == pytest.approx(1.0, abs=1e-12)
        for prec in WARP:
            got, st = pse.deposit_octree(pos, 2, tree, precision=prec, stats=True, **kw)
            assert st["degenerate_tets"] == 48
            assert float((got - ref).abs().max()) <= 1e-12
