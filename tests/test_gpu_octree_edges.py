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


@pytest.mark.parametrize("cap", [0, -1])
@pytest.mark.parametrize("prec", WARP)
def test_single_cell_just_below_the_box(prec, cap):
    """z a few 1e-20 below the box: float64 names the last leaf (of the image below), float32
    rounds the cell to the one after it."""
    rng = np.random.default_rng(2)
    pos = np.empty((8, 3))
    pos[:, :2] = 0.97 + rng.uniform(0, 0.01, (8, 2))
    pos[:, 2] = -1e-20 * rng.permutation(np.arange(1, 9))
    bc = 4
    tree = pse.octree_from_leaves(np.array(EIGHTHS, np.int32), bc, 1)
    got, st = deposit(pos, tree, bc, 1.0, precision=prec, stats=True, tuning={"guard_list_cap": cap})
    want = np.zeros_like(got)
    want[7, 3, 3, 3] = 1.0
    # (compensated sums hold a cell to 2^-48 of each addend)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-12)
    assert st["single_cell_tets"] + st["degenerate_tets"] == 48


@pytest.mark.parametrize("cap", [0, -1])
@pytest.mark.parametrize("prec", WARP)
def test_single_cell_across_a_leaf_plane(prec, cap):
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
    got = deposit(pos, tree, bc, box, precision=prec, tuning={"guard_list_cap": cap})
    # beside the plane: the last cell of the leaf below it, the first one of the leaf above
    assert got[node - 1, 5, 5, bc - 1] + got[node, 5, 5, 0] == pytest.approx(1.0, abs=1e-12)
    assert float(got.sum()) == pytest.approx(1.0, abs=1e-12)
