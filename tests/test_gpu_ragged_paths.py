"""The warp kernels where their work splits can go wrong: lattices that fill no warp or no item
evenly, one cube per axis, grids coarser and finer than the lattice (paced and unpaced items),
positions whole boxes away from the grid, vertices exactly on octree nodes, and explicit
tetrahedra from slivers to hundreds of cells.  The reference is the plain FP64 kernel, one thread
per tetrahedron and a clip per cell (itself pinned to the oracle).

Tolerances, relative to the largest cell: 1e-5 for FP32 clips (the guard's bound); 1e-11 for the
FP64 column clip (1e-12 of a cell per clip, a few overlapping tetrahedra a cell)."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1612_09491_gb300 as pse  # noqa: E402

pytestmark = pytest.mark.gpu

PLAIN = {"precision": pse.PSE_FP64_PLAIN, "schedule": pse.PSE_THREAD_PER_TET, "tuning": {"thread_fp64": 1}}
FAST64 = {"precision": pse.PSE_FP64_PLAIN, "schedule": pse.PSE_THREAD_PER_TET}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


def positions(n, seed, amp=0.6, wrap=True, boxes=0.0):
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*[np.arange(a) / a for a in n[::-1]], indexing="ij")
    q = np.stack([x.ravel(), y.ravel(), z.ravel()], 1)
    q = q + rng.uniform(-amp, amp, q.shape) / np.array(n)
    if wrap:
        q = np.mod(q, 1.0)
    p = (q + boxes).astype(np.float32)
    return torch.from_numpy(np.ascontiguousarray(p)).cuda()


def worst(a, ref):
    return float((a - ref).abs().max() / ref.abs().max())


LATTICES = [((2, 2, 2), (4, 4, 4)), ((3, 5, 33), (7, 11, 40)), ((33, 2, 9), (16, 9, 9)), ((31, 17, 8), (5, 3, 2)),
            ((12, 9, 10), (60, 47, 55)), ((64, 3, 65), (33, 3, 34))]


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,g", LATTICES)
def test_ragged_uniform(n, g, periodic):
    pos = positions(n, 3, wrap=periodic)
    ref = pse.deposit_uniform(pos, n, g, periodic=periodic, mass_fixup=False, **PLAIN)
    assert worst(pse.deposit_uniform(pos, n, g, periodic=periodic, **FAST64), ref) <= 1e-11
    for prec in (pse.PSE_FP32_FP64ACC, pse.PSE_FP32_COMPENSATED):
        got = pse.deposit_uniform(pos, n, g, periodic=periodic, precision=prec, mass_fixup=False)
        assert worst(got, ref) <= 1e-5


@pytest.mark.parametrize("size", [0.3, 3.0, 40.0])
@pytest.mark.parametrize("flat", [1.0, 1e-2, 1e-5])
def test_explicit_tetrahedra_fp64(size, flat):
    """Sizes in cells from a fraction to hundreds of cells a tetrahedron, slivers among them, with
    zero-volume ones and one cell wide ones at the ends of the batch."""
    rng = np.random.default_rng(11)
    g, t = 48, 77 if size < 10 else 9
    v = rng.uniform(0, 1, (t, 1, 3)) + (rng.uniform(-0.5, 0.5, (t, 4, 3)) * np.array([1, flat, 1])) * size / g
    v[0, 3] = v[0, 2]
    v[-1] = (np.array([[0.1, 0.1, 0.1], [0.9, 0.2, 0.3], [0.2, 0.8, 0.4], [0.3, 0.3, 0.9]]) + 7) / g
    verts = torch.from_numpy(v.astype(np.float32)).cuda()
    mass = torch.from_numpy(rng.uniform(0.5, 2, t)).cuda()
    ref = pse.deposit_tets(verts, mass, g, **PLAIN)
    got = pse.deposit_tets(verts, mass, g, **FAST64)
    # a sliver's density grows as its thickness falls: its clip's error with it
    assert worst(got, ref) <= 1e-11 / flat


@pytest.mark.parametrize("boxes", [0.0, -2.0, 3.0])
@pytest.mark.parametrize("n,amp", [((9, 12, 33), 0.6), ((16, 16, 16), 0.0), ((8, 40, 5), 0.3)])
def test_octree_walk(n, amp, boxes):
    """Leaves on three levels, tetrahedra across leaves and the box boundary, positions whole boxes
    away, and (amp = 0) vertices exactly on the nodes."""
    leaves = [(1, x, y, z) for z in range(2) for y in range(2) for x in range(2)][1:]
    inner = [(2, c & 1, (c >> 1) & 1, c >> 2) for c in range(8)]
    leaves += inner[1:] + [(3, c & 1, (c >> 1) & 1, c >> 2) for c in range(8)]
    tree = pse.octree_from_leaves(np.array(leaves, np.int32), 6, 4)
    pos = positions(n, 5, amp=amp, boxes=boxes)
    ref = pse.deposit_octree(pos, n, tree, mass_fixup=False, **PLAIN)
    assert worst(pse.deposit_octree(pos, n, tree, mass_fixup=False), ref) <= 1e-5
    total = float(pse.deposit_octree(pos, n, tree).sum())
    assert abs(total - 1.0) <= 1e-12
