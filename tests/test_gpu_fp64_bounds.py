"""The FP64 deposit of a uniform grid to float64 accuracy: slivers against the plain FP64 kernel with a
bound per cell, tetrahedra beyond the run queue (2^19 cells and more on a side) against the
oracle with the same bound.

Per-cell bound of a sliver: the clip's classification tolerance, 8 x 2^-52 (1 + extent) of a cell, is the
largest displacement that either side makes on purpose, on up to 4 faces: 8 of it together, times the
tetrahedron's density 6 m / |6V|.  |6V| is a sum of products of the extents e: 16 x 2^-53 e_x e_y e_z / |6V| of each
cell's mass on top.  (absolute: the oracle holds its coordinates from the box's corner, whose rounding
counts like the extent's.)"""
from __future__ import annotations

from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1612_09491_gb300 as pse  # noqa: E402

pytestmark = pytest.mark.gpu

FAST = {"precision": pse.PSE_FP64_PLAIN, "schedule": pse.PSE_THREAD_PER_TET}
PLAIN = {**FAST, "tuning": {"thread_fp64": 1}}
EPS = 2.0 ** -52


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


def volume6(x):
    """|6V| of float64 positions, exact up to its own rounding."""
    a, b, c = [[Fraction(float(x[q, i])) - Fraction(float(x[0, i])) for i in range(3)] for q in (1, 2, 3)]
    return abs(float(a[0] * (b[1] * c[2] - b[2] * c[1]) - a[1] * (b[0] * c[2] - b[2] * c[0]) + a[2] * (b[0] * c[1] - b[1] * c[0])))


def clip_bound(v, mass, grid, ref, absolute=0.0):
    bound = 64 * EPS * ref  # the sums over tetrahedra
    x = v.astype(np.float64) * np.array(grid)
    for k in range(len(v)):
        lo, hi = x[k].min(0), x[k].max(0)
        vol6 = volume6(x[k])
        if vol6 == 0.0:  # flat at its float32 positions: whole to one cell on both sides
            continue
        extent = (np.floor(hi) - np.floor(lo) + 1).sum() + absolute * np.abs(x[k]).max()
        err = 8 * 8 * EPS * (1 + extent) * 6 * mass[k] / vol6 + mass[k] * 8 * EPS * (hi - lo).prod() / vol6
        idx = [np.unique(np.arange(int(a), int(b) + 1) % n) for a, b, n in zip(np.floor(lo), np.floor(hi), grid)]
        bound[np.ix_(*idx[::-1])] += err
    return bound


@pytest.mark.parametrize("size", [0.3, 3.0, 40.0])
@pytest.mark.parametrize("flat", [1.0, 1e-2, 1e-4, 1e-6])
def test_slivers(size, flat):
    rng = np.random.default_rng(12)
    g, t = 64, 60 if size < 10 else 9
    turn = np.array([[1, 0, 0], [0.6, 1, 0], [0.3, -0.5, 1]])  # slivers oblique to the grid
    shape = rng.uniform(-0.5, 0.5, (t, 4, 3)) * np.array([1, 1, flat])
    v = (rng.uniform(0.3, 0.7, (t, 1, 3)) + shape @ turn * size / g).astype(np.float32)
    mass = rng.uniform(0.5, 2, t)
    kw = {"grid_n": g, "mass_fixup": False}
    verts, m = torch.from_numpy(v).cuda(), torch.from_numpy(mass).cuda()
    ref = pse.deposit_tets(verts, m, **kw, **PLAIN).cpu().numpy()
    got = pse.deposit_tets(verts, m, **kw, **FAST).cpu().numpy()
    worst = np.max(np.abs(got - ref) - clip_bound(v, mass, (g, g, g), ref))
    assert worst <= 0.0, worst


@pytest.mark.parametrize("grid,verts", [
    # 2^19 cells and more along x, all within one cell of y and z
    ((600000, 1, 1), [[0.02, 0.2, 0.3], [0.35, 0.9, 0.2], [0.6, 0.1, 0.8], [0.97, 0.7, 0.6]]),
    # along z, three cells across x
    ((3, 1, 540000), [[0.1, 0.2, 0.01], [0.8, 0.9, 0.36], [0.4, 0.1, 0.61], [0.6, 0.7, 0.99]]),
])
def test_beyond_the_run_queue(grid, verts):
    """With small tetrahedra in the same warp, and two large ones."""
    rng = np.random.default_rng(13)
    small = rng.uniform(0.1, 0.2, (7, 1, 3)) + rng.uniform(0, 0.75, (7, 4, 3)) / np.array(grid)
    large = np.array([verts, 1.0 - np.array(verts)])
    v = np.concatenate([small[:3], large[:1], small[3:], large[1:]]).astype(np.float32)
    mass = rng.uniform(0.5, 2, len(v))
    got = pse.deposit_tets(torch.from_numpy(v).cuda(), torch.from_numpy(mass).cuda(), grid, **FAST).cpu().numpy()
    ref, _ = oracle.deposit_tets(v.astype(np.float64), mass, grid)
    worst = np.max(np.abs(got - ref) - clip_bound(v, mass, grid, ref, absolute=1.0))
    assert worst <= 0.0, worst
    assert got.sum() == pytest.approx(mass.sum(), rel=1e-10)
