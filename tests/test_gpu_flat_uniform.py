"""Exactly coplanar tetrahedra a few float32 steps wide on a uniform grid whose cells per box is no power
of two: the grid units round, and the flat tetrahedron has a volume there.  It goes whole to one cell all the same: its
centroid's, or for float32 paths, whose scale from box to cells is rounded too (6e-8 of a position), the
one beside it that float32 shows it in."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1612_09491_gb300 as pse  # noqa: E402

pytestmark = pytest.mark.gpu

PATHS = [
    (pse.PSE_FP64_PLAIN, pse.PSE_THREAD_PER_TET, {}),
    (pse.PSE_FP64_PLAIN, pse.PSE_THREAD_PER_TET, {"thread_fp64": 1}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_THREAD_PER_TET, {}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_COOPERATIVE, {}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_COOPERATIVE, {"guard_list_cap": -1}),
    (pse.PSE_FP32_COMPENSATED, pse.PSE_WARP_COOPERATIVE, {}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_BINNED_PERSISTENT, {"split_cells": 1, "chunk_cells": 1}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_PER_TET, {}),
]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


def plane_points(box, g, count, rng):
    """count points of an oblique plane through a cell plane, float32 steps apart, exact in float32."""
    cell = box / g
    while True:
        c = np.float32(cell * (rng.integers(1, g, 3) + rng.uniform(0.1, 0.9, 3))).astype(np.float64)
        ax = rng.integers(3)
        c[ax] = np.float64(np.float32(cell * rng.integers(1, g)))
        step = np.array([np.spacing(np.float32(v)) for v in c], np.float64)
        w = int(rng.integers(1, 20))
        a, b = rng.integers(-w, w + 1, 3), rng.integers(-w, w + 1, 3)
        if np.linalg.matrix_rank(np.array([a, b])) < 2:
            continue
        p = c + step * (rng.integers(-2, 3, (count, 1)) * a + rng.integers(-2, 3, (count, 1)) * b)
        if np.array_equal(p.astype(np.float32).astype(np.float64), p):
            return p


@pytest.mark.parametrize("box,g", [(100.0, 24), (75.0, 100), (1.0, 100), (1.0, 128)])
@pytest.mark.parametrize("prec,sched,tuning", PATHS)
def test_coplanar(prec, sched, tuning, box, g):
    rng = np.random.default_rng(9)
    kw = {"box": box, "precision": prec, "schedule": sched, "tuning": tuning, "mass_fixup": False}
    for _ in range(12):
        v = plane_points(box, g, 4 * 40, rng).reshape(40, 4, 3)
        mass = rng.uniform(0.5, 2, 40)
        u = v.mean(1) * (g / box)
        sure = np.abs(u - np.round(u)).min(1) > 1e-9  # the cell of the centroid does not hang on rounding
        cells = np.floor(u).astype(int)
        want = np.zeros((g, g, g))
        np.add.at(want, tuple(cells[sure][:, ::-1].T), mass[sure])
        got, st = pse.deposit_tets(torch.from_numpy(v[sure].astype(np.float32)).cuda(), torch.from_numpy(mass[sure]).cuda(),
                                   g, stats=True, **kw)
        got = got.cpu().numpy()
        if prec != pse.PSE_FP64_PLAIN:  # the cells around the cluster as one
            near = [np.unique(np.concatenate([cells[:, a] - 1, cells[:, a], cells[:, a] + 1]) % g) for a in (2, 1, 0)]
            got, want = (np.append(m[np.ix_(*near)].sum(), m.sum()) for m in (got, want))
            assert st["degenerate_tets"] + st["single_cell_tets"] == st["tets"]
        # compensated sums hold a cell to 2^-46 of its addends
        assert np.abs(got - want).max() <= 1e-12 * mass.sum()
        assert st["tets"] == sure.sum()
        # the same points as a periodic lattice of 2^3 particles
        pos = torch.from_numpy(plane_points(box, g, 8, rng).astype(np.float32)).cuda()
        got = pse.deposit_uniform(pos, 2, g, particle_mass=0.125, **kw)
        assert float(got.sum()) == pytest.approx(1.0, abs=1e-12)
