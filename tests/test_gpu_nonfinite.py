"""A vertex with a NaN coordinate: its tetrahedra are an error (reported when statistics are asked
for) and leave every cell as the other tetrahedra make it."""
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
    (pse.PSE_FP32_FP64ACC, pse.PSE_BINNED_PERSISTENT, {"split_cells": 8}),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_PER_TET, {}),
]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


@pytest.mark.parametrize("fixup", [False, True])
@pytest.mark.parametrize("prec,sched,tuning", PATHS)
def test_explicit_tetrahedra(prec, sched, tuning, fixup):
    rng = np.random.default_rng(4)
    g, t = 16, 45
    v = rng.uniform(0.2, 0.6, (t, 1, 3)) + rng.uniform(0, 3.5 / g, (t, 4, 3))
    bad = v.copy()
    skip = np.arange(0, t, 5)
    for k, i in enumerate(skip):
        bad[i, 1 + (k // 3) % 3, k % 3] = np.nan  # every axis of every vertex but the first
    mass = rng.uniform(0.5, 2, t)
    kw = {"precision": prec, "schedule": sched, "tuning": tuning, "mass_fixup": fixup}

    def dep(verts, m, **more):
        return pse.deposit_tets(torch.from_numpy(verts.astype(np.float32)).cuda(), torch.from_numpy(m).cuda(), g, **kw, **more)

    keep = np.setdiff1d(np.arange(t), skip)
    ref, got = dep(v[keep], mass[keep]), dep(bad, mass)
    # the same tetrahedra in another order: the rounding of the sums, of pairs of float32 (compensated) 2^-46
    assert float((got - ref).abs().max() / ref.max()) <= 1e-12
    with pytest.raises(pse.PseError, match="non-finite"):
        dep(bad, mass, stats=True)


@pytest.mark.parametrize("prec,sched,tuning", [p for p in PATHS if p[1] in (pse.PSE_THREAD_PER_TET, pse.PSE_WARP_COOPERATIVE)])
def test_octree(prec, sched, tuning):
    n, bc = 8, 6
    rng = np.random.default_rng(5)
    z, y, x = np.meshgrid(*[np.arange(n) / n] * 3, indexing="ij")
    pos = np.stack([x.ravel(), y.ravel(), z.ravel()], 1) + rng.uniform(0.1, 0.6, (n ** 3, 3)) / n
    tree = pse.octree_from_leaves(np.array([(1, c & 1, (c >> 1) & 1, c >> 2) for c in range(8)], np.int32), bc, 1)
    pos[n * n * 3 + n * 4 + 2, 1] = np.nan
    p = torch.from_numpy(pos.astype(np.float32)).cuda()
    kw = {"precision": prec, "schedule": sched, "tuning": tuning, "mass_fixup": False}
    got = pse.deposit_octree(p, n, tree, **kw)
    assert bool(torch.isfinite(got).all())
    # 24 tetrahedra meet in a particle; the FP32 clips keep each one's mass to 1e-5
    assert float(got.sum()) == pytest.approx(1.0 - 24 / (6 * n ** 3), abs=1e-5)
    with pytest.raises(pse.PseError, match="non-finite"):
        pse.deposit_octree(p, n, tree, stats=True, **kw)
