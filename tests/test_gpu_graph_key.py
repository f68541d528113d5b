"""use_graph replays a captured launch sequence only for calls that launch the same kernels: calls on
one workspace and one output that differ in precision, schedule or pse_tuning.thread_fp64 only."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1612_09491_gb300 as pse  # noqa: E402

pytestmark = pytest.mark.gpu

# (precision, schedule, thread_fp64)
CALLS = [
    (pse.PSE_FP32_FP64ACC, pse.PSE_THREAD_PER_TET, 0),
    (pse.PSE_FP64_PLAIN, pse.PSE_THREAD_PER_TET, 0),
    (pse.PSE_FP64_PLAIN, pse.PSE_THREAD_PER_TET, 1),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_PER_TET, 0),
    (pse.PSE_FP32_FP64ACC, pse.PSE_WARP_COOPERATIVE, 0),
]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    build.build()
    pse._lib.load()
    yield


@pytest.mark.parametrize("order", [1, -1])
def test_each_call_runs_its_own_kernels(order):
    """One tetrahedron to a block of 4^3 cells, so that each cell gets one addend and a kernel's masses
    are the same bits every time; the kernels' masses differ in their last bits."""
    rng = np.random.default_rng(6)
    g, per = 32, 8
    at = np.stack(np.meshgrid(*[np.arange(per)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    verts = torch.from_numpy(((at * 4 + 0.5 + rng.uniform(0, 2.9, (per ** 3, 4, 3))) / g).astype(np.float32)).cuda()
    mass = torch.from_numpy(rng.uniform(0.5, 2, per ** 3)).cuda()
    ws = torch.empty(pse.workspace_size(schedule=pse.PSE_WARP_COOPERATIVE), dtype=torch.uint8, device="cuda")
    out = torch.empty((g, g, g), dtype=torch.float64, device="cuda")

    def call(prec, sched, thread, graph):
        return pse.deposit_tets(verts, mass, g, precision=prec, schedule=sched, mass_fixup=False, workspace=ws, out=out,
                                tuning={"thread_fp64": thread, "use_graph": graph}).clone()

    plain = [call(*c, 0) for c in CALLS]
    for i in range(len(CALLS)):
        for j in range(i):
            assert not torch.equal(plain[i], plain[j]), (CALLS[i], CALLS[j])
    for _ in range(2):
        for c, want in list(zip(CALLS, plain))[::order]:
            assert torch.equal(call(*c, 1), want), c
