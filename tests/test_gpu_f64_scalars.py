"""The float64 scalar steps of the column clip that are written without the float64 pipe's slow
instructions, as the GPU runs them (the host build of the same header divides and casts instead):
f64_rcp, f64_widen, f64_sat01, f64_key.

f64_rcp: the start's error e is at most 2^-23 (x cut to float32) + 2^-22 (the approximate reciprocal, 1 ulp)
< 2^-21; one cubic step leaves e^3 < 2^-63 and the rounding of its last operation, half an ulp.  So the result
is within 1 ulp of the correctly rounded one."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = r'''
#include "column.cuh"
using namespace pse;
__global__ void k_scalars(const double *x, const float *y, double *rcp, double *sat, long long *key, double *wide, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = f64_rcp(x[i]);
    sat[i] = f64_sat01(x[i]);
    key[i] = f64_key(x[i]);
    wide[i] = f64_widen(y[i]);
}
extern "C" int scalars(const double *x, const float *y, double *rcp, double *sat, long long *key, double *wide, int n)
{
    k_scalars<<<(n + 255) / 256, 256>>>(x, y, rcp, sat, key, wide, n);
    return (int)cudaDeviceSynchronize();
}
'''


def test_scalars(tmp_path):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1612_09491_gb300 import build
    src, lib = tmp_path / "scalars.cu", tmp_path / "libscalars.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), "-shared", *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-cudart", "static",
                    "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), "-o", str(lib), str(src)],
                   check=True, capture_output=True)
    rng = np.random.default_rng(14)
    m = rng.uniform(1, 2, 1 << 20)
    x = np.ldexp(m, rng.integers(-100, 100, m.size)) * rng.choice([-1.0, 1.0], m.size)
    two = np.ldexp(1.0, np.arange(-100, 100))
    edge = np.concatenate([two, np.nextafter(two[1:], 0), np.nextafter(two, np.inf), [np.nextafter(2.0 ** 100, 0)]])
    out = np.array([0.0, -0.0, 2.0 ** 100, -2.0 ** 100, np.nextafter(2.0 ** -100, 0), 1e300, -1e300, 1e-300, 5e-324])
    x = np.concatenate([x, edge, -edge, out])
    y = rng.integers(0, 1 << 32, x.size, dtype=np.uint64).astype(np.uint32).view(np.float32)
    y = np.where(np.isfinite(y), y, np.float32(1.5))
    y[:6] = np.array([0.0, -0.0, 1.1754944e-38, -1.1754944e-38, 3.4028235e38, 1.0], np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (x, y)]
    rcp, sat, wide = (torch.empty(x.size, dtype=torch.float64, device="cuda") for _ in range(3))
    key = torch.empty(x.size, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    L = ctypes.CDLL(str(lib))
    assert L.scalars(*[ctypes.c_void_p(t.data_ptr()) for t in (*dev, rcp, sat, key, wide)], ctypes.c_int(x.size)) == 0
    rcp, sat, key, wide = (t.cpu().numpy() for t in (rcp, sat, key, wide))

    inside = (np.abs(x) >= 2.0 ** -100) & (np.abs(x) < 2.0 ** 100)
    want = 1.0 / x[inside]
    assert np.max(np.abs(rcp[inside] - want) / np.spacing(np.abs(want))) <= 1.0
    assert np.all(rcp[~inside] == 0.0)
    np.testing.assert_array_equal(sat, np.clip(x, 0.0, 1.0))
    order = np.argsort(x[:-len(out)], kind="stable")  # (two zeros of one value have two keys)
    assert np.all(np.diff(key[:-len(out)][order])[np.diff(x[:-len(out)][order]) > 0] > 0)
    normal = (np.abs(y) >= 1.1754944e-38) | (y == 0)
    np.testing.assert_array_equal(wide[normal], y[normal].astype(np.float64))
    assert np.all(np.abs(wide[~normal]) < 2.0 ** -125)  # a denormal is not kept, but stays as small
