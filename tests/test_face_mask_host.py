"""The faces that the warp kernels leave out of a run before clipping (face_mask) are faces whose
clip finds an empty polygon: compiled for the host from the library's own header, every face left
out is clipped all the same, in float32 and in float64, and must add exactly nothing.

Random tetrahedra from a hundredth of a cell to 200 cells, slivers down to 1e-6 cells, vertices on
cell planes and edge-on faces; the float32 records as the kernels hold them."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1612_09491_gb300", "csrc")

HARNESS = r'''
#include <algorithm>
#include <cmath>
#include <math.h>
#include <cstdio>
#include "column.cuh"
using namespace pse;

static float urand(unsigned long long &s)
{
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return (float)((s >> 40) & 0xffffff) / 16777216.0f;
}

int main()
{
    unsigned long long seed = 77;
    float2 E[21 * 32];
    static double2 D[21 * 32];
    long faces = 0, out = 0, bad32 = 0, bad64 = 0;
    for (int it = 0; it < 6000; ++it) {
        const float spans[6] = {0.01f, 0.6f, 2.5f, 6.f, 30.f, 200.f};
        const float span = spans[it % 6];
        P3<float> v[4];
        for (auto &p : v)
            p = mk<float>(urand(seed) * span - 0.3f * span, urand(seed) * span - 0.3f * span, urand(seed) * span - 0.3f * span);
        if (it % 5 == 1) { v[1].x = v[0].x; v[2].y = 1.f; v[3].z = 0.f; }
        if (it % 7 == 2)  // a sliver, some of its faces edge-on
            for (auto &p : v) p.z = p.x * 0.5f + p.y + (it % 2 ? 1e-6f : 1e-2f) * p.z;
        if (it % 11 == 3) v[3].x = v[2].x, v[3].y = v[2].y;  // an edge along the axis
        TetSetup<float> ts;
        tet_setup<float>(v, ts);
        if (ts.vol6 == 0.0) continue;
        const int C = ts.axis, A = (C + 1) % 3, B = (C + 2) % 3;
        const int skip = std::max(1, ts.dim[A] * ts.dim[B] * ts.dim[C] / 400);  // a sample of large boxes
        long n = 0;
        for (int ia = 0; ia < ts.dim[A]; ++ia)
            for (int ib = 0; ib < ts.dim[B]; ++ib)
                for (int w = 0; w < ts.dim[C]; w += 2) {
                    if (n++ % skip) continue;
                    const int K = std::min(2, ts.dim[C] - w);
                    int cell[3];
                    cell[A] = ts.lo[A] + ia;
                    cell[B] = ts.lo[B] + ib;
                    cell[C] = ts.lo[C] + w;
                    P3<float> p[4], na[4];
                    unsigned up = 0;
                    for (int q = 0; q < 4; ++q) {
                        p[q] = to_axis(mk<float>(ts.v[q].x - cell[0], ts.v[q].y - cell[1], ts.v[q].z - cell[2]), C);
                        na[q] = to_axis(ts.n[q], C);
                        up |= na[q].z > 0.f ? 1u << q : 0u;
                    }
                    const unsigned mask = face_mask(p, up);
                    const RunFrame<float> F = run_frame<float>(TetArrays<float>{p, na}, ts.lx, ts.ly, K, w > 0);
                    RunFrame<double> G;
                    G.qx = F.qx; G.qy = F.qy; G.qz = F.qz; G.l0 = F.l0; G.lx = F.lx; G.ly = F.ly; G.K = F.K; G.j0 = F.j0;
                    for (int f = 0; f < 4; ++f) {
                        ++faces;
                        if (mask >> f & 1u) continue;
                        ++out;
                        int i, j, k;
                        face_vertices(f, i, j, k);
                        const P3<float> q = mk<float>(F.qx, F.qy, F.qz);
                        FaceRun<2, float> R;
                        face_run<2, float>(sub(p[i], q), sub(p[j], q), sub(p[k], q), na[f], F, EdgeSlots<float>{E}, R);
                        bool zero = R.n == 0 && R.m6 == 0.f && R.zmin > R.zmax && R.jlo > R.jhi;
                        for (float x : R.k6) zero = zero && x == 0.f;
                        bad32 += !zero && na[f].z != 0.f;
                        auto d = [&](int t) {
                            return mk<double>((double)p[t].x - F.qx, (double)p[t].y - F.qy, (double)p[t].z - F.qz);
                        };
                        FaceRun64<2> R64;
                        face_run_f64<2>(d(i), d(j), d(k), G, f64_tolerance(200.0), EdgeSlots<double>{D}, R64);
                        zero = R64.n == 0 && R64.m6 == 0.0 && R64.jlo > R64.jhi;
                        for (double x : R64.k6) zero = zero && x == 0.0;
                        bad64 += !zero;
                    }
                }
    }
    std::printf("%ld %ld %ld %ld\n", faces, out, bad32, bad64);
    return 0;
}
'''


def _cuda_include():
    for c in (os.environ.get("CUDA_HOME"), "/usr/local/cuda"):
        if c and os.path.exists(os.path.join(c, "include", "cuda_runtime.h")):
            return os.path.join(c, "include")
    nvcc = shutil.which("nvcc")
    if nvcc:
        inc = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
        if os.path.exists(os.path.join(inc, "cuda_runtime.h")):
            return inc
    return None


def test_faces_left_out_add_nothing(tmp_path):
    inc = _cuda_include()
    cxx = shutil.which("g++")
    if inc is None or cxx is None:
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "mask.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "mask"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", inc, "-o", str(exe), str(src)], check=True, capture_output=True)
    faces, out, bad32, bad64 = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                                       text=True).stdout.split())
    assert faces > 500_000 and out > 100_000, (faces, out)
    assert bad32 == 0, bad32
    assert bad64 == 0, bad64
