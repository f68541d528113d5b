"""may_be_flat, which decides whether a tetrahedron's exact volume is looked at, compiled for the host
from the library's own header: it holds for every exactly coplanar tetrahedron, whatever volume the
rounding of its float32 vertices makes up, and not for ordinary ones."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1612_09491_gb300", "csrc")

HARNESS = r'''
#include <cmath>
#include <math.h>
#include <cstdio>
#include "geom.cuh"
using namespace pse;

static unsigned long long seed = 5;
static unsigned rnd() { seed = seed * 6364136223846793005ull + 1442695040888963407ull; return (unsigned)(seed >> 33); }
static int pick(int lo, int hi) { return lo + (int)(rnd() % (unsigned)(hi - lo + 1)); }
static double unif() { return rnd() / 2147483648.0; }

// float32 vertices in cells relative to the base cell, as the deposit forms them: k periodic images
static void to_cells(const float (&x)[4][3], const int (&k)[4][3], long g, double box, TetSetup<float> &ts)
{
    const double sd = (double)g / box;
    const float sf = (float)sd;
    P3<float> v[4];
    long base[3];
    for (int a = 0; a < 3; ++a) base[a] = (long)std::floor((double)x[0][a] * sd);
    for (int q = 0; q < 4; ++q)
        v[q] = mk<float>(std::fma(x[q][0], sf, (float)(k[q][0] * g - base[0])), std::fma(x[q][1], sf, (float)(k[q][1] * g - base[1])),
                         std::fma(x[q][2], sf, (float)(k[q][2] * g - base[2])));
    tet_setup<float>(v, ts);
}

int main()
{
    struct { double box; long g; } grids[] = {{100, 24}, {100, 192}, {75, 100}, {1, 100}, {1, 384}, {33.3, 4096}, {1, 256}};
    long flat = 0, made_up = 0, missed = 0, plain = 0, tested = 0;
    for (auto gr : grids)
        for (int it = 0; it < 40000; ++it) {
            const bool image = it % 4 == 3;  // vertices on both sides of the box boundary, in x
            const double cell = gr.box / gr.g;
            double c[3], step = 0.0;
            for (int a = 0; a < 3; ++a) {
                c[a] = (float)(cell * (1 + rnd() % (unsigned)(gr.g - 1)));
                int e;
                std::frexp(c[a], &e);
                step = std::fmax(step, std::ldexp(1.0, e - 24));
            }
            if (image) {
                int e;
                std::frexp(gr.box * (1 - 1e-6), &e);
                step = std::ldexp(1.0, e - 24);
                c[0] = 0.0;
            }
            for (double &v : c) v = std::round(v / step) * step;
            const int w = 1 << pick(0, it % 3 == 2 ? 9 : 5);
            double A[3], B[3];
            for (int a = 0; a < 3; ++a) A[a] = step * pick(-w, w), B[a] = step * pick(-w, w);
            const int m = pick(-2, 2), n = pick(-2, 2);
            float x[4][3];
            int k[4][3] = {};
            bool exact = true;
            double u[4][3];
            for (int q = 0; q < 4; ++q)
                for (int a = 0; a < 3; ++a) {
                    u[q][a] = c[a] + (q == 1 ? A[a] : q == 2 ? B[a] : q == 3 ? m * A[a] + n * B[a] : 0.0);
                    double y = u[q][a];
                    if (y < 0.0) y += gr.box, k[q][a] = -1;
                    x[q][a] = (float)y;
                    exact = exact && (double)x[q][a] == y;
                }
            for (int a = 0; a < 3; ++a)
                for (int q = 3; q >= 0; --q) k[q][a] -= k[0][a];
            if (!exact) continue;
            TetSetup<float> ts;
            to_cells(x, k, gr.g, gr.box, ts);
            bool any = false;
            for (auto &r : k)
                for (int v : r) any = any || v != 0;
            ++flat;
            made_up += ts.kappa <= 1e4f;
            missed += !may_be_flat(ts.kappa, (float)ts.vol6, any ? 2.f + gr.g : 2.f);
        }
    // ordinary tetrahedra of a hundredth of a cell to 30 cells
    for (int it = 0; it < 100000; ++it) {
        const double size = std::pow(10.0, -2 + 3.5 * unif());
        P3<float> v[4];
        for (auto &p : v) p = mk<float>((float)(0.5 + size * unif()), (float)(0.5 + size * unif()), (float)(0.5 + size * unif()));
        TetSetup<float> ts;
        tet_setup<float>(v, ts);
        if (!(ts.kappa <= 100.f)) continue;
        ++plain;
        tested += may_be_flat(ts.kappa, (float)ts.vol6, 2.f);
    }
    std::printf("%ld %ld %ld %ld %ld\n", flat, made_up, missed, plain, tested);
    return 0;
}
'''


def _cuda_include():
    for c in (os.environ.get("CUDA_HOME"), "/usr/local/cuda"):
        if c and os.path.exists(os.path.join(c, "include", "cuda_runtime.h")):
            return os.path.join(c, "include")
    return None


def test_flat_tetrahedra_are_looked_at(tmp_path):
    inc = _cuda_include()
    cxx = shutil.which("g++")
    if inc is None or cxx is None:
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "flat.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "flat"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", inc, "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    flat, made_up, missed, plain, tested = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                                                   text=True).stdout.split())
    assert flat > 100_000 and made_up > 5_000, (flat, made_up)  # kappa alone would miss made_up of them
    assert missed == 0, missed
    assert plain > 50_000 and tested == 0, (plain, tested)
