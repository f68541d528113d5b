#!/usr/bin/env python
"""Throughput of the exact tetrahedron deposit on one GB300 (or N independent replicas).

Default workload: 1024^3 particles (6,442,450,944 tetrahedra), Zel'dovich P(k) ~ k^-2 with
rms displacement 3 lattice spacings, periodic unit box, deposited onto the octree of 128^3-cell
leaf blocks, levels 0-4 (2048^3 cells at the finest level).  One step is one pass of the whole
hot path over the lattice: the octree built from the tetrahedra's sizes (one pass over every
tetrahedron, histograms, refinement decisions), then every tetrahedron generated on the fly
from its particles, classified against the cells of its bounding box in each leaf it
reaches, clipped exactly where partial, and its mass accumulated into the float64 leaf
blocks (the call overwrites them, FP32 clips renormalised to the exact total mass).

* value: the step with the positions resident in HBM (12.9 GB), CUDA events on the stream.
* e2e: the same step through the host-buffer C ABI (pse_build_octree_streamed and
  pse_deposit_octree_streamed: positions copied from pinned host memory in z-slabs inside the
  calls) plus the read-back of the step's total deposited mass.
* cpu_baseline: the FP64 CPU oracle on the host cores, on contiguous sub-lattices of the same
  workload deposited at the same cell size (bounded sample); the GPU deposits the same
  sub-lattices for the error on the sample.
* Beside it, as extra keys: the plain FP64 one-thread-per-tetrahedron GPU path on a block of
  the lattice, and the 128^3 precision workload (FP32 vs FP64 vs the oracle's full deposit)
  and the 512^3 cost-model workload.

``--config 2|3|4|6|7`` prints the line of another workload alone; ``--impl reference`` times the
oracle alone (host cores).  Prints one JSON line on rank 0.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "tetrahedra deposited/sec and tet-cell clips/sec at stated density error vs plain FP64 GPU"
UNIT = "tets/s"
L2_FLUSH_BYTES = 512 << 20  # > 129 MB L2
SLAB = 64                    # z-slab of the streamed calls, cube layers
THRESHOLD_CELLS = 2.0        # octree refinement: median mean edge below 2 cells
TUNING = {"blocks_per_sm": 4}

# Algorithmic work per unit for the ALU roofline (floating-point operations, FMA = 2; min,
# max, compares and floor are not counted): per tetrahedron the set-up (determinant, bounding
# box, face planes, divergence axis, reference plane, conditioning); per bounding-box cell one
# classification against the 4 face planes; per clipped run (up to 2 cells of one column) the
# column clip.  tests/test_flop_model_host.py counts these on Zel'dovich tetrahedra of the
# deposit workloads' spectrum at three cell scales, with the kernels' own templates, and
# checks these figures against the counts.
FLOP_PER_TET = 222.0
FLOP_PER_BBOX_CELL = 29.0
FLOP_PER_RUN = 1310.0
SM_COUNT_GB300 = 152
SM_MAX_MHZ_GB300 = 2070.0  # the part's maximum SM clock
FP32_LANES_PER_SM = 128
PRECISION = "fp32 clip, fp64 clip of guarded tetrahedra (exact vertices), fp64 accumulation, mass fix-up"
PROFILES = os.path.join(ROOT, "profiles")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="pse", choices=["pse", "reference"])
    ap.add_argument("--config", type=int, default=5)
    ap.add_argument("--no-baseline", action="store_true", help="skip the FP64 GPU baseline")
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle CPU baseline")
    ap.add_argument("--no-extra", action="store_true", help="skip the extra workload keys")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--e2e-steps", type=int, default=3)
    return ap.parse_args()


# ---------------------------------------------------------------- clocks ----
class ClockSampler:
    """nvidia-smi clock / throttle-reason samples every 200 ms while running."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, bus_id: str | None):
        self.rows = []
        self.proc = None
        self.bus_id = bus_id

    def __enter__(self):
        cmd = ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200"]
        if self.bus_id:
            cmd += ["-i", self.bus_id]
        try:
            self.proc = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                self.rows.append(parts)

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.thread.join(timeout=5)

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"], "samples": 0}
        sm = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows for i in range(4) if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


def bus_id_of(dev_index: int):
    import torch
    try:
        p = torch.cuda.get_device_properties(dev_index)
        return f"{p.pci_domain_id:08X}:{p.pci_bus_id:02X}:{p.pci_device_id:02X}.0"
    except Exception:
        return None


# ------------------------------------------------------------- replicas ----
def replica_throughput(step_ms, units_per_rank, dist=None, device="cpu"):
    """Whole-job throughput of N independent replicas: every rank processed units_per_rank
    per step; the step time is the slowest rank's mean (max over ranks).
    Returns (ms_per_step, units per second over all ranks)."""
    import torch
    ms = sum(step_ms) / len(step_ms)
    world = 1
    if dist is not None:
        world = dist.get_world_size()
        t = torch.tensor([ms], device=device, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms = float(t.item())
    return ms, world * units_per_rank / (ms * 1e-3)


# ------------------------------------------------------------ profiles ----
def source_digest() -> str:
    """sha256 (16 hex) of the CUDA sources and the public header: ncu figures taken on other
    sources do not describe the kernel this run times."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_1612_09491_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(csrc, name), "rb") as f:
                h.update(name.encode() + b"\0" + f.read())
    with open(os.path.join(ROOT, "include", "pse.h"), "rb") as f:
        h.update(b"pse.h\0" + f.read())
    return h.hexdigest()[:16]


def profile_figures(name: str) -> dict:
    """The `key: value` figures of profiles/<name>.txt (ncu summary), or {} if absent."""
    out = {}
    try:
        with open(os.path.join(PROFILES, name + ".txt")) as f:
            for line in f:
                if ":" in line and not line.startswith(("#", " ", "|")):
                    k, v = line.split(":", 1)
                    out[k.strip()] = v.strip()
    except OSError:
        pass
    return out


def roofline_alu(st, kernel_ms, sms, peaks, prof, units_key, units):
    """ALU roofline of the deposit kernel: algorithmic FP32 work of the call's counters over the
    kernel's measured duration, against 152 SMs x 128 lanes x 2 FLOP x max clock.  DRAM traffic
    and issued instructions come from the committed ncu summary when it was taken on these
    very sources (else null)."""
    alg = FLOP_PER_TET * st["tets"] + FLOP_PER_BBOX_CELL * st["bbox_cells"] + FLOP_PER_RUN * st["column_runs"]
    peak = sms * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ_GB300 * 1e6 / 1e12
    achieved = alg / (kernel_ms * 1e-3) / 1e12
    fresh = prof.get("source_digest") == source_digest()
    traffic = None
    issue = None
    if fresh and prof.get(f"dram_bytes_per_{units_key}"):
        traffic = float(prof[f"dram_bytes_per_{units_key}"]) * units
    if fresh and prof.get("thread_inst_per_clip"):
        tin = float(prof["thread_inst_per_clip"])
        rate = tin * st["partial_clips"] / (kernel_ms * 1e-3)
        pk = sms * 4 * 32 * SM_MAX_MHZ_GB300 * 1e6
        issue = {"thread_inst_per_clip": tin, "achieved_tinst_per_s": rate, "peak_tinst_per_s": pk, "frac": rate / pk,
                 "note": "instructions issued by the kernel (ncu) against one warp instruction per scheduler per "
                         "clock (4 per SM), all 32 lanes"}
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
            "traffic": traffic,
            "traffic_unit": "bytes per launch (ncu dram read + write per unit x units)",
            "traffic_source": prof.get("file") if fresh else
            ("ncu summary taken on other sources" if prof else "no ncu summary"),
            "peak_source": f"derived: {sms} SMs x {FP32_LANES_PER_SM} FP32 lanes x 2 FLOP x "
                           f"{SM_MAX_MHZ_GB300:.0f} MHz (of measured: FMA microbenchmark beside it)",
            "measured_fma_tflops": peaks["fp32_tflops"] if peaks else None,
            "flop_model": {"per_tet": FLOP_PER_TET, "per_bbox_cell": FLOP_PER_BBOX_CELL, "per_clipped_run":
                           FLOP_PER_RUN}}, issue


# ------------------------------------------------------------ oracle legs ----
def sample_blocks(h_np, n, g_fine, m, count, seed, margin=24):
    """`count` contiguous blocks of m^3 particles of the periodic lattice (float32 [n^3, 3]),
    each unwrapped around its first particle and moved by a whole number of finest cells into a
    local open box of gl^3 cells (the shift is a multiple of the cell size, so every tetrahedron
    keeps its position relative to the cell planes, exactly).  Returns [(pos [m^3,3], gl, box)]."""
    import numpy as np
    rng = np.random.default_rng(seed)
    h = 1.0 / g_fine
    P = h_np.reshape(n, n, n, 3)
    out = []
    for _ in range(count):
        i0, j0, k0 = (int(v) for v in rng.integers(0, n, 3))
        ii, jj, kk = (np.arange(m) + i0) % n, (np.arange(m) + j0) % n, (np.arange(m) + k0) % n
        pts = P[np.ix_(kk, jj, ii)].astype(np.float64)
        d = pts - pts[0, 0, 0]
        d -= np.round(d)
        q = pts[0, 0, 0] + d
        lo = np.floor(q.reshape(-1, 3).min(0) / h) - margin
        local = q - lo * h
        gl = int(np.ceil(local.reshape(-1, 3).max() / h)) + margin
        gl = (gl + 7) // 8 * 8
        out.append((np.ascontiguousarray(local.reshape(-1, 3).astype(np.float32)), gl, gl * h))
    return out


def oracle_blocks(blocks, m, n, seconds):
    """The oracle on as many sample blocks as fit `seconds` of host time (all cores)."""
    import oracle
    threads = os.cpu_count() or 1
    grids, used, t_tot = [], 0, 0.0
    for pos, gl, box in blocks:
        t0 = time.perf_counter()
        g, st = oracle.deposit_lattice(pos, (m, m, m), gl, box=box, periodic=False, particle_mass=1.0 / n ** 3,
                                       nthreads=threads)
        t_tot += time.perf_counter() - t0
        grids.append(g)
        used += 1
        if t_tot >= seconds:
            break
    tets = 6 * (m - 1) ** 3 * used
    return {"value": tets / t_tot, "unit": UNIT, "cores": int(st["threads"]), "kind": "oracle",
            "sample": f"{used} contiguous blocks of {m}^3 particles ({tets} tetrahedra) of the workload, each "
                      f"deposited alone at the workload's finest cell size, {t_tot:.1f} s"}, grids


KUHN_PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


def lattice_tets_cells(pos, dims, cubes, scale, periodic):
    """float64 vertices [T, 4, 3] in cells (positions x scale) of the Kuhn tetrahedra of the
    given cubes (int64 tensor of cube ids, x fastest) of a lattice of dims particles: corners
    000, e_a, e_a + e_b, 111 for the six axis orders, each corner moved to the periodic image
    nearest corner 000 when `periodic`."""
    import torch
    n0, n1, n2 = dims
    c0, c1 = (n0, n1) if periodic else (n0 - 1, n1 - 1)
    i, j, k = cubes % c0, (cubes // c0) % c1, cubes // (c0 * c1)

    def corner(di, dj, dk):
        ii, jj, kk = i + di, j + dj, k + dk
        if periodic:
            ii, jj, kk = ii % n0, jj % n1, kk % n2
        return pos[ii + n0 * (jj + n1 * kk)].double()

    p0 = corner(0, 0, 0)
    unit = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    out = []
    for a, b, _ in KUHN_PERMS:
        ea = unit[a]
        eab = tuple(x + y for x, y in zip(unit[a], unit[b]))
        vs = [p0]
        for off in (ea, eab, (1, 1, 1)):
            d = corner(*off) - p0
            if periodic:
                d -= torch.round(d)
            vs.append(p0 + d)
        out.append(torch.stack(vs, 1))
    return torch.cat(out, 0) * scale


def density_floor_cells(verts, m_t, cell_index, n_cells):
    """Per cell: the mass of a whole cell at the density of the densest tetrahedron whose
    bounding box covers it (the per-cell floor of the relative error of sparse deposits: a
    cell holding only a sliver of one tetrahedron carries the clip's absolute error at that
    tetrahedron's density).  verts: [T, 4, 3] in cells; cell_index(ix, iy, iz) -> flat index
    into the n_cells outputs, or -1 for cells not compared."""
    import itertools

    import torch
    e1, e2, e3 = verts[:, 1] - verts[:, 0], verts[:, 2] - verts[:, 0], verts[:, 3] - verts[:, 0]
    vol = torch.abs((e1 * torch.cross(e2, e3, dim=1)).sum(1)) / 6.0
    keep = vol > 0
    verts, dens = verts[keep], m_t / vol[keep]
    lo = torch.floor(verts.min(1).values).long()
    dim = torch.floor(verts.max(1).values).long() - lo + 1
    floor = torch.zeros(n_cells, dtype=torch.float64, device=verts.device)
    dmax = int(dim.max().item()) if dim.numel() else 0
    for dx, dy, dz in itertools.product(range(dmax), repeat=3):
        ok = (dim[:, 0] > dx) & (dim[:, 1] > dy) & (dim[:, 2] > dz)
        if not bool(ok.any()):
            continue
        c = lo[ok] + torch.tensor([dx, dy, dz], device=lo.device)
        idx = cell_index(c[:, 0], c[:, 1], c[:, 2])
        sel = idx >= 0
        floor.scatter_reduce_(0, idx[sel], dens[ok][sel], reduce="amax")
    return floor


def block_floor(pos_np, m, gl, box, n, dev):
    """density_floor_cells of one open m^3 sample block on its gl^3 grid ([z, y, x] flat)."""
    import torch
    pos = torch.from_numpy(pos_np).to(dev)
    cubes = torch.arange((m - 1) ** 3, device=dev)
    v = lattice_tets_cells(pos, (m, m, m), cubes, gl / box, periodic=False)

    def index(ix, iy, iz):
        inside = (ix >= 0) & (ix < gl) & (iy >= 0) & (iy < gl) & (iz >= 0) & (iz < gl)
        return torch.where(inside, ix + gl * (iy + gl * iz), torch.full_like(ix, -1))
    return density_floor_cells(v, 1.0 / (6 * n ** 3), index, gl ** 3).cpu().numpy()


def octree_subset_floor(pos, n, cube_ids, octree, touched):
    """density_floor_cells of the cubes `cube_ids` of the periodic n^3 lattice over the leaf blocks
    `touched` of `octree` ([len(touched), bc^3] flat), when all of them are at the finest level;
    else None."""
    import torch
    leaves = torch.from_numpy(octree.leaves()).to(pos.device)
    ml, bc = octree.max_level, octree.bc
    if not bool((leaves[touched, 0] == ml).all()):
        return None
    side = 1 << ml
    g = bc * side
    leaf_of = torch.full((side ** 3,), -1, dtype=torch.long, device=pos.device)
    fin = leaves[:, 0] == ml
    lid = torch.nonzero(fin).ravel()
    lv = leaves[fin].long()
    leaf_of[lv[:, 1] + side * (lv[:, 2] + side * lv[:, 3])] = lid
    pos_of = torch.full((leaves.shape[0],), -1, dtype=torch.long, device=pos.device)
    pos_of[touched] = torch.arange(touched.numel(), device=pos.device)
    v = lattice_tets_cells(pos, (n, n, n), cube_ids, float(g), periodic=True)

    def index(ix, iy, iz):
        ix, iy, iz = ix % g, iy % g, iz % g
        lf = leaf_of[ix // bc + side * (iy // bc + side * (iz // bc))]
        p = torch.where(lf >= 0, pos_of[lf.clamp(min=0)], torch.full_like(lf, -1))
        loc = (ix % bc) + bc * ((iy % bc) + bc * (iz % bc))
        return torch.where(p >= 0, p * bc ** 3 + loc, torch.full_like(p, -1))
    return density_floor_cells(v, 1.0 / (6 * n ** 3), index, touched.numel() * bc ** 3).cpu().numpy()


def gpu_blocks_error(pse, blocks, grids, m, n, dev, g_fine):
    """The GPU's FP32 deposit of the oracle's sample blocks against the oracle, cell by cell."""
    import numpy as np
    import torch
    from paper_1612_09491_gb300.metrics import cell_errors
    fast, ref, flo = [], [], []
    for (pos, gl, box), g in zip(blocks, grids):
        d = torch.from_numpy(pos).to(dev)
        out = pse.deposit_uniform(d, (m, m, m), gl, box=box, periodic=False, particle_mass=1.0 / n ** 3,
                                  precision=pse.PSE_FP32_FP64ACC, schedule=pse.PSE_WARP_COOPERATIVE)
        fast.append(out.cpu().numpy().ravel())
        ref.append(g.ravel())
        flo.append(block_floor(pos, m, gl, box, n, dev))
    fast, ref, flo = np.concatenate(fast), np.concatenate(ref), np.concatenate(flo)
    mean_cell = 1.0 / g_fine ** 3  # the full deposit's mean cell mass
    e = cell_errors(fast, ref, floor_mass=flo)
    e["floor"] = ("per cell: a whole cell at the density of the densest tetrahedron whose bounding box "
                  "covers it (sparse deposits: each block is deposited alone)")
    filled = ref >= 0.5 * mean_cell
    e["on_filled_cells"] = cell_errors(fast[filled], ref[filled])
    e["filled_cells"] = int(filled.sum())
    e["with_mean_cell_floor"] = cell_errors(fast, ref, floor_mass=1e-3 * mean_cell)["max_rel"]
    e["sample"] = "the cpu_baseline blocks, deposited alone on both sides"
    return e


def run_reference(args, cfg):
    """The reference arm: the FP64 CPU oracle on the host cores, each step a bounded sample of the
    workload (contiguous sub-lattices at the workload's cell size for the 1024^3 workload, random
    Lagrangian cubes otherwise)."""
    import numpy as np

    import oracle
    from pse_inputs import config_positions, zeldovich_positions_device
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    threads = os.cpu_count() or 1
    budget = 150.0 / max(1, args.steps + args.warmup)  # whole run within a few minutes
    n = cfg.n
    if cfg.index == 5:
        import torch
        dev = torch.device("cuda", 0) if torch.cuda.is_available() else None
        pos = zeldovich_positions_device(n, cfg.spectral_index, cfg.rms_disp, cfg.seed, device=dev or "cpu")
        h_np = pos.cpu().numpy()
        del pos
        m = 40
        cal = sample_blocks(h_np, n, cfg.grid_n, m, 1, seed=11)
        t0 = time.perf_counter()
        oracle.deposit_lattice(cal[0][0], (m, m, m), cal[0][1], box=cal[0][2], periodic=False,
                               particle_mass=1.0 / n ** 3, nthreads=threads)
        per_block = time.perf_counter() - t0
        nb = max(1, int(budget / max(per_block, 1e-9)))
        times, rng_seed = [], 12
        for k in range(args.warmup + args.steps):
            blocks = sample_blocks(h_np, n, cfg.grid_n, m, nb, seed=rng_seed + k)
            t0 = time.perf_counter()
            for p, gl, box in blocks:
                oracle.deposit_lattice(p, (m, m, m), gl, box=box, periodic=False, particle_mass=1.0 / n ** 3,
                                       nthreads=threads)
            if k >= args.warmup:
                times.append(time.perf_counter() - t0)
        tets = 6 * (m - 1) ** 3 * nb
        sample = f"{nb} contiguous blocks of {m}^3 particles ({tets} tetrahedra) per step, finest cell size"
        grid = f"octree bc={cfg.bc} levels 0-{cfg.max_level} (finest {cfg.grid_n}^3)"
    else:
        pos = config_positions(cfg)
        rng = np.random.default_rng(11)
        calib = np.sort(rng.choice(n ** 3, size=min(n ** 3, 2048), replace=False))
        t0 = time.perf_counter()
        oracle.deposit_lattice(pos, n, cfg.grid_n, cube_ids=calib, nthreads=threads)
        per_cube = (time.perf_counter() - t0) / calib.size
        m = int(min(n ** 3, max(256, budget / max(per_cube, 1e-9))))
        times = []
        for k in range(args.warmup + args.steps):
            ids = np.sort(rng.choice(n ** 3, size=m, replace=False))
            t0 = time.perf_counter()
            oracle.deposit_lattice(pos, n, cfg.grid_n, cube_ids=ids, nthreads=threads)
            if k >= args.warmup:
                times.append(time.perf_counter() - t0)
        tets = 6 * m
        sample = f"{m} random Lagrangian cubes ({tets} tetrahedra) per step"
        grid = f"uniform {cfg.grid_n}^3"
    t = sum(times) / len(times)
    value = tets / t
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": cfg.name, "particles": f"{n}^3", "grid": grid, "step": sample + " (bounded sample)"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------- helpers ----
def _timed(step, steps, warmup, flush, stream):
    """CUDA-event times (ms) of `steps` calls of step() after `warmup` untimed ones, L2 flushed between."""
    import torch
    for _ in range(warmup):
        step()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for k in range(steps):
        if flush is not None:
            flush.fill_(k & 0xFF)
        evs[k][0].record(stream)
        step()
        evs[k][1].record(stream)
    torch.cuda.synchronize()
    return [a.elapsed_time(b) for a, b in evs]


def _tet_size_sample(pos, n, g, layers=8):
    """Quantiles of the tetrahedra's mean edge length in cells of a g^3 grid, from the cost-model
    features of `layers` cube layers in the middle of the lattice.  The rows are moved to the
    periodic image nearest their Lagrangian sites and deposited as an open lattice, so no
    tetrahedron of the sample wraps."""
    import numpy as np
    import torch
    k0 = n // 2
    rows = pos[k0 * n * n:(k0 + layers + 1) * n * n].to("cuda", non_blocking=False).view(layers + 1, n, n, 3)
    ax = torch.arange(n, device=rows.device, dtype=torch.float32) / n
    q = torch.stack(torch.broadcast_tensors(ax.view(1, 1, n),
                                            ax.view(1, n, 1),
                                            ((k0 + torch.arange(layers + 1, device=rows.device)) / n)
                                            .float().view(layers + 1, 1, 1)), -1)
    d = rows - q
    d -= torch.round(d)
    x = (q + d).reshape(-1, 3).contiguous()
    from paper_1612_09491_gb300 import costmodel as cm
    e = cm.features(x, (n, n, layers + 1), g, periodic=False)[:, 11]
    e = e[:: max(1, e.numel() // 4_000_000)].cpu().numpy()
    return {"mean_edge_cells_quantiles": dict(zip(("min", "p01", "median", "p99", "max"),
                                                  [float(v) for v in np.quantile(e, [0, .01, .5, .99, 1])])),
            "sample": f"{layers} cube layers in the middle of the lattice, cells of the {g}^3 grid"}


def _dist_init():
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return dist, world, rank, local


# ------------------------------------------------- the 1024^3 octree workload --
def run_scale(args, cfg):
    import numpy as np
    import torch

    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_09491_gb300 as pse
    from pse_inputs import zeldovich_positions_device

    dist, world, rank, local = _dist_init()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    n, bc, ml = cfg.n, cfg.bc, cfg.max_level
    n_tets = cfg.n_tets
    prec = pse.PSE_FP32_FP64ACC

    def barrier():
        if dist is not None:
            dist.barrier()

    t0 = time.perf_counter()
    pos = zeldovich_positions_device(n, cfg.spectral_index, cfg.rms_disp, cfg.seed, device=dev)
    torch.cuda.synchronize()
    gen_s = time.perf_counter() - t0
    h_pos = torch.empty((n ** 3, 3), dtype=torch.float32).pin_memory()
    h_pos.copy_(pos)
    tet_sizes = _tet_size_sample(pos, n, cfg.grid_n)

    def build():
        return pse.build_octree_from_tet_sizes(pos, n, bc, ml, THRESHOLD_CELLS)

    # the tree, the output blocks and the call's counters (counting kernels, outside the timing)
    oct_ = build()
    out = torch.empty((oct_.n_leaves, bc, bc, bc), dtype=torch.float64, device=dev)
    _, st = pse.deposit_octree(pos, n, oct_, out=out, stats=True, precision=prec, tuning=TUNING)
    leaf_levels = {int(l): int(c) for l, c in zip(*np.unique(oct_.leaves()[:, 0], return_counts=True))}
    n_leaves = oct_.n_leaves
    del oct_

    def step(ev=None):
        if ev is not None:
            ev[0].record(stream)
        o = build()
        if o.n_leaves != n_leaves:
            raise RuntimeError("the octree changed between steps")
        if ev is not None:
            ev[1].record(stream)
        pse.deposit_octree(pos, n, o, out=out, precision=prec, tuning=TUNING)
        if ev is not None:
            ev[2].record(stream)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]
    with ClockSampler(bus_id_of(local)) as clk:
        t_wall0 = time.perf_counter()
        for k in range(args.steps):
            step(evs[k])
        torch.cuda.synchronize()
        t_wall = time.perf_counter() - t_wall0
    barrier()
    step_ms = [e[0].elapsed_time(e[2]) for e in evs]
    build_ms = [e[0].elapsed_time(e[1]) for e in evs]
    dep_ms = [e[1].elapsed_time(e[2]) for e in evs]
    ms, value = replica_throughput(step_ms, n_tets, dist, dev)
    mass_error = abs(float(out.sum()) - 1.0)

    # end to end through the host-buffer C ABI: both calls stream the positions from pinned
    # host memory in z-slabs; the step's result read back is its total deposited mass
    ke = max(1, min(args.e2e_steps, args.steps))
    del pos
    torch.cuda.empty_cache()
    e2e_ms = []
    mass_h = torch.empty(1, dtype=torch.float64).pin_memory()
    for k in range(ke + 1):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record(stream)
        o = pse.build_octree_streamed(h_pos, n, bc, ml, SLAB, THRESHOLD_CELLS)
        pse.deposit_octree_streamed(h_pos, n, o, SLAB, out=out, precision=prec, tuning=TUNING)
        mass_h.copy_(out.sum().view(1), non_blocking=True)
        b.record(stream)
        torch.cuda.synchronize()
        if k > 0:  # the first call warms the slab buffers
            e2e_ms.append(a.elapsed_time(b))
    e2e_mean = sum(e2e_ms) / len(e2e_ms)
    if dist is not None:
        t = torch.tensor([e2e_mean], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e_mean = float(t.item())
    h2d = int(2 * h_pos.numel() * 4 * (1 + 1 / SLAB))  # the build's pass and the deposit's pass
    hist_bytes = sum(64 * 8 ** l for l in range(ml)) * 4

    result = {}
    if rank == 0:
        h_np = h_pos.numpy()
        base = None
        if not args.no_baseline:
            # the plain FP64 one-thread-per-tetrahedron path and the timed FP32 path on a contiguous
            # block of 64 x 64 x 32 cubes (positions back on the GPU for this check)
            pos_d = h_pos.to(dev)
            o = pse.build_octree_from_tet_sizes(pos_d, n, bc, ml, THRESHOLD_CELLS)
            i, j, k = np.meshgrid(np.arange(64), np.arange(64), np.arange(32), indexing="ij")
            ids = torch.from_numpy(np.sort((i + n * (j + n * (k + n // 2))).ravel())).to(dev)
            pse.deposit_octree(pos_d, n, o, out=out, cube_ids=ids, precision=prec, tuning=TUNING)
            touched = torch.nonzero(out.view(out.shape[0], -1).abs().sum(1) > 0).ravel()
            fast = out[touched].cpu().numpy()
            bms = _timed(lambda: pse.deposit_octree(pos_d, n, o, out=out, cube_ids=ids,
                                                    precision=pse.PSE_FP64_PLAIN, schedule=pse.PSE_THREAD_PER_TET),
                         1, 1, None, stream)[0]
            fms = _timed(lambda: pse.deposit_octree(pos_d, n, o, out=out, cube_ids=ids, precision=prec,
                                                    tuning=TUNING), 1, 1, None, stream)[0]
            pse.deposit_octree(pos_d, n, o, out=out, cube_ids=ids, precision=pse.PSE_FP64_PLAIN,
                               schedule=pse.PSE_THREAD_PER_TET)
            slow = out[touched].cpu().numpy()
            from paper_1612_09491_gb300.metrics import cell_errors
            cells = float(cfg.grid_n) ** 3
            filled = slow >= 0.5 / cells
            base = {"tets_per_s": 6 * ids.numel() / (bms * 1e-3), "ms_on_sample": bms,
                    "fp32_ms_on_sample": fms, "sample": "64 x 64 x 32 contiguous cubes",
                    "speedup": value / (6 * ids.numel() / (bms * 1e-3)),
                    "speedup_on_sample": bms / fms,
                    "error_on_filled_cells": cell_errors(fast[filled], slow[filled]),
                    "filled_cells": int(filled.sum()), "leaves_compared": int(touched.numel())}
            flo = octree_subset_floor(pos_d, n, ids, o, touched)
            if flo is not None:
                base["error_of_timed_arm_on_sample"] = cell_errors(fast, slow, floor_mass=flo.reshape(fast.shape))
                base["error_floor"] = ("per cell: a whole cell at the density of the densest tetrahedron whose "
                                       "bounding box covers it (the sample is a sparse deposit)")
            else:
                base["error_of_timed_arm_on_sample"] = cell_errors(fast, slow, floor_mass=1e-3 / cells)
                base["error_floor"] = "1e-3 of the full deposit's mean cell mass"
            base["with_mean_cell_floor"] = cell_errors(fast, slow, floor_mass=1e-3 / cells)["max_rel"]
            del pos_d
        cpu = oracle_err = None
        if not args.no_cpu:
            blocks = sample_blocks(h_np, n, cfg.grid_n, 40, 64, seed=7)
            cpu, grids = oracle_blocks(blocks, 40, n, args.cpu_seconds)
            oracle_err = gpu_blocks_error(pse, blocks[:len(grids)], grids, 40, n, dev, cfg.grid_n)
        props = torch.cuda.get_device_properties(dev)
        sms = props.multi_processor_count or SM_COUNT_GB300
        peaks = pse.measure_peaks(stream)
        prof = profile_figures("k_oct_warp_scale-1024c-octree128")
        prof["file"] = "profiles/k_oct_warp_scale-1024c-octree128.txt"
        kern = sum(dep_ms) / len(dep_ms)
        roof, issue = roofline_alu(st, kern, sms, peaks, prof, "tet", n_tets)
        extra = {}
        if not args.no_extra:
            extra["workload_precision_128c"] = run_precision(args, pse, dev, stream, standalone=False)
            extra["workload_learned_512c"] = run_learned(args, pse, dev, stream)
        result = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": cfg.name, "particles": f"{n}^3", "tets": n_tets,
                       "spectrum": f"P(k)~k^{cfg.spectral_index}", "rms_disp_spacings": cfg.rms_disp,
                       "grid": f"octree bc={bc} levels 0-{ml} (finest {cfg.grid_n}^3), refined where the "
                               f"median mean edge < {THRESHOLD_CELLS} cells", "leaves": n_leaves,
                       "leaf_levels": leaf_levels, "precision": PRECISION, "schedule": "warp-cooperative",
                       "tuning": TUNING,
                       "step": "octree build from tetrahedron sizes + octree deposit, positions resident",
                       "l2": "inputs larger than L2 (12.9 GB positions, 68.7 GB leaf blocks); no flush",
                       "input_generation": f"torch generator + torch.fft on the GPU (float32), {gen_s:.1f} s",
                       "parallelism": f"replicas x{world}"},
            "clips_per_s": world * st["partial_clips"] / (ms * 1e-3),
            "step_parts_ms": {"octree_build": sum(build_ms) / len(build_ms), "deposit": kern},
            "counters": {k: st[k] for k in ("tets", "bbox_cells", "inside_cells", "partial_clips", "fp64_redos",
                                            "degenerate_tets", "single_cell_tets", "inverted_tets",
                                            "column_runs")},
            "tet_sizes": tet_sizes,
            "mass_error": mass_error,
            "fp64_gpu_baseline": base,
            "error_vs_oracle": oracle_err,
            "kernel_ms": kern,
            "roofline": roof,
            "issue": issue,
            "atomics": {"reductions_per_s": st["overlapped_cells"] / (kern * 1e-3),
                        "peak_per_s": peaks["red_f64_per_s"],
                        "frac": st["overlapped_cells"] / (kern * 1e-3) / peaks["red_f64_per_s"],
                        "note": "one red.global.add.f64 per (tetrahedron, cell) pair that received mass, against "
                                "pse_microbench_red (pseudo-random FP64 reductions over a 134 MB array)"},
            "cpu_baseline": cpu,
            "e2e": {"value": world * n_tets / (e2e_mean * 1e-3), "unit": UNIT, "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": hist_bytes + 8, "ms_per_step": e2e_mean, "steps": len(e2e_ms),
                    "path": "pse_build_octree_streamed + pse_deposit_octree_streamed from pinned host memory "
                            f"(z-slabs of {SLAB} cube layers, double-buffered), then the total mass read back; "
                            "the leaf blocks stay on the GPU",
                    "total_mass": float(mass_h.item())},
            # per step: k_tet_size_hist, the two k_oct_warp passes, k_finish (the ncu launch list
            # of this command in profiles/)
            "gpu_launches": 4 * args.steps,
            "clocks": clk.summary(),
            "wall_s_timed": t_wall,
            **extra,
        }
        print(json.dumps(result), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()


# ------------------------------------------------- the 128^3 precision workload --
def run_precision(args, pse, dev, stream, standalone=True):
    """128^3 particles onto the uniform 256^3 grid: the timed FP32 path (autotuned), the plain FP64
    GPU path, compensated FP32 accumulation, the paper's warp-per-tetrahedron design, and the
    oracle's full deposit (timed: the cpu_baseline of this workload) with every cell compared."""
    import numpy as np
    import torch

    from paper_1612_09491_gb300 import autotune
    from paper_1612_09491_gb300 import costmodel as cm
    from paper_1612_09491_gb300.metrics import cell_errors
    from pse_inputs import CONFIGS, config_positions
    cfg = CONFIGS[2]
    n, g = cfg.n, cfg.grid_n
    n_tets = cfg.n_tets
    pos_host = config_positions(cfg)
    pos = torch.from_numpy(pos_host).to(dev)
    out = torch.empty((g, g, g), dtype=torch.float64, device=dev)
    ws = torch.empty(pse.workspace_size(schedule=pse.PSE_BINNED_PERSISTENT), dtype=torch.uint8, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    prec = pse.PSE_FP32_FP64ACC

    def call(tu, **kw):
        knobs = {k: v for k, v in tu.items() if k != "schedule"}
        sched = pse.PSE_BINNED_PERSISTENT if tu["schedule"] == "binned" else pse.PSE_WARP_COOPERATIVE
        return pse.deposit_uniform(pos, n, g, out=out, workspace=ws, precision=prec, schedule=sched, tuning=knobs,
                                   **kw)

    tuned, tune_ms = autotune.tune(call, signature=f"uniform:{cfg.name}", candidates=autotune.UNIFORM_CANDIDATES)
    _, st = call(tuned, stats=True)
    fast_grid = out.cpu().numpy().copy()
    steps = max(1, args.steps) if standalone else 5
    step_ms = _timed(lambda: call(tuned), steps, 3, flush, stream)
    ms = sum(step_ms) / len(step_ms)
    kern_ms = sum(_timed(lambda: call(tuned, accumulate=True), steps, 1, flush, stream)) / steps
    # end to end: positions from pinned host memory in, the grid back out, every step
    pos_pin = torch.from_numpy(pos_host).pin_memory()
    out_pin = torch.empty((g, g, g), dtype=torch.float64).pin_memory()

    def e2e_step():
        pos.copy_(pos_pin, non_blocking=True)
        call(tuned)
        out_pin.copy_(out, non_blocking=True)
    e2e_ms = sum(_timed(e2e_step, steps, 1, flush, stream)) / steps
    res = {"workload": cfg.name, "particles": f"{n}^3", "tets": n_tets, "grid": f"uniform {g}^3 float64",
           "tets_per_s": n_tets / (ms * 1e-3), "ms_per_step": ms, "steps": steps, "kernel_ms": kern_ms,
           "clips_per_s": st["partial_clips"] / (ms * 1e-3),
           "schedule": {"binned": "binned persistent", "warp": "warp-cooperative"}[tuned["schedule"]],
           "tuning": tuned, "autotune_ms": tune_ms,
           "counters": {k: st[k] for k in ("tets", "bbox_cells", "inside_cells", "partial_clips", "fp64_redos",
                                           "inverted_tets", "bin_counts")},
           "e2e": {"tets_per_s": n_tets / (e2e_ms * 1e-3), "ms_per_step": e2e_ms,
                   "h2d_bytes_per_step": int(pos_host.nbytes), "d2h_bytes_per_step": int(out.numel() * 8)}}
    if not args.no_baseline:
        bms = _timed(lambda: pse.deposit_uniform(pos, n, g, out=out, workspace=ws, precision=pse.PSE_FP64_PLAIN,
                                                 schedule=pse.PSE_THREAD_PER_TET, tuning={"thread_fp64": 1}),
                     1, 1, flush, stream)[0]
        ref64 = out.cpu().numpy()
        base = {"tets_per_s": n_tets / (bms * 1e-3), "ms_per_step": bms, "speedup": bms / ms,
                "error_of_timed_arm": cell_errors(fast_grid, ref64)}
        pms = sum(_timed(lambda: pse.deposit_uniform(pos, n, g, out=out, workspace=ws, precision=prec,
                                                     schedule=pse.PSE_WARP_PER_TET), 3, 1, flush, stream)) / 3
        base["paper_design_warp_per_tet"] = {"tets_per_s": n_tets / (pms * 1e-3), "ms_per_step": pms,
                                             "speedup_of_timed_arm": pms / ms}
        knobs = {k: v for k, v in tuned.items() if k != "schedule"}
        csched = pse.PSE_BINNED_PERSISTENT if tuned["schedule"] == "binned" else pse.PSE_WARP_COOPERATIVE
        cms = sum(_timed(lambda: pse.deposit_uniform(pos, n, g, out=out, workspace=ws, tuning=knobs, schedule=csched,
                                                     precision=pse.PSE_FP32_COMPENSATED), 3, 1, flush, stream)) / 3
        base["fp32_compensated_accumulation"] = {"tets_per_s": n_tets / (cms * 1e-3), "ms_per_step": cms,
                                                 "error_vs_fp64": cell_errors(out.cpu().numpy(), ref64)}
        res["fp64_gpu_baseline"] = base
    if not args.no_cpu:
        import oracle
        t0 = time.perf_counter()
        ref, ost = oracle.deposit_lattice(pos_host, n, g, nthreads=os.cpu_count() or 1)
        dt = time.perf_counter() - t0
        res["cpu_baseline"] = {"value": n_tets / dt, "unit": UNIT, "cores": int(ost["threads"]), "kind": "oracle",
                               "sample": f"the whole workload ({n_tets} tetrahedra), {dt:.1f} s"}
        e = cell_errors(fast_grid, ref)
        e["cells"] = "every cell of the 256^3 grid, floor 1e-3 of the mean occupied cell"
        res["error_vs_oracle"] = e
    tet = cm.features(pos, n, g)[:, 11].cpu().numpy()
    res["tet_sizes"] = {"mean_edge_cells_quantiles": dict(zip(("min", "p01", "median", "p99", "max"),
                                                              [float(v) for v in np.quantile(tet, [0, .01, .5, .99, 1])]))}
    return res


# ------------------------------------------------- the 512^3 cost-model workload --
def run_learned(args, pse, dev, stream):
    """512^3 particles onto the uniform 512^3 grid: the cost model trained on the counts the exact
    deposit produces on the 32^3 and 128^3 workloads, then the warp schedule, the bbox-binned and
    the model-binned persistent schedules (one warm-up and one timed call each)."""
    import torch

    from paper_1612_09491_gb300 import costmodel as cm
    from pse_inputs import CONFIGS, config_positions, zeldovich_positions_device
    cfg = CONFIGS[4]
    n, g = cfg.n, cfg.grid_n
    prec = pse.PSE_FP32_FP64ACC
    pos = zeldovich_positions_device(n, cfg.spectral_index, cfg.rms_disp, cfg.seed, device=dev)
    out = torch.empty((g, g, g), dtype=torch.float64, device=dev)
    ws = torch.empty(pse.workspace_size(pse._lib.PSE_OP_DEPOSIT_UNIFORM, pse.lattice(n),
                                        schedule=pse.PSE_BINNED_PERSISTENT, cost_model=cm.CostModel()),
                     dtype=torch.uint8, device=dev)
    t0 = time.perf_counter()
    feats, targs = [], []
    for c in (CONFIGS[1], CONFIGS[2]):
        p = torch.from_numpy(config_positions(c)).to(dev)
        feats.append(cm.features(p, c.n, c.grid_n))
        targs.append(cm.labels(cm.tet_counts(p, c.n, c.grid_n)))
    feat, targ = torch.cat(feats), torch.cat(targs)
    mu, sd = cm.standardisation(feat[:: max(1, feat.shape[0] // 200000)].cpu().numpy())
    model = cm.CostModel(cm.pack({**cm.he_init(0), "mu": mu, "sigma": sd}))
    hist = cm.fit(model, feat, targ, steps=2000, batch=8192, lr=3e-3)
    train_s = time.perf_counter() - t0
    del feat, targ, feats, targs
    arms = {"warp": dict(schedule=pse.PSE_WARP_COOPERATIVE, tuning=TUNING, precision=prec),
            "binned-bbox": dict(schedule=pse.PSE_BINNED_PERSISTENT, precision=prec,
                                tuning={"blocks_per_sm": 4, "split_cells": 512, "chunk_cells": 512}),
            "binned-model": dict(schedule=pse.PSE_BINNED_PERSISTENT, cost_model=model, precision=prec,
                                 tuning={"blocks_per_sm": 4, "split_cells": 256, "chunk_cells": 512})}
    arm_ms = {}
    for name, kw in arms.items():
        arm_ms[name] = _timed(lambda: pse.deposit_uniform(pos, n, g, out=out, workspace=ws, **kw), 1, 1, None,
                              stream)[0]
    _, st = pse.deposit_uniform(pos, n, g, out=out, workspace=ws, stats=True, **arms["warp"])
    best = min(arm_ms, key=arm_ms.get)
    return {"workload": cfg.name, "particles": f"{n}^3", "tets": cfg.n_tets, "grid": f"uniform {g}^3 float64",
            "arms_ms": arm_ms, "fastest": best, "tets_per_s": cfg.n_tets / (arm_ms[best] * 1e-3),
            "model_vs_warp": arm_ms["warp"] / arm_ms["binned-model"],
            "cost_model": {"training_s": train_s, "loss_first_last": [hist[0], hist[-1]]},
            "counters": {k: st[k] for k in ("tets", "bbox_cells", "partial_clips", "fp64_redos")},
            "mass_error": abs(float(out.sum()) - 1.0),
            "note": "one warm-up and one timed call per arm; the model steers which tetrahedra are split "
                    "across warps, never a deposited value"}


# -------------------------------------- the 256^3 octree workloads (3, and 6 for profiling) --
def run_octree256(args, cfg):
    import numpy as np
    import torch

    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_09491_gb300 as pse
    from paper_1612_09491_gb300 import autotune
    from paper_1612_09491_gb300.metrics import cell_errors
    from pse_inputs import config_positions
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    prec = pse.PSE_FP32_FP64ACC
    n = cfg.n
    pos = torch.from_numpy(config_positions(cfg)).to(dev)
    oct_ = pse.build_octree_from_tet_sizes(pos, n, cfg.bc, cfg.max_level, THRESHOLD_CELLS)
    out = torch.empty((oct_.n_leaves, cfg.bc, cfg.bc, cfg.bc), dtype=torch.float64, device=dev)
    if cfg.index == 6:  # the profiling case runs the 1024^3 workload's launch configuration
        tuned, tune_ms = dict(TUNING), None
    else:
        tuned, tune_ms = autotune.tune(lambda tu: pse.deposit_octree(pos, n, oct_, out=out, tuning=tu,
                                                                     precision=prec),
                                       signature=f"octree:{cfg.name}")
    _, st = pse.deposit_octree(pos, n, oct_, out=out, stats=True, tuning=tuned, precision=prec)

    def step():
        o = pse.build_octree_from_tet_sizes(pos, n, cfg.bc, cfg.max_level, THRESHOLD_CELLS)
        pse.deposit_octree(pos, n, o, out=out, tuning=tuned, precision=prec)

    with ClockSampler(bus_id_of(0)) as clk:
        step_ms = _timed(step, args.steps, args.warmup, flush, stream)
    ms = sum(step_ms) / len(step_ms)
    value = cfg.n_tets / (ms * 1e-3)
    fast = out.cpu().numpy()
    base = None
    if not args.no_baseline:
        bms = _timed(lambda: pse.deposit_octree(pos, n, oct_, out=out, precision=pse.PSE_FP64_PLAIN,
                                                schedule=pse.PSE_THREAD_PER_TET), 1, 1, flush, stream)[0]
        base = {"tets_per_s": cfg.n_tets / (bms * 1e-3), "ms_per_step": bms, "speedup": bms / ms,
                "error_of_timed_arm": cell_errors(fast, out.cpu().numpy())}
    result = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1, "steps": args.steps,
              "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
              "vs_baseline": None, "dtype": "f32", "data": "synthetic",
              "config": {"workload": cfg.name, "particles": f"{n}^3", "tets": cfg.n_tets,
                         "grid": f"octree bc={cfg.bc} levels 0-{cfg.max_level} (finest {cfg.grid_n}^3)",
                         "collapsed_regions": ({"regions": cfg.collapse[0], "R": cfg.collapse[1], "R2": cfg.collapse[2],
                                                "f": cfg.collapse[3]} if cfg.collapse else None),
                         "leaves": int(oct_.n_leaves),
                         "leaf_levels": {int(l): int(c) for l, c in
                                         zip(*np.unique(oct_.leaves()[:, 0], return_counts=True))},
                         "tuning": tuned, "autotune_ms": tune_ms, "precision": PRECISION,
                         "l2": "512 MB buffer written between timed steps", "parallelism": "replicas x1"},
              "clips_per_s": st["partial_clips"] / (ms * 1e-3),
              "counters": {k: st[k] for k in ("tets", "bbox_cells", "inside_cells", "partial_clips", "fp64_redos",
                                              "inverted_tets")},
              "mass_error": abs(float(fast.sum()) - 1.0),
              "fp64_gpu_baseline": base,
              "clocks": clk.summary(),
              "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0,
                      "note": "inputs resident (no host copies in this workload's step)"}}
    print(json.dumps(result), flush=True)


def main():
    args = parse()
    from pse_inputs import CONFIGS
    cfg = CONFIGS[args.config]
    if args.impl == "reference":
        run_reference(args, cfg)
        return
    if args.config == 5:
        run_scale(args, cfg)
    elif args.config in (3, 6, 7):
        run_octree256(args, cfg)
    else:
        import torch

        import __graft_entry__
        __graft_entry__.build()
        import paper_1612_09491_gb300 as pse
        dist, world, rank, local = _dist_init()
        dev = torch.device("cuda", local)
        stream = torch.cuda.current_stream(dev)
        if args.config == 4:
            with ClockSampler(bus_id_of(local)) as clk:
                res = run_learned(args, pse, dev, stream)
        else:
            with ClockSampler(bus_id_of(local)) as clk:
                res = run_precision(args, pse, dev, stream, standalone=True)
        if rank == 0:
            ms = res.get("ms_per_step") or res["arms_ms"][res["fastest"]]
            line = {"metric": METRIC, "value": res["tets_per_s"], "unit": UNIT, "n_gpus": world,
                    "steps": res.get("steps", 1), "warmup": args.warmup, "ms_per_step": ms,
                    "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                    "data": "synthetic", "config": {"workload": res["workload"], "parallelism": f"replicas x{world}"},
                    "cpu_baseline": res.get("cpu_baseline"),
                    "e2e": {"value": res.get("e2e", {}).get("tets_per_s", res["tets_per_s"]), "unit": UNIT,
                            "h2d_bytes_per_step": res.get("e2e", {}).get("h2d_bytes_per_step", 0),
                            "d2h_bytes_per_step": res.get("e2e", {}).get("d2h_bytes_per_step", 0)},
                    "clocks": clk.summary(), "detail": res}
            print(json.dumps(line), flush=True)
        if dist is not None:
            dist.barrier()
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
