// deposit.cu -- tetrahedron deposit kernels for sm_103a.
//
//  * k_thread_per_tet<T>: one thread per tetrahedron walks its bounding-box cells,
//    classifies each, clips the partial ones and adds m_t V_ov/|V_t| with a global
//    float64 atomic.  With T = double this is the plain FP64 baseline.
//  * k_warp_plain: the same results in float64 by the warp-cooperative column clip (calls without
//    statistics).
//  * k_warp_coop (coop.cuh): the warp-cooperative FP32 kernel; this file instantiates
//    its FP64-reduction variants, deposit_comp.cu the compensated-FP32 ones.
//  * k_warp_per_tet: the paper's warp-per-tetrahedron design (Sec. 6.2), a baseline.
//  * k_bin_pass, k_chunk_scan: the binned schedule's queue of large tetrahedra.
//  * k_finish: pair conversion and mass renormalisation at the end of an FP32 deposit.
//  * k_build_tets: particle indices and signed volumes of every tetrahedron.
#include "coop.cuh"
#include "costmodel.cuh"

namespace pse {

namespace {

// ---------------------------------------------------------------------------
// thread per tetrahedron
// ---------------------------------------------------------------------------
template <class T, bool STATS>
__global__ void __launch_bounds__(128) k_thread_per_tet(const DepositParams P)
{
    Counters cnt;
    if (STATS) cnt.zero();
    cnt.zero_mass();
    const int64_t n_tets = (P.src == SRC_TETS) ? P.n_units : 6 * P.n_units;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n_tets;
         t += (int64_t)gridDim.x * blockDim.x) {
        cnt.fold_dep();  // the previous tetrahedron's deposits
        P3<T> v[4];
        P3<float> res[4];
        int base[3];
        double m_t;
        if (P.src == SRC_TETS) {
            explicit_tet<T>(P, t, v, base, res);
            m_t = P.tet_mass[t];
        } else {
            int64_t i, j, k;
            if (!cube_of_unit(P, t / 6, i, j, k)) {
                set_error(P.ws, 3, (int)((t / 6) & 0x7fffffff));
                continue;
            }
            lattice_tet<T>(P, i, j, k, (int)(t % 6), v, base, res);
            m_t = P.m_tet;
        }
        TetSetup<T> ts;
        const bool negative = tet_setup<T>(v, ts);
        if (negative) swap12(res);
        if (STATS) {
            cnt.u[ST_TETS]++;
            cnt.mass_in += m_t;
            cnt.u[ST_INVERTED] += (negative != (P.src != SRC_TETS && kuhn_negative((int)(t % 6)))) ? 1 : 0;
        }
        if (!tet_ok(base, ts)) {
            set_error(P.ws, 4, (int)(t & 0x7fffffff));
            continue;
        }
        cnt.add_tgt(P, m_t);
        if (ts.vol6 == 0.0) {
            int c[3];
            centroid_cell(ts.v, c);
            if (!deposit_cell(P, base[0] + c[0], base[1] + c[1], base[2] + c[2], m_t) && STATS) cnt.dropped += m_t;
            cnt.add_dep(m_t);
            if (STATS) { cnt.u[ST_DEGENERATE]++; cnt.u[ST_OVERLAPPED]++; }
            continue;
        }
        const int64_t ncell = (int64_t)ts.dim[0] * ts.dim[1] * ts.dim[2];
        if (STATS) { cnt.u[ST_BBOX_CELLS] += ncell; cnt.u[ST_BIN0 + size_bin(ncell)]++; }
        if (ncell == 1) {
            if (!deposit_cell(P, base[0] + ts.lo[0], base[1] + ts.lo[1], base[2] + ts.lo[2], m_t) && STATS)
                cnt.dropped += m_t;
            cnt.add_dep(m_t);
            if (STATS) { cnt.u[ST_SINGLE_CELL]++; cnt.u[ST_OVERLAPPED]++; }
            continue;
        }
        // FP32 guard: ill-conditioned tetrahedra are clipped in float64 from their exact vertices
        const bool g64 = (sizeof(T) == 4) && !(ts.kappa <= P.kappa_max);
        bool flat;
        if constexpr (sizeof(T) == 4) flat = g64 && near_flat(P, ts);
        else flat = near_flat(P, ts.vol6, ts.dim, base);
        int c[3];
        if (flat && exactly_flat(P, t, c)) {
            if (!deposit_cell(P, c[0], c[1], c[2], m_t) && STATS) cnt.dropped += m_t;
            cnt.add_dep(m_t);
            if (STATS) { cnt.u[ST_DEGENERATE]++; cnt.u[ST_OVERLAPPED]++; }
            continue;
        }
        double rho = 6.0 * m_t / ts.vol6;
        if constexpr (sizeof(T) == 4) {
            if (g64) rho = 6.0 * m_t / exact_vol6(ts.v, res, ts.vol6);
        }
        for (int iz = 0; iz < ts.dim[2]; ++iz)
            for (int iy = 0; iy < ts.dim[1]; ++iy)
                for (int ix = 0; ix < ts.dim[0]; ++ix) {
                    const int cx = ts.lo[0] + ix, cy = ts.lo[1] + iy, cz = ts.lo[2] + iz;
                    const int cls = classify_cell<T>(ts.n, ts.e, ts.pos, ts.neg, (T)cx, (T)cy, (T)cz);
                    double vol = 0.0;
                    if (cls == CELL_INSIDE) {
                        vol = 1.0;
                        if (STATS) cnt.u[ST_INSIDE_CELLS]++;
                    } else if (cls == CELL_PARTIAL) {
                        P3<T> p[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) p[q] = mk<T>(ts.v[q].x - (T)cx, ts.v[q].y - (T)cy, ts.v[q].z - (T)cz);
                        if constexpr (sizeof(T) == 4) {
                            if (g64) {
                                P3<double> pd[4];
                                exact_vertices(ts.v, res, cx, cy, cz, pd);
                                vol = overlap_volume_fp64(pd);
                                if (STATS) cnt.u[ST_FP64_REDOS]++;
                            } else {
                                T err;
                                vol = (double)overlap_volume_ax<T>(p, ts.n, ts.axis, ts.lx, ts.ly, err);
                            }
                        } else {
                            T err;
                            vol = (double)overlap_volume_ax<T>(p, ts.n, ts.axis, ts.lx, ts.ly, err);
                        }
                        if (STATS) cnt.u[ST_PARTIAL_CLIPS]++;
                    }
                    if (vol > 0.0) {
                        if (STATS) cnt.u[ST_OVERLAPPED]++;
                        const double m = rho * vol;
                        cnt.add_dep(m);
                        if (!deposit_cell(P, base[0] + cx, base[1] + cy, base[2] + cz, m) &&
                            STATS)
                            cnt.dropped += m;
                    }
                }
    }
    if (STATS) cnt.flush(P.ws);
    if (P.fixup || STATS) cnt.flush_mass(P, P.ws);
}

// ---------------------------------------------------------------------------
// every step in float64, by the warp-cooperative column clip
// ---------------------------------------------------------------------------
// Cell by cell for a tetrahedron that the run queue cannot hold (more than 2^25 cells, or 2^19 and more
// on a side), record t: its cells dealt to the lanes in turn.
__device__ __noinline__ void plain_cells(const DepositParams &P, WarpSmem *S, int t, int lane)
{
    const GuardSmem *G = guard_smem(S);
    P3<double> v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = mk<double>(G->v[3 * q][t], G->v[3 * q + 1][t], G->v[3 * q + 2][t]);
    TetSetup<double> ts;
    tet_setup<double>(v, ts);
    const double rho = G->rho[t];
    const int bx = S->base[0][t], by = S->base[1][t], bz = S->base[2][t];
    // cell number lane, then 32 on: each coordinate moves by less than its range, with one carry
    const int dx = ts.dim[0], dy = ts.dim[1];
    const int sx = 32 % dx, sy = 32 / dx % dy, sz = 32 / dx / dy;
    int ix = lane % dx, iy = lane / dx % dy, iz = lane / dx / dy;
    while (iz < ts.dim[2]) {
        const int cx = ts.lo[0] + ix, cy = ts.lo[1] + iy, cz = ts.lo[2] + iz;
        const int cls = classify_cell<double>(ts.n, ts.e, ts.pos, ts.neg, (double)cx, (double)cy, (double)cz);
        double vol = cls == CELL_INSIDE ? 1.0 : 0.0;
        if (cls == CELL_PARTIAL) {
            P3<double> p[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) p[q] = mk<double>(ts.v[q].x - cx, ts.v[q].y - cy, ts.v[q].z - cz);
            double err;
            vol = overlap_volume_ax<double>(p, ts.n, ts.axis, ts.lx, ts.ly, err);
        }
        if (vol > 0.0) deposit_cell<Acc::F64>(P, bx + cx, by + cy, bz + cz, rho * vol);
        ix += sx;
        if (ix >= dx) { ix -= dx; ++iy; }
        iy += sy;
        if (iy >= dy) { iy -= dy; ++iz; }
        iz += sz;
    }
}

// PSE_FP64_PLAIN without statistics: the warp-cooperative schedule with the guarded pass's
// float64 column clip for every tetrahedron.  Vertices, volume, bounding box and deposits are
// float64; the float32 copies in the record only choose work: the clip's axis, frame and faces,
// and the runs that lie wholly inside or outside by a margin above their rounding (1e-6 (L + 1)^3
// on the plane values for an extent of L cells); everything else is clipped.
//
// The float64 pipe bounds both this and the thread-per-tetrahedron kernel (16 cycles a warp
// instruction).  That kernel clips cell by cell with 9 of 32 lanes active; here one clip serves
// two cells, with 2.5 times fewer float64 operations, and the lanes are full: 48^3 on 96^3 takes 213 ms
// there and 16.4 here, the masses equal to 3e-16 (norm).
__global__ void __launch_bounds__(kCoopThreads, 2) k_warp_plain(const DepositParams P)
{
    WarpSmem *S = warp_smem(true);
    GuardSmem *G = guard_smem(S);
    const int lane = threadIdx.x & 31;
    Counters cnt;
    cnt.zero_mass();
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(&P.ws->work_counter, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if ((int64_t)item >= P.n_items) break;
        int64_t g = (int64_t)item, ci = 0, cj = 0, ck = 0;
        int s = 0;
        if (P.src != SRC_TETS) {
            s = (int)(item % 6);
            g = (int64_t)(item / 6);
        }
        const int64_t u = g * P.group + lane;
        bool have = lane < P.group && u < P.n_units;
        if (have && P.src != SRC_TETS && !cube_of_unit(P, u, ci, cj, ck)) {
            set_error(P.ws, 3, (int)(u & 0x7fffffff));
            have = false;
        }
        int npairs = 0;
        bool large = false;
        if (have) {
            P3<double> v[4];
            int base[3];
            double m_t;
            if (P.src == SRC_TETS) {
                explicit_tet<double>(P, u, v, base);
                m_t = P.tet_mass[u];
            } else {
                lattice_tet<double>(P, ci, cj, ck, s, v, base);
                m_t = P.m_tet;
            }
            const double d6 = det6(v), vol6 = fabs(d6);
            if (d6 < 0.0) {
                const P3<double> t = v[1];
                v[1] = v[2];
                v[2] = t;
            }
            TetSetup<float> ts;  // of the float32 vertices; its cell range replaced by the float64 one
            P3<float> vf[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) vf[q] = mk<float>((float)v[q].x, (float)v[q].y, (float)v[q].z);
            {
                const double mnx = fmin(fmin(v[0].x, v[1].x), fmin(v[2].x, v[3].x)), mxx = fmax(fmax(v[0].x, v[1].x), fmax(v[2].x, v[3].x));
                const double mny = fmin(fmin(v[0].y, v[1].y), fmin(v[2].y, v[3].y)), mxy = fmax(fmax(v[0].y, v[1].y), fmax(v[2].y, v[3].y));
                const double mnz = fmin(fmin(v[0].z, v[1].z), fmin(v[2].z, v[3].z)), mxz = fmax(fmax(v[0].z, v[1].z), fmax(v[2].z, v[3].z));
                P3<float> w[4] = {vf[0], vf[1], vf[2], vf[3]};
                tet_setup<float>(w, ts);
                const double big = 16777216.0;
                const bool fin = d6 == d6 && mnx > -big && mxx < big && mny > -big && mxy < big && mnz > -big && mxz < big;
                ts.lo[0] = fin ? (int)floor(mnx) : 0;
                ts.lo[1] = fin ? (int)floor(mny) : 0;
                ts.lo[2] = fin ? (int)floor(mnz) : 0;
                ts.dim[0] = fin ? (int)floor(mxx) - ts.lo[0] + 1 : 0;
                ts.dim[1] = fin ? (int)floor(mxy) - ts.lo[1] + 1 : 0;
                ts.dim[2] = fin ? (int)floor(mxz) - ts.lo[2] + 1 : 0;
            }
            const int64_t ncell = (int64_t)ts.dim[0] * ts.dim[1] * ts.dim[2];
            if (!tet_ok(base, ts)) {
                set_error(P.ws, 4, lane);
            } else if (vol6 == 0.0) {
                int c[3];
                centroid_cell(v, c);
                deposit_cell<Acc::F64>(P, base[0] + c[0], base[1] + c[1], base[2] + c[2], m_t);
            } else if (ncell == 1) {
                deposit_cell<Acc::F64>(P, base[0] + ts.lo[0], base[1] + ts.lo[1], base[2] + ts.lo[2], m_t);
            } else if (!near_flat(P, vol6, ts.dim, base) ||
                       deposit_flat<Acc::F64>(P, P.src == SRC_TETS ? u : 6 * u + s, m_t) == 0) {
                large = ncell > (int64_t)(1 << 25) || !dims_fit_queue(ts.dim);
                npairs = large ? 0 : (int)run_count(ts.dim, ts.axis);
                const float l1 = 1.f + (float)max(ts.dim[0], max(ts.dim[1], ts.dim[2])), margin = 1e-6f * l1 * l1 * l1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    S->v[3 * q][lane] = vf[q].x;
                    S->v[3 * q + 1][lane] = vf[q].y;
                    S->v[3 * q + 2][lane] = vf[q].z;
                    G->v[3 * q][lane] = v[q].x;
                    G->v[3 * q + 1][lane] = v[q].y;
                    G->v[3 * q + 2][lane] = v[q].z;
                    S->n[3 * q][lane] = ts.n[q].x;
                    S->n[3 * q + 1][lane] = ts.n[q].y;
                    S->n[3 * q + 2][lane] = ts.n[q].z;
                    S->e[q][lane] = ts.e[q];
                    S->pos[q][lane] = ts.pos[q] + margin;
                    S->neg[q][lane] = ts.neg[q] - margin;
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    S->lo[a][lane] = ts.lo[a];
                    S->dim[a][lane] = ts.dim[a];
                    S->base[a][lane] = base[a];
                }
                S->lx[lane] = ts.lx;
                S->ly[lane] = ts.ly;
                S->axis[lane] = ts.axis;
                G->rho[lane] = 6.0 * m_t / vol6;
                G->tol[lane] = f64_tolerance((double)(ts.dim[0] + ts.dim[1] + ts.dim[2]));
            }
        }
        for (unsigned left = __ballot_sync(kFull, large); left != 0u; left &= left - 1u) {
            __syncwarp();  // the records are written
            plain_cells(P, S, __ffs((int)left) - 1, lane);
        }
        coop_runs<false, false, Acc::F64, double, true>(P, S, lane, npairs, 0, cnt);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// the paper's design (Sec. 6.2), kept as a baseline: one warp per tetrahedron; its
// bounding-box cells are classified 32 at a time and the partial ones buffered and
// clipped 32 at a time (the same pair machinery and clip, with one record per warp)
// ---------------------------------------------------------------------------
template <bool STATS>
__global__ void __launch_bounds__(kCoopThreads, 2) k_warp_per_tet(const DepositParams P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WarpSmem *S = reinterpret_cast<WarpSmem *>(smem_raw) + (threadIdx.x >> 5);
    bind_residuals(P, S);
    const int lane = threadIdx.x & 31;
    Counters cnt;
    if (STATS) cnt.zero();
    cnt.zero_mass();
    const int64_t n_tets = (P.src == SRC_TETS) ? P.n_units : 6 * P.n_units;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(&P.ws->work_counter, 1ull);
        t = __shfl_sync(kFull, t, 0);
        if ((int64_t)t >= n_tets) break;
        int npairs = 0;
        if (lane == 0) {
            P3<float> v[4], res[4];
            int base[3];
            double m_t;
            bool ok = true;
            if (P.src == SRC_TETS) {
                explicit_tet<float>(P, (int64_t)t, v, base, res);
                m_t = P.tet_mass[t];
            } else {
                int64_t ci, cj, ck;
                ok = cube_of_unit(P, (int64_t)t / 6, ci, cj, ck);
                if (!ok) set_error(P.ws, 3, (int)(((int64_t)t / 6) & 0x7fffffff));
                if (ok) lattice_tet<float>(P, ci, cj, ck, (int)(t % 6), v, base, res);
                m_t = P.m_tet;
            }
            if (ok) {
                TetSetup<float> ts;
                const bool negative = tet_setup<float>(v, ts);
                if (negative) swap12(res);
                if (STATS) {
                    cnt.u[ST_TETS]++;
                    cnt.mass_in += m_t;
                    cnt.u[ST_INVERTED] += (negative != (P.src != SRC_TETS && kuhn_negative((int)(t % 6)))) ? 1 : 0;
                }
                const int64_t ncell = (int64_t)ts.dim[0] * ts.dim[1] * ts.dim[2];
                const bool ok_tet = tet_ok(base, ts);
                int c[3];
                const bool flat = ok_tet && ts.vol6 != 0.0 && ncell > 1 && !(ts.kappa <= P.kappa_max) && near_flat(P, ts) &&
                                  exactly_flat(P, (int64_t)t, c);
                if (!ok_tet) {
                    set_error(P.ws, 4, (int)(t & 0x7fffffff));
                } else if (flat || ts.vol6 == 0.0 || ncell == 1) {
                    if (!flat) {
                        if (ts.vol6 == 0.0) centroid_cell(ts.v, c);
                        else { c[0] = ts.lo[0]; c[1] = ts.lo[1]; c[2] = ts.lo[2]; }
                        c[0] += base[0];
                        c[1] += base[1];
                        c[2] += base[2];
                    }
                    if (!deposit_cell(P, c[0], c[1], c[2], m_t) && STATS) cnt.dropped += m_t;
                    cnt.add_tgt(P, m_t);
                    cnt.add_dep(m_t);
                    if (STATS) {
                        cnt.u[flat || ts.vol6 == 0.0 ? ST_DEGENERATE : ST_SINGLE_CELL]++;
                        cnt.u[ST_OVERLAPPED]++;
                        if (ts.vol6 != 0.0) { cnt.u[ST_BBOX_CELLS] += ncell; cnt.u[ST_BIN0 + size_bin(ncell)]++; }
                    }
                } else if (ncell > (int64_t)(1 << 25) || !dims_fit_queue(ts.dim)) {
                    set_error(P.ws, 2, (int)(t & 0x7fffffff));
                } else {
                    npairs = (int)ncell;
                    cnt.add_tgt(P, m_t);
                    if (STATS) { cnt.u[ST_BBOX_CELLS] += ncell; cnt.u[ST_BIN0 + size_bin(ncell)]++; }
                    store_record<kPassAll>(S, 0, ts, res, ts.lo, ts.dim, base, m_t, P.kappa_max, false);
                }
            }
        }
        __syncwarp();
        coop_cells<STATS, Acc::RUNTIME>(P, S, lane, npairs, cnt);
        __syncwarp();
    }
    if (STATS) cnt.flush(P.ws);
    if (P.fixup || STATS) cnt.flush_mass(P, P.ws);
}

// ---------------------------------------------------------------------------
// binned schedule: the bin pass queues every tetrahedron whose bounding box has more
// than split_cells cells (warp-aggregated appends); the scan turns their cell counts
// into work items of chunk_cells cells.
// ---------------------------------------------------------------------------
// Without a cost model a tetrahedron is queued when its bounding box has more than
// split_cells cells (the row path recomputes the same test).  With one, the bin pass
// predicts each tetrahedron's partial clips (warp MLP on the tensor cores), queues it
// when the prediction exceeds split_cells, and marks it in the qbits bitmap that the row
// path reads.
template <bool MODEL>
__global__ void __launch_bounds__(128) k_bin_pass(const DepositParams P)
{
    __shared__ MlpSmem msm[MODEL ? 4 : 1];
    const int lane = threadIdx.x & 31;
    const int64_t n_tets = (P.src == SRC_TETS) ? P.n_units : 6 * P.n_units;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // whole warps iterate together so that the ballot and the warp MLP see every lane
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < n_tets; t0 += stride) {
        const int64_t t = t0 + lane;
        bool cand = false;
        int64_t ncell = 0, npair = 0;
        float f[kNFeat];
        if (MODEL) {
#pragma unroll
            for (int q = 0; q < kNFeat; ++q) f[q] = 0.f;
        }
        if (t < n_tets) {
            P3<float> v[4];
            int base[3];
            bool ok = true;
            if (P.src == SRC_TETS) {
                explicit_tet<float>(P, t, v, base);
            } else {
                int64_t ci, cj, ck;
                ok = cube_of_unit(P, t / 6, ci, cj, ck);
                if (ok) lattice_tet<float>(P, ci, cj, ck, (int)(t % 6), v, base);
            }
            if (ok) {
                TetSetup<float> ts;
                tet_setup<float>(v, ts);
                ncell = (int64_t)ts.dim[0] * ts.dim[1] * ts.dim[2];
                cand = tet_ok(base, ts) && ts.vol6 != 0.0 && ncell > 1 && ncell <= (int64_t)INT32_MAX;
                // the work items count pairs: column runs (both passes clip runs)
                if (cand) npair = run_count(ts.dim, ts.axis);
                if (MODEL && cand) tet_features(ts, f);
            }
        }
        bool queue;
        if (MODEL) {
            float y[kNOut];
            mlp_warp(P.model, msm[(threadIdx.x >> 5) & 3], lane, f, y);
            queue = cand && expm1f(y[1]) > (float)P.split_cells;
        } else {
            queue = cand && ncell > P.split_cells;
        }
        const unsigned bal = __ballot_sync(kFull, queue);
        if (bal) {
            unsigned long long b0 = 0;
            if (lane == 0) b0 = atomicAdd(&P.ws->queue_count, (unsigned long long)__popc(bal));
            b0 = __shfl_sync(kFull, b0, 0);
            if (queue) {
                const int64_t idx = (int64_t)b0 + __popc(bal & ((1u << lane) - 1u));
                if (idx < P.q_cap) {
                    P.q_tet[idx] = t;
                    P.q_cells[idx] = (int32_t)npair;
                    if (MODEL) atomicOr(P.qbits + (t >> 5), 1u << (t & 31));
                } else {
                    P.ws->queue_overflow = 1;
                }
            }
        }
    }
}

// One block: chunk_start = exclusive prefix of ceil(q_cells / chunk_cells).
__global__ void __launch_bounds__(1024) k_chunk_scan(const DepositParams P)
{
    __shared__ long long part[1024];
    Workspace *ws = P.ws;
    if (ws->queue_overflow) {
        if (threadIdx.x == 0) ws->n_chunk_items = 0;
        return;
    }
    const int64_t q = min((int64_t)ws->queue_count, P.q_cap);
    const int64_t per = (q + blockDim.x - 1) / blockDim.x;
    const int64_t b = threadIdx.x * per, e = min(q, b + per);
    const int64_t cc = P.chunk_cells;
    long long sum = 0;
    for (int64_t i = b; i < e; ++i) sum += (P.q_cells[i] + cc - 1) / cc;
    part[threadIdx.x] = sum;
    __syncthreads();
    // inclusive scan of the per-thread sums (Hillis-Steele)
    for (int o = 1; o < (int)blockDim.x; o <<= 1) {
        const long long y = (threadIdx.x >= (unsigned)o) ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += y;
        __syncthreads();
    }
    long long run = part[threadIdx.x] - sum;
    for (int64_t i = b; i < e; ++i) {
        P.chunk_start[i] = run;
        run += (P.q_cells[i] + cc - 1) / cc;
    }
    if (threadIdx.x == blockDim.x - 1) {
        P.chunk_start[q] = part[threadIdx.x];
        ws->n_chunk_items = (unsigned long long)part[threadIdx.x];
    }
}

// ---------------------------------------------------------------------------
// end of an FP32 deposit: compensated pairs (hi, lo) become hi + lo in FP64, in place (COMP),
// and the mass renormalisation out *= (sum of m_t) / (sum of deposits) (SCALE)
// ---------------------------------------------------------------------------
template <bool COMP, bool SCALE>
__global__ void k_finish(double *__restrict__ out, long long n, const Workspace *__restrict__ ws)
{
    double f = 1.0;
    if (SCALE) {
        const double dep = ws->mass_deposited + ws->mass_deposited_lo;
        if (dep > 0.0) f = (ws->mass_target + ws->mass_target_lo) / dep;
        else if (!COMP) return;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double v;
        if (COMP) {
            const float2 p = reinterpret_cast<const float2 *>(out)[i];
            v = (double)p.x + (double)p.y;
        } else {
            v = out[i];
        }
        out[i] = v * f;
    }
}

// ---------------------------------------------------------------------------
// tessellation builder
// ---------------------------------------------------------------------------
__global__ void k_build_tets(const float *__restrict__ pos, long long n0, long long n1, long long n2, long long nc0,
                             long long nc1, int periodic, double box, int32_t *__restrict__ vidx,
                             float *__restrict__ vol, long long n_tets)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n_tets;
         t += (long long)gridDim.x * blockDim.x) {
        const long long c = t / 6;
        const int s = (int)(t % 6);
        const long long ci = c % nc0, cj = (c / nc0) % nc1, ck = c / (nc0 * nc1);
        int o1[3], o2[3];
        kuhn_offsets(s, o1, o2);
        long long id[4];
        double x[4][3];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            long long i = ci, j = cj, k = ck;
            if (q == 1) { i += o1[0]; j += o1[1]; k += o1[2]; }
            if (q == 2) { i += o2[0]; j += o2[1]; k += o2[2]; }
            if (q == 3) { i += 1; j += 1; k += 1; }
            if (periodic) { i = wrap_idx(i, n0); j = wrap_idx(j, n1); k = wrap_idx(k, n2); }
            id[q] = i + n0 * (j + n1 * k);
#pragma unroll
            for (int a = 0; a < 3; ++a) x[q][a] = (double)__ldg(pos + 3 * id[q] + a);
        }
        if (periodic) {
#pragma unroll
            for (int q = 1; q < 4; ++q)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double d = x[q][a] - x[0][a];
                    x[q][a] -= (d >= 0.5 * box) ? box : ((d < -0.5 * box) ? -box : 0.0);
                }
        }
        if (vidx) {
#pragma unroll
            for (int q = 0; q < 4; ++q) vidx[4 * t + q] = (int32_t)id[q];
        }
        if (vol) {
            const double ax = x[1][0] - x[0][0], ay = x[1][1] - x[0][1], az = x[1][2] - x[0][2];
            const double bx = x[2][0] - x[0][0], by = x[2][1] - x[0][1], bz = x[2][2] - x[0][2];
            const double cx = x[3][0] - x[0][0], cy = x[3][1] - x[0][1], cz = x[3][2] - x[0][2];
            vol[t] = (float)((ax * (by * cz - bz * cy) - ay * (bx * cz - bz * cx) + az * (bx * cy - by * cx)) / 6.0);
        }
    }
}

}  // namespace

cudaError_t launch_thread_per_tet(const DepositParams &p, bool fp64, bool stats, cudaStream_t st)
{
    const int threads = 128;
    const int64_t n_tets = (p.src == SRC_TETS) ? p.n_units : 6 * p.n_units;
    const void *k = fp64 ? (stats ? (const void *)k_thread_per_tet<double, true> : (const void *)k_thread_per_tet<double, false>)
                         : (stats ? (const void *)k_thread_per_tet<float, true> : (const void *)k_thread_per_tet<float, false>);
    int64_t blocks = (n_tets + threads - 1) / threads;
    const int64_t cap = (int64_t)persistent_blocks(k, threads, 0) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (fp64) {
        if (stats) k_thread_per_tet<double, true><<<(unsigned)blocks, threads, 0, st>>>(p);
        else k_thread_per_tet<double, false><<<(unsigned)blocks, threads, 0, st>>>(p);
    } else {
        if (stats) k_thread_per_tet<float, true><<<(unsigned)blocks, threads, 0, st>>>(p);
        else k_thread_per_tet<float, false><<<(unsigned)blocks, threads, 0, st>>>(p);
    }
    return cudaGetLastError();
}

cudaError_t launch_warp_plain(const DepositParams &p, cudaStream_t st)
{
    const void *k = (const void *)k_warp_plain;
    const size_t smem = warp_smem_bytes(kCoopThreads / 32, true);
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    int64_t blocks = persistent_blocks(k, kCoopThreads, smem);
    const int64_t need = (p.n_items + kCoopThreads / 32 - 1) / (kCoopThreads / 32);
    if (need < blocks) blocks = need < 1 ? 1 : need;
    void *args[] = {const_cast<DepositParams *>(&p)};
    return cudaLaunchKernel(k, dim3((unsigned)blocks), dim3(kCoopThreads), args, smem, st);
}

cudaError_t launch_warp_coop(const DepositParams &p, bool stats, int blocks_per_sm, cudaStream_t st)
{
    if (p.comp) return launch_coop_comp(p, stats, blocks_per_sm, false, p.n_items, st);
    return launch_coop<false, Acc::F64>(p, stats, blocks_per_sm, p.n_items, st);
}

cudaError_t launch_warp_per_tet(const DepositParams &p, bool stats, cudaStream_t st)
{
    const int threads = kCoopThreads;
    const size_t smem = warp_smem_bytes(threads / 32, false);
    const void *k = stats ? (const void *)k_warp_per_tet<true> : (const void *)k_warp_per_tet<false>;
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    int blocks = persistent_blocks(k, threads, smem);
    if (blocks > kMaxWarpBlocks) blocks = kMaxWarpBlocks;
    void *args[] = {const_cast<DepositParams *>(&p)};
    return cudaLaunchKernel(k, dim3(blocks), dim3(threads), args, smem, st);
}

cudaError_t launch_binned(const DepositParams &p, bool stats, int blocks_per_sm, cudaStream_t st)
{
    const int64_t n_tets = (p.src == SRC_TETS) ? p.n_units : 6 * p.n_units;
    int64_t blocks = (n_tets + 127) / 128;
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (blocks < 1) blocks = 1;
    if (p.model) k_bin_pass<true><<<(unsigned)blocks, 128, 0, st>>>(p);
    else k_bin_pass<false><<<(unsigned)blocks, 128, 0, st>>>(p);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_chunk_scan<<<1, 1024, 0, st>>>(p);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    // the chunk count is known only on the device: size the grid for the rows plus the
    // largest possible number of chunk items (the persistent grid is capped anyway)
    if (p.comp) return launch_coop_comp(p, stats, blocks_per_sm, true, p.n_items + p.q_cap, st);
    return launch_coop<true, Acc::F64>(p, stats, blocks_per_sm, p.n_items + p.q_cap, st);
}

cudaError_t launch_finish(double *out, int64_t n, const Workspace *ws, bool comp, bool scale, cudaStream_t st)
{
    const int threads = 256;
    int64_t blocks = (n + threads - 1) / threads;
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (blocks < 1) blocks = 1;
    if (comp && scale) k_finish<true, true><<<(unsigned)blocks, threads, 0, st>>>(out, n, ws);
    else if (comp) k_finish<true, false><<<(unsigned)blocks, threads, 0, st>>>(out, n, ws);
    else if (scale) k_finish<false, true><<<(unsigned)blocks, threads, 0, st>>>(out, n, ws);
    return cudaGetLastError();
}

cudaError_t launch_build_tets(const float *pos, const int64_t n[3], const int64_t nc[3], int periodic, double box,
                              int32_t *vidx, float *vol, int64_t n_tets, cudaStream_t st)
{
    const int threads = 256;
    int64_t blocks = (n_tets + threads - 1) / threads;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (blocks < 1) blocks = 1;
    k_build_tets<<<(unsigned)blocks, threads, 0, st>>>(pos, n[0], n[1], n[2], nc[0], nc[1], periodic, box, vidx, vol,
                                                        n_tets);
    return cudaGetLastError();
}

}  // namespace pse
