// common.cuh -- device building blocks shared by the uniform-grid (deposit.cu) and
// octree (octree.cu) deposit kernels: tetrahedron sources, cell deposits, counters
// and the warp-cooperative (tetrahedron, cell) pair machinery.
#pragma once

#include "column.cuh"
#include "internal.h"

namespace pse {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void kuhn_offsets(int s, int (&o1)[3], int (&o2)[3])
{
    // axis permutations (a, b, c): xyz, xzy, yxz, yzx, zxy, zyx
    const int a = (s < 2) ? 0 : (s < 4) ? 1 : 2;
    const int b = (s == 0) ? 1 : (s == 1) ? 2 : (s == 2) ? 0 : (s == 3) ? 2 : (s == 4) ? 0 : 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o1[k] = (k == a) ? 1 : 0;
        o2[k] = (k == a || k == b) ? 1 : 0;
    }
}

// The Lagrangian orientation of Kuhn tetrahedron s is the parity of its axis permutation:
// xzy, yxz and zyx are odd, so those tetrahedra start with a negative signed volume.  A
// tetrahedron is inverted (turned inside out by shell crossing) when its signed volume
// now has the other sign.
__device__ __forceinline__ bool kuhn_negative(int s) { return s == 1 || s == 2 || s == 5; }

// floor to int for coordinates in grid units; non-finite or out-of-range values map to
// kBadCoord, which tet_ok() rejects before anything is indexed with them.
constexpr int kBadCoord = -(1 << 30);

__device__ __forceinline__ int safe_floor(double x)
{
    return (x > -1073741824.0 && x < 1073741824.0) ? (int)floor(x) : kBadCoord;
}

// A tetrahedron is processed only if its base cell, bounding box and volume are sane.  A NaN
// coordinate drops out of the bounding box's minima and maxima but not of the volume (looked at in
// float32, as kappa takes it).
template <class T>
__device__ __forceinline__ bool tet_ok(const int (&base)[3], const TetSetup<T> &ts)
{
    bool ok = !isnan((float)ts.vol6);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ok = ok && base[a] != kBadCoord && ts.dim[a] >= 1 && ts.dim[a] <= (1 << 24) &&
             ts.lo[a] > -(1 << 24) && ts.lo[a] < (1 << 24);
    }
    return ok;
}

__device__ __forceinline__ int64_t wrap_idx(int64_t i, int64_t n)
{
    if (i >= n) i -= n;
    if (i < 0) i += n;
    return i;
}

// The float32 positions of the vertices of tetrahedron s of Lagrangian cube (ci, cj, ck).  The
// four particles are reached from corner 000 by steps along the axes (wrapped on periodic
// lattices), so one particle index is formed and the others are added to it.
__device__ __forceinline__ void lattice_positions(const DepositParams &P, int64_t ci, int64_t cj, int64_t ck, int s,
                                                  float (&x)[4][3])
{
    const int64_t r1 = 3 * P.n[0], r2 = r1 * P.n[1];
    const int64_t d0 = (P.periodic && ci + 1 == P.n[0]) ? 3 - r1 : 3;
    const int64_t d1 = (P.periodic && cj + 1 == P.n[1]) ? r1 - r2 : r1;
    const int64_t d2 = (P.periodic && !P.slab && ck + 1 == P.n[2]) ? r2 - r2 * P.n[2] : r2;
    // axis permutations (a, b, c): xyz, xzy, yxz, yzx, zxy, zyx
    const int a = s >> 1, b = (s == 0 || s == 5) ? 1 : ((s == 1 || s == 3) ? 2 : 0);
    const float *p[4];
    p[0] = P.pos + (3 * ci + r1 * cj + r2 * ck);
    p[1] = p[0] + (a == 0 ? d0 : (a == 1 ? d1 : d2));
    p[2] = p[1] + (b == 0 ? d0 : (b == 1 ? d1 : d2));
    p[3] = p[0] + (d0 + d1 + d2);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) x[q][c] = __ldg(p[q] + c);
}

// Whether a vertex may need a periodic shift: some coordinate is not within 0.49 box of corner
// 000's in float32 (a tetrahedron across the box boundary, or non-finite).  When not, every
// nearest image is the vertex itself and the float64 decisions are not needed.
__device__ __forceinline__ bool may_shift(const DepositParams &P, const float (&x)[4][3])
{
    const float near = 0.49f * (float)P.box;
    bool all = true;
#pragma unroll
    for (int q = 1; q < 4; ++q)
#pragma unroll
        for (int a = 0; a < 3; ++a) all = all && fabsf(x[q][a] - x[0][a]) < near;
    return P.periodic && !all;
}

// Periodic unwrap: coordinate v is moved by -box when v - v0 >= box/2 and by +box when
// v - v0 < -box/2 (nearest image), decided in float64 on the float32 inputs.
__device__ __forceinline__ int image_shift(const DepositParams &P, float v, float v0)
{
    const double d = (double)v - (double)v0;
    return (d >= 0.5 * P.box) ? -1 : ((d < -0.5 * P.box) ? 1 : 0);
}

// The nine shifts of vertices 1..3 against vertex 0, 2 bits each (0, 1: +box, 2: -box; see
// shift_of), for the tetrahedra that may_shift picks out; out of line to keep hot code small.
__device__ __noinline__ unsigned far_shifts(double box, float a0, float a1, float a2, float b0, float b1, float b2,
                                            float c0, float c1, float c2, float d0, float d1, float d2)
{
    const float v0[3] = {a0, a1, a2}, v[9] = {b0, b1, b2, c0, c1, c2, d0, d1, d2};
    unsigned bits = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double d = (double)v[i] - (double)v0[i % 3];
        bits |= ((d >= 0.5 * box) ? 2u : ((d < -0.5 * box) ? 1u : 0u)) << (2 * i);
    }
    return bits;
}
__device__ __forceinline__ unsigned tet_shift_bits(const DepositParams &P, const float (&x)[4][3])
{
    if (!may_shift(P, x)) return 0u;
    return far_shifts(P.box, x[0][0], x[0][1], x[0][2], x[1][0], x[1][1], x[1][2], x[2][0], x[2][1], x[2][2], x[3][0],
                      x[3][1], x[3][2]);
}
__device__ __forceinline__ int shift_of(unsigned bits, int q, int a)
{
    const int b = q == 0 ? 0 : (int)((bits >> (2 * (3 * (q - 1) + a))) & 3u);
    return b == 2 ? -1 : b;
}

// Vertices of tetrahedron s of Lagrangian cube (ci, cj, ck), in grid units relative to
// the base cell (the cell holding corner 000), each corner at its periodic image nearest to
// corner 000.
template <class T>
__device__ __forceinline__ void lattice_tet(const DepositParams &P, int64_t ci, int64_t cj, int64_t ck, int s,
                                            P3<T> (&v)[4], int (&base)[3], P3<float> *res = nullptr)
{
    float x[4][3];
    lattice_positions(P, ci, cj, ck, s, x);
#pragma unroll
    for (int a = 0; a < 3; ++a) base[a] = safe_floor((double)x[0][a] * P.scale_d[a]);
    T c[4][3];
    float rr[4][3];
    // off: the vertex's periodic image and the base cell, in cells (at most 2^30 + 2^24)
    auto place = [&](int q, int a, int off) {
        if constexpr (sizeof(T) == 4) {
            c[q][a] = fmaf(x[q][a], P.scale_f[a], (float)off);
            if (res) rr[q][a] = (float)(fma((double)x[q][a], P.scale_d[a], (double)off) - (double)c[q][a]);
        } else {
            c[q][a] = fma((double)x[q][a], P.scale_d[a], (double)off);
        }
    };
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int a = 0; a < 3; ++a) place(q, a, -base[a]);
    const unsigned shifts = tet_shift_bits(P, x);
    if (shifts != 0) {
#pragma unroll
        for (int q = 1; q < 4; ++q)
#pragma unroll
            for (int a = 0; a < 3; ++a) place(q, a, shift_of(shifts, q, a) * (int)P.g[a] - base[a]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v[q] = mk<T>(c[q][0], c[q][1], c[q][2]);
        if (sizeof(T) == 4 && res) res[q] = mk<float>(rr[q][0], rr[q][1], rr[q][2]);
    }
}

template <class T>
__device__ __forceinline__ void explicit_tet(const DepositParams &P, int64_t t, P3<T> (&v)[4], int (&base)[3],
                                             P3<float> *res = nullptr)
{
    const float *p = P.verts + 12 * t;
    float x[4][3];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int a = 0; a < 3; ++a) x[q][a] = __ldg(p + 3 * q + a);
#pragma unroll
    for (int a = 0; a < 3; ++a) base[a] = safe_floor((double)x[0][a] * P.scale_d[a]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        T c[3];
        float rr[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if constexpr (sizeof(T) == 4) {
                c[a] = fmaf(x[q][a], P.scale_f[a], (float)(-base[a]));
                if (res) rr[a] = (float)(fma((double)x[q][a], P.scale_d[a], (double)(-base[a])) - (double)c[a]);
            } else {
                c[a] = fma((double)x[q][a], P.scale_d[a], (double)(-base[a]));
            }
        }
        v[q] = mk<T>(c[0], c[1], c[2]);
        if (sizeof(T) == 4 && res) res[q] = mk<float>(rr[0], rr[1], rr[2]);
    }
}

// The float32 vertices of the FP32 path are rounded; res holds the rounding residuals
// (exact value = (double)v + (double)res, both terms exact in float64), so that the
// guarded float64 clips and volume use the exact tetrahedron.
__device__ __forceinline__ void swap12(P3<float> (&r)[4])
{
    const P3<float> t = r[1];
    r[1] = r[2];
    r[2] = t;
}

// exact vertices in the frame of cell (cx, cy, cz) of the base frame
__device__ __forceinline__ void exact_vertices(const P3<float> (&v)[4], const P3<float> (&r)[4], int cx, int cy,
                                               int cz, P3<double> (&pd)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        pd[q] = mk<double>(((double)v[q].x + (double)r[q].x) - (double)cx, ((double)v[q].y + (double)r[q].y) - (double)cy,
                           ((double)v[q].z + (double)r[q].z) - (double)cz);
}

// |6V| of the exact tetrahedron (falls back to the float32 one if that is 0); flip is set
// when the exact tetrahedron's orientation is the opposite of the float32 one's (a sliver
// thinner than float32 rounding can turn over when rounded)
__device__ __forceinline__ double exact_vol6(const P3<float> (&v)[4], const P3<float> (&r)[4], double vol6_f32,
                                             bool *flip = nullptr)
{
    P3<double> pd[4];
    exact_vertices(v, r, 0, 0, 0, pd);
    const double s = det6(pd);
    if (flip) *flip = s < 0.0;
    const double d = fabs(s);
    return d > 0.0 ? d : vol6_f32;
}

// Coordinates of Lagrangian cube c.  Lattices of 2^32 cubes and more divide out of line.
__device__ __noinline__ void cube_coords_far(const int64_t (&nc)[3], int64_t c, int64_t &i, int64_t &j, int64_t &k)
{
    i = c % nc[0];
    j = (c / nc[0]) % nc[1];
    k = c / (nc[0] * nc[1]);
}
__device__ __forceinline__ void cube_coords(const DepositParams &P, int64_t c, int64_t &i, int64_t &j, int64_t &k)
{
    if (P.nc[0] * P.nc[1] * P.nc[2] <= (int64_t)0xffffffffll) {
        const unsigned n0 = (unsigned)P.nc[0], n1 = (unsigned)P.nc[1];
        const unsigned row = (unsigned)c / n0, layer = row / n1;
        i = (unsigned)c - row * n0;
        j = row - layer * n1;
        k = layer;
    } else {
        cube_coords_far(P.nc, c, i, j, k);
    }
}

// Lagrangian cube of work unit u; false (and nothing read) for an out-of-range cube id.
__device__ __forceinline__ bool cube_of_unit(const DepositParams &P, int64_t u, int64_t &i, int64_t &j, int64_t &k)
{
    const int64_t c = (P.src == SRC_CUBE_LIST) ? P.cube_ids[u] : u;
    if (c < 0 || c >= P.nc[0] * P.nc[1] * P.nc[2]) return false;
    cube_coords(P, c, i, j, k);
    return true;
}

// How many listed guarded tetrahedra a work item of the guarded pass takes: 32 when there are
// plenty, fewer when the grid's warps would otherwise share only a few items (a listed
// tetrahedron can cover thousands of cells).
__device__ __forceinline__ int listed_per_item(int64_t listed)
{
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t per = listed / (4 * warps);
    return per < 1 ? 1 : (per > 32 ? 32 : (int)per);
}

__device__ __forceinline__ int64_t fold_cell(int64_t c, int64_t g)
{
    if (c >= -g && c < 2 * g) {
        if (c < 0) c += g;
        if (c >= g) c -= g;
        return c;
    }
    c %= g;
    return c < 0 ? c + g : c;
}

// The same for int32 cells (a base cell within +-2^30 plus an offset within 2^25; a grid has at
// most 2^24 cells a side).  A cell more than one period away is rare, and its remainder is kept
// out of line: the deposit kernels are sensitive to the size of their hot code.
__device__ __noinline__ int fold_far(int c, int g)
{
    c %= g;
    return c < 0 ? c + g : c;
}
__device__ __forceinline__ int fold_near(int c, int g)
{
    if ((unsigned)c >= (unsigned)g) {
        c += c < 0 ? g : -g;
        if ((unsigned)c >= (unsigned)g) c = fold_far(c, g);
    }
    return c;
}

// How a kernel adds to the output cells (compile-time, so that the FP64 kernels carry
// no trace of the other mode):
//  * F64: one global FP64 reduction per addend.
//  * COMP: compensated FP32 accumulation.  Until the end of the call each cell holds an
//    FP32 pair (hi at the lower 4 bytes, lo at the upper 4).  hi takes m rounded to float
//    with an atomic add that returns the previous value; the exact rounding error of that
//    add (Knuth's two-sum, exact under round-to-nearest) and the error of rounding m to
//    float go to lo.  hi + lo then carries the cell's sum to about 2^-48 relative per addend.
//  * RUNTIME: either, from P.comp (the baseline kernels).
enum class Acc : int { F64 = 0, COMP = 1, RUNTIME = 2 };

__device__ __forceinline__ void cell_add_compensated(double *addr, double m)
{
    float *hl = reinterpret_cast<float *>(addr);
    const float v = __double2float_rn(m);
    const float r = __double2float_rn(m - (double)v);
    const float old = atomicAdd(hl, v);
    const float s = __fadd_rn(old, v);
    const float bv = __fsub_rn(s, old);
    const float e = __fadd_rn(__fsub_rn(old, __fsub_rn(s, bv)), __fsub_rn(v, bv));
    const float c = __fadd_rn(e, r);
    if (c != 0.f) atomicAdd(hl + 1, c);
}

template <Acc A = Acc::RUNTIME>
__device__ __forceinline__ void cell_add(const DepositParams &P, double *addr, double m)
{
    if constexpr (A == Acc::F64) {
        atomicAdd(addr, m);
    } else if constexpr (A == Acc::COMP) {
        cell_add_compensated(addr, m);
    } else {
        if (P.comp) cell_add_compensated(addr, m);
        else atomicAdd(addr, m);
    }
}

// Add m to cell (cx, cy, cz) (unfolded grid indices); returns false if the cell is
// outside an open grid (then the mass is dropped).
template <Acc A = Acc::RUNTIME>
__device__ __forceinline__ bool deposit_cell(const DepositParams &P, int cx, int cy, int cz, double m)
{
    const int g0 = (int)P.g[0], g1 = (int)P.g[1], g2 = (int)P.g[2];
    if (P.periodic) {
        cx = fold_near(cx, g0);
        cy = fold_near(cy, g1);
        cz = fold_near(cz, g2);
    } else if ((unsigned)cx >= (unsigned)g0 || (unsigned)cy >= (unsigned)g1 || (unsigned)cz >= (unsigned)g2) {
        return false;
    }
    cell_add<A>(P, P.out + ((int64_t)cx + g0 * ((int64_t)cy + (int64_t)g1 * cz)), m);
    return true;
}

template <class T>
__device__ __forceinline__ void centroid_cell(const P3<T> (&v)[4], int (&c)[3])
{
    c[0] = (int)floor(((double)v[0].x + (double)v[1].x + (double)v[2].x + (double)v[3].x) * 0.25);
    c[1] = (int)floor(((double)v[0].y + (double)v[1].y + (double)v[2].y + (double)v[3].y) * 0.25);
    c[2] = (int)floor(((double)v[0].z + (double)v[1].z + (double)v[2].z + (double)v[3].z) * 0.25);
}

// Exactly degenerate tetrahedra on uniform grids.  The set-up works in cells, where float32 positions
// round unless cells per box is a power of two, and with them the volume of a coplanar tetrahedron: dividing by
// it gives any density.
//
// near_flat: whether the volume in cells of a tetrahedron's float64 vertices (of the float32 passes: the float32 ones
// and their residuals) may be rounding alone.  Their error is at most 6.3e-15 (|coordinates from the box's corner| +
// extent) cells, 6V's that times the normals' lengths; hardly any tetrahedron is within it.
__device__ __forceinline__ bool near_flat(const DepositParams &P, double vol6, const int (&dim)[3], const int (&base)[3])
{
    const float L = (float)(dim[0] + dim[1] + dim[2]);
    const float far = (float)(max(abs(base[0]), max(abs(base[1]), abs(base[2]))) + 2) + (float)max(P.g[0], max(P.g[1], P.g[2]));
    return fabsf((float)vol6) <= 5e-14f * (far + L) * L * L;
}
__device__ __forceinline__ bool near_flat(const DepositParams &P, const TetSetup<float> &ts, const P3<float> (&res)[4],
                                          const int (&base)[3])
{
    P3<double> pd[4];
    exact_vertices(ts.v, res, 0, 0, 0, pd);
    return near_flat(P, det6(pd), ts.dim, base);
}
// (from the float32 vertices alone, for the kernels that set up every tetrahedron and its float64 vertices rarely)
__device__ __forceinline__ bool near_flat(const DepositParams &P, const TetSetup<float> &ts)
{
    return may_be_flat(ts.kappa, (float)ts.vol6, 2.f + (float)max(P.g[0], max(P.g[1], P.g[2])));
}
// Such a tetrahedron, id (unit * 6 + s; of an explicit set its number): whether 6V is 0 from its float32 positions, in
// float64 and box units, where the products of close positions are exact; c: the cell of its centroid.
__device__ __forceinline__ bool exactly_flat(const DepositParams &P, int64_t id, int (&c)[3])
{
    float x[4][3];
    unsigned shifts = 0;
    if (P.src == SRC_TETS) {
        for (int i = 0; i < 12; ++i) x[i / 3][i % 3] = __ldg(P.verts + 12 * id + i);
    } else {
        int64_t ci, cj, ck;
        if (!cube_of_unit(P, id / 6, ci, cj, ck)) return false;
        lattice_positions(P, ci, cj, ck, (int)(id % 6), x);
        shifts = tet_shift_bits(P, x);
    }
    P3<double> p[4];
    for (int q = 0; q < 4; ++q)
        p[q] = mk<double>((double)x[q][0] + (double)shift_of(shifts, q, 0) * P.box,
                          (double)x[q][1] + (double)shift_of(shifts, q, 1) * P.box,
                          (double)x[q][2] + (double)shift_of(shifts, q, 2) * P.box);
    c[0] = safe_floor(0.25 * (p[0].x + p[1].x + p[2].x + p[3].x) * P.scale_d[0]);
    c[1] = safe_floor(0.25 * (p[0].y + p[1].y + p[2].y + p[3].y) * P.scale_d[1]);
    c[2] = safe_floor(0.25 * (p[0].z + p[1].z + p[2].z + p[3].z) * P.scale_d[2]);
    return det6(p) == 0.0;
}
// If it is flat, m_t goes to that cell.  Returns 0 (not flat, nothing done), 1 (deposited) or 2 (outside an
// open grid).  Out of line for the hot kernels: few get here.  (The baselines lose 1% and 4% by the call.)
template <Acc A>
__device__ __noinline__ int deposit_flat(const DepositParams &P, int64_t id, double m_t)
{
    int c[3];
    if (!exactly_flat(P, id, c)) return 0;
    return deposit_cell<A>(P, c[0], c[1], c[2], m_t) ? 1 : 2;
}

__device__ __forceinline__ int size_bin(int64_t cells)
{
    int b = 0;
    int64_t edge = 1;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        b += (cells > edge) ? 1 : 0;
        edge *= 8;
    }
    return b;
}

// Mass sums for the FP32 renormalisation, always kept: the target sum of m_t and the sum
// of every computed deposit.  A persistent lane adds up to ~10^6 terms, so plain running
// sums would drift by up to n x 2^-53 (the same mass added repeatedly rounds the same way):
// equal lattice masses are counted as an integer (times m_t at the end) and deposits are
// summed with Kahan's compensation.
struct Counters {
    unsigned long long u[ST_NUM_U64];
    double mass_in, dropped;
    double tgt;            // explicit tetrahedra: sum of m_t
    unsigned ntgt;         // lattice tetrahedra (each P.m_tet)
    double dep, dep_c;     // Kahan sum of deposits and its compensation
    double dep_b;          // plain sum of the deposits since the last fold (a few dozen)
    __device__ void zero()
    {
#pragma unroll
        for (int i = 0; i < ST_NUM_U64; ++i) u[i] = 0;
        mass_in = 0.0;
        dropped = 0.0;
    }
    __device__ void zero_mass()
    {
        tgt = 0.0;
        ntgt = 0;
        dep = 0.0;
        dep_c = 0.0;
        dep_b = 0.0;
    }
    __device__ __forceinline__ void add_tgt(const DepositParams &P, double m_t)
    {
        if (P.src == SRC_TETS) tgt += m_t;
        else ++ntgt;
    }
    __device__ __forceinline__ void add_dep(double m) { dep_b += m; }
    // fold the batch into the Kahan sum (after every round of pairs, every tetrahedron of
    // the thread kernels, and before the flush)
    __device__ __forceinline__ void fold_dep()
    {
        const double y = dep_b - dep_c;
        const double t = dep + y;
        dep_c = (t - dep) - y;
        dep = t;
        dep_b = 0.0;
    }
    // *sum += x, and the addition's rounding error (two-sum) to *lo: thousands of warps add
    // similar values, whose roundings would drift together
    static __device__ __forceinline__ void add_exact(double *sum, double *lo, double x)
    {
        const double old = atomicAdd(sum, x), s = old + x, xx = s - old;
        atomicAdd(lo, (old - (s - xx)) + (x - xx));
    }
    __device__ void flush_mass(const DepositParams &P, Workspace *ws)
    {
        fold_dep();
        double a = fma((double)ntgt, P.m_tet, tgt), b = dep - dep_c;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(kFull, a, o);
            b += __shfl_down_sync(kFull, b, o);
        }
        if ((threadIdx.x & 31) == 0 && (a != 0.0 || b != 0.0)) {
            add_exact(&ws->mass_target, &ws->mass_target_lo, a);
            add_exact(&ws->mass_deposited, &ws->mass_deposited_lo, b);
        }
    }
    __device__ void flush(Workspace *ws)
    {
        // warp-aggregate, then one atomic per warp and counter
#pragma unroll
        for (int i = 0; i < ST_NUM_U64; ++i) {
            unsigned long long x = u[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
            if ((threadIdx.x & 31) == 0 && x) atomicAdd(&ws->stats[i], x);
        }
        double a = mass_in, b = dropped;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(kFull, a, o);
            b += __shfl_down_sync(kFull, b, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&ws->mass_in, a);
            if (b != 0.0) atomicAdd(&ws->mass_dropped, b);
        }
    }
};

__device__ __forceinline__ void set_error(Workspace *ws, int code, int detail)
{
    if (atomicCAS(&ws->error_code, 0, code) == 0) ws->error_detail = detail;
}

struct WarpSmem {
    float v[12][32];      // base-frame vertices (x0 y0 z0 x1 ...), positively oriented
    float n[12][32];      // outward face normals
    float e[4][32];
    float pos[4][32];
    float neg[4][32];
    float lx[32], ly[32];  // reference-plane slopes (in the clip's frame)
    int axis[32];          // bits 0-1: the clip's divergence axis (to_axis); kRecCut; kRecGuard
    int lo[3][32];
    int dim[3][32];
    int base[3][32];      // uniform grid: the base cell; octree: the leaf's first cell, base-cell frame
    int leaf[32];         // octree: leaf of this (tetrahedron, leaf) pair
    float rho[32];        // 6 m_t / |6V| (deposit = rho * overlap volume, formed in float32)
    int start[32];        // exclusive prefix of the pair counts
    float *vres;          // warp-per-tetrahedron baseline: this warp's residual block in global
                          // memory: [12][32] floats, the rounding residuals of guarded records
                          // (exact vertex = v + vres)
    union {
        struct {
            unsigned long long q[64];   // baseline: queued partial pairs: t | ix << 5 | iy << 24 | iz << 43
            unsigned long long gq[64];  // baseline: queued partial pairs of guarded tetrahedra (float64 clips)
        };
        struct {
            float4 ra[64];  // queued runs (a ring): first cell along A, B, C; run word (see kRun*)
            float4 rb[64];  // the run's clip frame: qx, qy, qz, l0
        };
    };
    unsigned char fan[32];     // level fans of one round: the lane that holds the face, first level << 5
    union {
        float2 poly[21][32];   // baseline: each lane's 7 edge slots, 3 float2 each
        struct {
            float4 eh[7][32];  // column clip: each lane's 7 edge slots (EdgeSlots4)
            float2 el[7][32];
        };
        float comb[6][32];     // face terms of one round, after its fans
    };
};
constexpr int kRecCut = 4;    // octree: the record's cell range starts above the tetrahedron's own
                              // first layer along its divergence axis (a leaf block cuts it)
constexpr int kRecGuard = 8;  // a guarded tetrahedron (clipped in float64)

// What the guarded pass keeps per warp in place of the float slots and beyond them.
struct GuardSmem {
    double2 slots[21][32];  // each lane's 7 edge slots, 3 double2 each
    double v[12][32];       // exact vertices, positively oriented
    double tol[32];         // classification tolerance of the clip (f64_tolerance)
    double rho[32];         // the plain float64 path: 6 m_t / |6V|
};

constexpr int kQBits = 19;  // per-axis cell offset bits in a queue entry
constexpr unsigned long long kQMask = (1ull << kQBits) - 1;

__device__ __forceinline__ unsigned long long q_pack(int t, int ix, int iy, int iz)
{
    return (unsigned long long)t | ((unsigned long long)ix << 5) | ((unsigned long long)iy << (5 + kQBits)) |
           ((unsigned long long)iz << (5 + 2 * kQBits));
}

__device__ __forceinline__ void decompose(int local, int dx, int dy, int &ix, int &iy, int &iz)
{
    const int dxy = dx * dy;
    iz = local / dxy;
    const int r = local - iz * dxy;
    iy = r / dx;
    ix = r - iy * dx;
}

// The float64 clip of guarded record t against cell (cx, cy, cz) in the cell-by-cell
// schedule (the warp-per-tetrahedron baseline), kept out of line so that the FP32 hot loop
// stays small; it rebuilds the exact vertices from the float32 vertices and their residuals.
__device__ __noinline__ double redo_fp64(const WarpSmem *S, int t, int cx, int cy, int cz)
{
    P3<float> v[4], r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v[q] = mk<float>(S->v[3 * q][t], S->v[3 * q + 1][t], S->v[3 * q + 2][t]);
        r[q] = mk<float>(S->vres[(3 * q) * 32 + t], S->vres[(3 * q + 1) * 32 + t], S->vres[(3 * q + 2) * 32 + t]);
    }
    P3<double> pd[4];
    exact_vertices(v, r, cx, cy, cz, pd);
    return overlap_volume_fp64(pd);
}

// Record a guarded tetrahedron's residuals for redo_fp64.
__device__ __forceinline__ void store_residuals(WarpSmem *S, int lane, const P3<float> (&r)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        S->vres[(3 * q) * 32 + lane] = r[q].x;
        S->vres[(3 * q + 1) * 32 + lane] = r[q].y;
        S->vres[(3 * q + 2) * 32 + lane] = r[q].z;
    }
}

// Which records a kernel holds, and so which clips it carries:
//  * kPassAll: records on both sides of the guard, enumerated by cells; FP32 clips and FP64
//    clips in the same kernel (the warp-per-tetrahedron baseline);
//  * kPassFp32: records below the guard only, enumerated by column runs (FP32 column clips);
//  * kPassGuard: guarded records only, enumerated by column runs (FP64 column clips from
//    the exact vertices).
// The warp-cooperative and octree schedules run kPassFp32 and then kPassGuard over the same
// tetrahedra, so neither kernel carries the other's clip code or registers.
enum { kPassAll = 0, kPassFp32 = 1, kPassGuard = 2 };
// the scalar of a pass's column clips
template <int PASS>
struct PassScalar {
    using type = float;
};
template <>
struct PassScalar<kPassGuard> {
    using type = double;
};

__device__ __forceinline__ GuardSmem *guard_smem(WarpSmem *S)
{
    return reinterpret_cast<GuardSmem *>(reinterpret_cast<unsigned char *>(S) + offsetof(WarpSmem, poly));
}

// Record lane's tetrahedron for the pair machinery: cells [lo, lo + dim) of the base-cell frame;
// base: what deposit_pair adds to (uniform) or takes off (octree) a cell of that frame.  In the
// guarded pass the exact vertices are kept too, oriented by their own determinant, and the
// float32 vertices take the same order.
template <int PASS>
__device__ __forceinline__ void store_record(WarpSmem *S, int lane, const TetSetup<float> &ts,
                                             const P3<float> (&res)[4], const int (&lo)[3], const int (&dim)[3],
                                             const int (&base)[3], double m_t, float kappa_max, bool cut)
{
    const bool guard = PASS == kPassGuard || (PASS == kPassAll && !(ts.kappa <= kappa_max));
    bool flip = false;
    S->rho[lane] = guard ? (float)(6.0 * m_t / exact_vol6(ts.v, res, ts.vol6, &flip))
                         : __fdiv_rn((float)(6.0 * m_t), (float)ts.vol6);
    const bool turn = PASS == kPassGuard && flip;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int k = (q == 1 && turn) ? 2 : ((q == 2 && turn) ? 1 : q);
        S->v[3 * k][lane] = ts.v[q].x;
        S->v[3 * k + 1][lane] = ts.v[q].y;
        S->v[3 * k + 2][lane] = ts.v[q].z;
        S->n[3 * q][lane] = ts.n[q].x;
        S->n[3 * q + 1][lane] = ts.n[q].y;
        S->n[3 * q + 2][lane] = ts.n[q].z;
        S->e[q][lane] = ts.e[q];
        S->pos[q][lane] = ts.pos[q];
        S->neg[q][lane] = ts.neg[q];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        S->lo[a][lane] = lo[a];
        S->dim[a][lane] = dim[a];
        S->base[a][lane] = base[a];
    }
    S->lx[lane] = ts.lx;
    S->ly[lane] = ts.ly;
    S->axis[lane] = ts.axis | (cut ? kRecCut : 0) | (guard ? kRecGuard : 0);
    if constexpr (PASS == kPassGuard) {
        GuardSmem *G = guard_smem(S);
        P3<double> pd[4];
        exact_vertices(ts.v, res, 0, 0, 0, pd);
        G->tol[lane] = f64_tolerance((double)(ts.dim[0] + ts.dim[1] + ts.dim[2]));
        if (turn) {
            const P3<double> t = pd[1];
            pd[1] = pd[2];
            pd[2] = t;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            G->v[3 * q][lane] = pd[q].x;
            G->v[3 * q + 1][lane] = pd[q].y;
            G->v[3 * q + 2][lane] = pd[q].z;
        }
    }
    if constexpr (PASS == kPassAll) {
        if (guard) store_residuals(S, lane, res);
    }
}

// ---------------------------------------------------------------------------
// Column runs.  A tetrahedron below the FP32 guard is enumerated by runs of up to kRun
// cells along its divergence axis C (to_axis: A = C + 1, B = C + 2 mod 3): pair index
// ia + dA (ib + dB w) is the run of cells (A, B) = (lo_A + ia, lo_B + ib) and C in
// [lo_C + kRun w, lo_C + kRun w + kw).  One column clip (column_volumes) serves the run.
// ---------------------------------------------------------------------------
constexpr int kRun = 2;  // longer runs lose accuracy: the level terms grow with the run's height

__device__ __forceinline__ int axis_a(int C) { return C == 2 ? 0 : C + 1; }
__device__ __forceinline__ int axis_b(int C) { return C == 0 ? 2 : C - 1; }

// pairs of an unguarded record: its runs
__device__ __forceinline__ int64_t run_count(const int (&dim)[3], int C)
{
    const int dC = C == 0 ? dim[0] : (C == 1 ? dim[1] : dim[2]);
    const int dA = C == 2 ? dim[0] : (C == 0 ? dim[1] : dim[2]);
    const int dB = C == 0 ? dim[2] : (C == 1 ? dim[0] : dim[1]);
    return (int64_t)dA * dB * ((dC + kRun - 1) / kRun);
}

// A record's cell offsets must fit the kQBits-bit fields of a queue entry.
__device__ __forceinline__ bool dims_fit_queue(const int (&dim)[3])
{
    return dim[0] < (1 << 19) && dim[1] < (1 << 19) && dim[2] < (1 << 19);
}

// Record t as the column clip reads it: vertices relative to the run's first cell and relabelled
// so that axis C is z (to_axis), face normals likewise.  The relabelling is bound as three row
// pointers, (C+1)%3, (C+2)%3 and C, into the record arrays (vertex or face i is 3 rows = 96
// scalars further on; the normals follow the vertices at 12 rows = 384 scalars), so a fetch is
// three loads at fixed offsets and no selects.  T = float reads the float32 record; T = double
// the guarded pass's exact vertices (no normals: the float64 clip needs none).
template <class T>
struct RecordRun {
    const T *va, *vb, *vc;  // row pointers
    T fa, fb, fc;           // the run's first cell along the same three axes
    __device__ __forceinline__ P3<T> vtx(int i) const
    {
        return mk<T>(va[96 * i] - fa, vb[96 * i] - fb, vc[96 * i] - fc);
    }
    __device__ __forceinline__ P3<T> nrm(int f) const
    {
        return mk<T>(va[384 + 96 * f], vb[384 + 96 * f], vc[384 + 96 * f]);
    }
};
static_assert(offsetof(WarpSmem, n) == offsetof(WarpSmem, v) + 384 * sizeof(float), "RecordRun reads n after v");

template <class T>
__device__ __forceinline__ RecordRun<T> record_run(WarpSmem *S, int t, int C, T la, T lb, T lc)
{
    const T *rows;
    if constexpr (sizeof(T) == sizeof(float)) rows = &S->v[0][t];
    else rows = &guard_smem(S)->v[0][t];
    return RecordRun<T>{rows + 32 * axis_a(C), rows + 32 * axis_b(C), rows + 32 * C, la, lb, lc};
}

// Lane `lane`'s edge slots of the column clip.
__device__ __forceinline__ EdgeSlots4 lane_slots(WarpSmem *S, int lane, float) { return {&S->eh[0][lane], &S->el[0][lane]}; }
__device__ __forceinline__ EdgeSlots<double> lane_slots(WarpSmem *S, int lane, double)
{
    return {&guard_smem(S)->slots[0][lane]};
}

// Classify the box of kw cells from cell (cx, cy, cz) along axis C against record t's
// face planes (classify_cell for kw = 1).
__device__ __forceinline__ int classify_run(const WarpSmem *S, int t, int C, float cx, float cy, float cz, int kw)
{
    bool inside = true, outside = false;
    const float ext = (float)(kw - 1);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const float nx = S->n[3 * f][t], ny = S->n[3 * f + 1][t], nz = S->n[3 * f + 2][t];
        const float nc = C == 0 ? nx : (C == 1 ? ny : nz);
        const float s = fmaf(nx, cx, fmaf(ny, cy, fmaf(nz, cz, -S->e[f][t])));
        inside = inside && (s + fmaf(ext, fmaxf(nc, 0.f), S->pos[f][t]) <= 0.f);
        outside = outside || (s + fmaf(ext, fminf(nc, 0.f), S->neg[f][t]) >= 0.f);
    }
    return outside ? CELL_OUTSIDE : (inside ? CELL_INSIDE : CELL_PARTIAL);
}

// Add m to cell (cx, cy, cz) (base-cell frame) of virtual tetrahedron t: the uniform
// grid (folded / dropped as deposit_cell does) or t's octree leaf block.
template <bool OCT, Acc A>
__device__ __forceinline__ bool deposit_pair(const DepositParams &P, const WarpSmem *S, int t, int cx, int cy, int cz,
                                             double m)
{
    if constexpr (OCT) {
        // bc <= 4096: a cell's place in its leaf block needs up to 36 bits
        const int bc = P.bc;
        const int lx = cx - S->base[0][t], ly = cy - S->base[1][t], lz = cz - S->base[2][t];
        cell_add<A>(P, P.out + ((int64_t)(S->leaf[t] * (int64_t)bc + lz) * (bc * bc) + (lx + bc * ly)), m);
        return true;
    } else {
        return deposit_cell<A>(P, S->base[0][t] + cx, S->base[1][t] + cy, S->base[2][t] + cz, m);
    }
}

// Decode queue entry `ent` of record t: the cell (base-cell frame).
__device__ __forceinline__ void q_cell(const WarpSmem *S, unsigned long long ent, int &t, int &cx, int &cy, int &cz)
{
    t = (int)(ent & 31u);
    cx = S->lo[0][t] + (int)((ent >> 5) & kQMask);
    cy = S->lo[1][t] + (int)((ent >> (5 + kQBits)) & kQMask);
    cz = S->lo[2][t] + (int)((ent >> (5 + 2 * kQBits)) & kQMask);
}

template <bool STATS, bool OCT, Acc A>
__device__ __forceinline__ void deposit_clip(const DepositParams &P, const WarpSmem *S, int t, int cx, int cy, int cz,
                                             double vol, Counters &cnt)
{
    if (STATS) cnt.u[ST_PARTIAL_CLIPS]++;
    if (vol > 0.0) {
        if (STATS) cnt.u[ST_OVERLAPPED]++;
        const double m = (double)(S->rho[t] * (float)vol);
        cnt.add_dep(m);
        if (!deposit_pair<OCT, A>(P, S, t, cx, cy, cz, m) && STATS) cnt.dropped += m;
    }
}

// FP32 clips of the first `count` entries of S->q (tetrahedra below the guard).
template <bool STATS, bool OCT, Acc A>
__device__ __forceinline__ void clip_round(const DepositParams &P, WarpSmem *S, int count, int lane, Counters &cnt)
{
    if (lane < count) {
        int t, cx, cy, cz;
        q_cell(S, S->q[lane], t, cx, cy, cz);
        const float fx = (float)cx, fy = (float)cy, fz = (float)cz;
        P3<float> p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            p[q] = mk<float>(S->v[3 * q][t] - fx, S->v[3 * q + 1][t] - fy, S->v[3 * q + 2][t] - fz);
        P3<float> n[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) n[f] = mk<float>(S->n[3 * f][t], S->n[3 * f + 1][t], S->n[3 * f + 2][t]);
        P3<float> pa[4], na[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            pa[q] = to_axis(p[q], S->axis[t] & 3);
            na[q] = to_axis(n[q], S->axis[t] & 3);
        }
        float err;
        const double vol = (double)overlap_volume_rolled(pa, na, S->lx[t], S->ly[t], err, &S->poly[0][lane]);
        deposit_clip<STATS, OCT, A>(P, S, t, cx, cy, cz, vol, cnt);
    }
    __syncwarp();
}

// The face terms of a pass's clips, and a float32 value as its scalar.
template <class T>
struct FaceOf {
    using type = FaceRun<kRun, float>;
};
template <>
struct FaceOf<double> {
    using type = FaceRun64<kRun>;
};
template <class T>
__device__ __forceinline__ T widen(float x)
{
    if constexpr (sizeof(T) == sizeof(float)) return x;
    else return f64_widen(x);
}

// The run word (ra.w): record t (bits 0-4), faces to clip (bits 5-8), cells kw (9-10), axis C
// (11-12), lo_open (13).
constexpr int kRunMask = 5, kRunLen = 9, kRunAxis = 11, kRunOpen = 13;
constexpr int kRunsPerRound = 16;

// One clip round: the faces of up to 16 queued runs (32 faces at most), one face per lane.
//
// The clip is bound by instruction issue, so lanes must not idle: a run needs 2.8 of its 4
// faces on average, and a face straddles 0.5 levels on average but 2 or 3 somewhere in a warp.
// One run per lane therefore paid 4 faces and 8 level fans for everybody (19 of 32 lanes
// active); here faces are dealt to lanes, then the fans of their straddled levels are dealt
// again, and the cells of the runs (2 lanes a run) sum their faces' terms in face order, as one
// thread would, so the sums are the same bit for bit.  128^3 onto 256^3 takes 45.2 ms with one run a
// lane and 33.8 this way.
template <bool STATS, bool OCT, Acc A, class T, bool F64RHO>
__device__ __forceinline__ void job_round(const DepositParams &P, WarpSmem *S, int lane, int &head, int &qn, int &jobs,
                                          Counters &cnt)
{
    const unsigned le_mask = kFull >> (31 - lane);
    // ---- runs: as many from the head as have at most 32 faces together
    unsigned word = 0;
    if (lane < kRunsPerRound && lane < qn) word = __float_as_uint(S->ra[(head + lane) & 63].w);
    const int nface = __popc((word >> kRunMask) & 15u);
    int incl = nface;
#pragma unroll
    for (int o = 1; o < kRunsPerRound; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int first = incl - nface;  // this run's first job
    const bool fits = lane < kRunsPerRound && lane < qn && incl <= 32;
    const int R = __popc(__ballot_sync(kFull, fits));
    const int J = __shfl_sync(kFull, incl, R - 1);
    const unsigned starts = __reduce_or_sync(kFull, fits ? 1u << first : 0u);

    // ---- one face per lane
    typename FaceOf<T>::type fr;
    face_none(fr);
    T qz = T(0);
    {
        const int r = __popc(starts & le_mask) - 1;
        const unsigned w = __shfl_sync(kFull, word, r);
        int k = lane - __shfl_sync(kFull, first, r);
        if (lane < J) {
            unsigned m = (w >> kRunMask) & 15u;
#pragma unroll
            for (int i = 0; i < 3; ++i) m = (i < k) ? (m & (m - 1u)) : m;
            const int f = __ffs((int)m) - 1;
            const int slot = (head + r) & 63;
            const float4 ra = S->ra[slot], rb = S->rb[slot];
            const int t = (int)(w & 31u), C = (int)((w >> kRunAxis) & 3u);
            RunFrame<T> F;
            F.qx = widen<T>(rb.x);
            F.qy = widen<T>(rb.y);
            F.qz = widen<T>(rb.z);
            F.l0 = widen<T>(rb.w);
            F.lx = widen<T>(S->lx[t]);
            F.ly = widen<T>(S->ly[t]);
            F.K = (int)((w >> kRunLen) & 3u);
            F.j0 = ((w >> kRunOpen) & 1u) ? 0 : 1;
            qz = F.qz;
            int ia, ib, ic;
            face_vertices(f, ia, ib, ic);
            if constexpr (sizeof(T) == sizeof(float)) {
                const RecordRun<float> src = record_run<float>(S, t, C, ra.x, ra.y, ra.z);
                const P3<float> q = mk<float>(F.qx, F.qy, F.qz);
                const P3<float> a = sub(src.vtx(ia), q), b = sub(src.vtx(ib), q), c = sub(src.vtx(ic), q);
                const P3<float> nf = src.nrm(f);
                if (face_meets_column<float>(a, b, c, nf.z, F))
                    face_run<kRun, float, OCT>(a, b, c, nf, F, lane_slots(S, lane, 0.f), fr);
            } else {
                // straight into the frame: first cell + q is exact
                const RecordRun<double> src = record_run<double>(S, t, C, widen<double>(ra.x) + F.qx,
                                                                 widen<double>(ra.y) + F.qy, widen<double>(ra.z) + F.qz);
                face_run_f64<kRun>(src.vtx(ia), src.vtx(ib), src.vtx(ic), F, guard_smem(S)->tol[t],
                                   lane_slots(S, lane, 0.0), fr);
            }
        }
    }
    __syncwarp();

    // ---- level fans, one per lane: whole faces in order, 32 fans at most per pass
    int pend = fr.jhi >= fr.jlo ? fr.jhi - fr.jlo + 1 : 0;
#pragma unroll 1
    while (__any_sync(kFull, pend > 0)) {
        int inc = pend;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        const bool take = pend > 0 && inc <= 32;
        const int at = inc - pend;
        if (take) S->fan[at] = (unsigned char)(lane | (fr.jlo << 5));
        const unsigned heads = __reduce_or_sync(kFull, take ? 1u << at : 0u);
        const int nfan = (int)__reduce_max_sync(kFull, take ? (unsigned)inc : 0u);
        __syncwarp();
        int from = lane, j = 0;
        if (lane < nfan) {
            const int p = 31 - __clz((int)(heads & le_mask));
            const int e = S->fan[p];
            from = e & 31;
            j = (e >> 5) + lane - p;
        }
        const T fq = __shfl_sync(kFull, qz, from);
        const int ne = __shfl_sync(kFull, fr.n, from);
        T g = T(0);
        if constexpr (sizeof(T) == sizeof(float)) {
            const float nx = __shfl_sync(kFull, fr.nx, from), ny = __shfl_sync(kFull, fr.ny, from),
                        nz = __shfl_sync(kFull, fr.nz, from), ef = __shfl_sync(kFull, fr.ef, from);
            if (lane < nfan) {
                const float cj = (float)j - fq;
                g = level_fan<OCT, float>(lane_slots(S, from, 0.f), ne, cj, fan_anchor<float>(nx, ny, nz, ef, cj), nx, ny);
            }
        } else {
            if (lane < nfan) g = level_fan_f64(lane_slots(S, from, 0.0), ne, widen<double>((float)j) - fq);
        }
#pragma unroll
        for (int i = 0; i <= kRun; ++i) {
            const T x = __shfl_sync(kFull, g, (at + i - fr.jlo) & 31);
            if (take && i >= fr.jlo && i <= fr.jhi) fr.k6[i] -= x;
        }
        if (take) pend = 0;
        __syncwarp();
    }

    // ---- the runs' cells, two lanes a run
    T(*comb)[32];
    if constexpr (sizeof(T) == sizeof(float)) comb = S->comb;
    else comb = reinterpret_cast<double(*)[32]>(&guard_smem(S)->slots[0][0]);
    if (lane < J) {
#pragma unroll
        for (int i = 0; i <= kRun; ++i) comb[i][lane] = fr.k6[i];
        if constexpr (sizeof(T) == sizeof(float)) {
            comb[3][lane] = fr.zmin;
            comb[4][lane] = fr.zmax;
        } else {
            comb[3][lane] = __longlong_as_double(fr.kmin);
            comb[4][lane] = __longlong_as_double(fr.kmax);
        }
        comb[5][lane] = fr.m6;
    }
    __syncwarp();
    {
        static_assert(kRun == 2, "two lanes a run");
        const int r = lane >> 1, j = lane & 1;
        const unsigned w = __shfl_sync(kFull, word, r);
        const int j0 = __shfl_sync(kFull, first, r);
        const int kw = (int)((w >> kRunLen) & 3u);
        if (r < R && j < kw) {
            const int nf = __popc((w >> kRunMask) & 15u);
            T s0 = T(0), s1 = T(0), msum = T(0);
            float colmin = 1e30f, colmax = -1e30f;
            long long kmin = kKeyMax, kmax = kKeyMin;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < nf) {
                    s0 += comb[j][j0 + i];
                    s1 += comb[j + 1][j0 + i];
                    msum += comb[5][j0 + i];
                    if constexpr (sizeof(T) == sizeof(float)) {
                        colmin = fminf(colmin, comb[3][j0 + i]);
                        colmax = fmaxf(colmax, comb[4][j0 + i]);
                    } else {
                        const long long kl = __double_as_longlong(comb[3][j0 + i]), kh = __double_as_longlong(comb[4][j0 + i]);
                        kmin = kl < kmin ? kl : kmin;
                        kmax = kh > kmax ? kh : kmax;
                    }
                }
            }
            const int slot = (head + r) & 63;
            const float4 ra = S->ra[slot];
            const float fq = S->rb[slot].z;
            const float c0 = (float)j - fq, c1 = (float)(j + 1) - fq;  // exact: multiples of 1/256
            T vol;
            if constexpr (sizeof(T) == sizeof(float)) vol = level_volume<float>(c0, c1, s0, s1, colmin, colmax, msum);
            else vol = level_volume_f64(widen<double>(c0), widen<double>(c1), s0, s1, kmin, kmax, msum);
            const int t = (int)(w & 31u), C = (int)((w >> kRunAxis) & 3u);
            const int la = (int)ra.x, lb = (int)ra.y, lc = (int)ra.z + j;
            const int ex = C == 0 ? lc : (C == 1 ? lb : la), ey = C == 1 ? lc : (C == 2 ? lb : la),
                      ez = C == 2 ? lc : (C == 0 ? lb : la);
            if (STATS) {
                // the same per-cell classification as the cell schedules, for the counters
                if (j == 0) cnt.u[ST_RUNS]++;
                P3<float> n[4];
                float e[4], ps[4], ng[4];
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    n[f] = mk<float>(S->n[3 * f][t], S->n[3 * f + 1][t], S->n[3 * f + 2][t]);
                    e[f] = S->e[f][t];
                    ps[f] = S->pos[f][t];
                    ng[f] = S->neg[f][t];
                }
                const int cls = classify_cell<float>(n, e, ps, ng, (float)ex, (float)ey, (float)ez);
                if (cls == CELL_PARTIAL) {
                    cnt.u[ST_PARTIAL_CLIPS]++;
                    if (sizeof(T) != sizeof(float)) cnt.u[ST_FP64_REDOS]++;
                } else if (cls == CELL_INSIDE) {
                    cnt.u[ST_INSIDE_CELLS]++;
                }
            }
            if (vol > T(0)) {
                if (STATS) cnt.u[ST_OVERLAPPED]++;
                double m;
                if constexpr (sizeof(T) == sizeof(float)) m = (double)(S->rho[t] * (float)vol);
                else if constexpr (F64RHO) m = guard_smem(S)->rho[t] * vol;
                else m = (double)S->rho[t] * vol;
                cnt.add_dep(m);
                if (!deposit_pair<OCT, A>(P, S, t, ex, ey, ez, m) && STATS) cnt.dropped += m;
            }
        }
    }
    head = (head + R) & 63;
    qn -= R;
    jobs -= J;
    __syncwarp();
}

// Float64 clips (exact vertices) of the first `count` entries of S->gq.  Guarded pairs
// are queued apart so that these rounds run with full warps.
template <bool STATS, bool OCT, Acc A>
__device__ __forceinline__ void redo_round(const DepositParams &P, WarpSmem *S, int count, int lane, Counters &cnt)
{
    if (lane < count) {
        int t, cx, cy, cz;
        q_cell(S, S->gq[lane], t, cx, cy, cz);
        const double vol = redo_fp64(S, t, cx, cy, cz);
        if (STATS) cnt.u[ST_FP64_REDOS]++;
        deposit_clip<STATS, OCT, A>(P, S, t, cx, cy, cz, vol, cnt);
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// The guarded-tetrahedron list.  The FP32 pass already sets up every tetrahedron; it lists
// the guarded multi-cell ones so that the guarded pass visits only those instead of
// generating and setting up every tetrahedron again (on a lattice with few guarded
// tetrahedra that second scan was most of the guarded pass).
// ---------------------------------------------------------------------------
// Append the id of this lane's guarded tetrahedron (want) with one atomic per warp.  Ids past
// the capacity are not stored, but the count still grows, which sends the guarded pass back
// to a full scan.  Called by all 32 lanes.
__device__ __forceinline__ void list_guarded(const DepositParams &P, bool want, int64_t id, int lane)
{
    const unsigned m = __ballot_sync(kFull, want);
    if (m == 0u || P.guard_cap == 0) return;
    unsigned long long first = 0;
    if (lane == 0) first = atomicAdd(&P.ws->guard_count, (unsigned long long)__popc(m));
    first = __shfl_sync(kFull, first, 0);
    if (want) {
        const unsigned long long k = first + (unsigned long long)__popc(m & ((1u << lane) - 1u));
        if (k < (unsigned long long)P.guard_cap) P.guard_list[k] = id;
    }
}

// The guarded pass: the number of listed tetrahedra when the FP32 pass listed all of them,
// else -1 (scan every tetrahedron).
__device__ __forceinline__ int64_t listed_guarded(const DepositParams &P)
{
    if (P.guard_cap == 0) return -1;
    const unsigned long long c = *reinterpret_cast<const volatile unsigned long long *>(&P.ws->guard_count);
    return c > (unsigned long long)P.guard_cap ? -1 : (int64_t)c;
}

// 6 m_t / |6V| of record t: float32, or float64 in the plain float64 path (F64RHO).
template <bool F64RHO>
__device__ __forceinline__ auto record_rho(WarpSmem *S, int t)
{
    if constexpr (F64RHO) return guard_smem(S)->rho[t];
    else return S->rho[t];
}

// Inclusive prefix of the lanes' pair counts into S->start (exclusive) and their total.
__device__ __forceinline__ int pair_prefix(WarpSmem *S, int lane, int npairs)
{
    int incl = npairs;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    S->start[lane] = incl - npairs;
    __syncwarp();
    return __shfl_sync(kFull, incl, 31);
}

// The record that holds pair idx.
__device__ __forceinline__ int pair_record(const WarpSmem *S, int idx)
{
    int t = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1)
        if (S->start[t + step] <= idx && t + step < 32) t += step;
    return t;
}

// Enumerate every (virtual tetrahedron, run) pair of the 32 records in S (npairs: this lane's
// run count; skip: the first run of the records, for pieces of a split tetrahedron), 32 per
// step: classify; deposit the cells of "inside" runs; queue the partial runs with their clip
// frame and the faces that reach their column, and clip 32 faces at a time.
template <bool STATS, bool OCT, Acc A, class T, bool F64RHO = false>
__device__ __forceinline__ void coop_runs(const DepositParams &P, WarpSmem *S, int lane, int npairs, int skip,
                                          Counters &cnt)
{
    const unsigned lt_mask = (1u << lane) - 1u;
    const int total = pair_prefix(S, lane, npairs);
    int head = 0, qn = 0, jobs = 0;  // the ring of queued runs; the faces they hold
#pragma unroll 1
    for (int b0 = 0; b0 < total; b0 += 32) {
        const int idx = b0 + lane;
        unsigned word = 0;
        float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra;
        if (idx < total) {
            const int t = pair_record(S, idx);
            int local = idx - S->start[t] + skip;
            const int rec = S->axis[t];
            const int C = rec & 3, iA = axis_a(C), iB = axis_b(C);
            // run number `local`: ia fastest, then ib, then w
            const int dA = S->dim[iA][t], dB = S->dim[iB][t];
            const int rest = local / dA, w = rest / dB;
            const int kw = min(kRun, S->dim[C][t] - w * kRun);
            const int la = S->lo[iA][t] + (local - rest * dA), lb = S->lo[iB][t] + (rest - w * dB),
                      lc = S->lo[C][t] + w * kRun;
            const int cx = C == 0 ? lc : (C == 1 ? lb : la), cy = C == 1 ? lc : (C == 2 ? lb : la),
                      cz = C == 2 ? lc : (C == 0 ? lb : la);
            const int cls = classify_run(S, t, C, (float)cx, (float)cy, (float)cz, kw);
            if (cls == CELL_INSIDE) {
                const double m = (double)record_rho<F64RHO>(S, t);
                for (int j = 0; j < kw; ++j) {
                    cnt.add_dep(m);
                    if (!deposit_pair<OCT, A>(P, S, t, cx + (C == 0 ? j : 0), cy + (C == 1 ? j : 0),
                                              cz + (C == 2 ? j : 0), m) && STATS)
                        cnt.dropped += m;
                }
                if (STATS) { cnt.u[ST_INSIDE_CELLS] += kw; cnt.u[ST_OVERLAPPED] += kw; }
            } else if (cls == CELL_PARTIAL) {
                const RecordRun<float> near = record_run<float>(S, t, C, (float)la, (float)lb, (float)lc);
                P3<float> p[4];
                unsigned up = 0, flat = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) p[q] = near.vtx(q);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float nz;
                    if constexpr (sizeof(T) == sizeof(float)) {
                        nz = near.vc[384 + 96 * q];
                        flat |= nz == 0.f ? 1u << q : 0u;  // vertical: no projected area
                    } else {
                        // (the guarded pass may have turned the vertices over)
                        int ia, ib, ic;
                        face_vertices(q, ia, ib, ic);
                        nz = (p[ib].x - p[ia].x) * (p[ic].y - p[ia].y) - (p[ib].y - p[ia].y) * (p[ic].x - p[ia].x);
                    }
                    up |= nz > 0.f ? 1u << q : 0u;
                }
                unsigned mask = face_mask(p, up) & ~flat;
                if (STATS && mask == 0u) mask = 1u;  // counted as a run all the same
                if (mask != 0u) {
                    const bool lo_open = w > 0 || (rec & kRecCut) != 0;
                    word = (unsigned)t | (mask << kRunMask) | ((unsigned)kw << kRunLen) | ((unsigned)C << kRunAxis) |
                           (lo_open ? 1u << kRunOpen : 0u);
                    ra = make_float4((float)la, (float)lb, (float)lc, __uint_as_float(word));
                    // (the float64 clip takes the float32 frame too: any nearby origin and
                    // reference plane serve)
                    const RunFrame<float> F = run_frame<float>(near, S->lx[t], S->ly[t], kw, lo_open);
                    rb = make_float4(F.qx, F.qy, F.qz, F.l0);
                }
            }
        }
        const unsigned bal = __ballot_sync(kFull, word != 0u);
        if (word != 0u) {
            const int slot = (head + qn + __popc(bal & lt_mask)) & 63;
            S->ra[slot] = ra;
            S->rb[slot] = rb;
        }
        qn += __popc(bal);
        jobs += (int)__reduce_add_sync(kFull, (unsigned)__popc((word >> kRunMask) & 15u));
        __syncwarp();
        const bool last = b0 + 32 >= total;
#pragma unroll 1
        while (jobs >= 32 || (last && qn > 0)) job_round<STATS, OCT, A, T, F64RHO>(P, S, lane, head, qn, jobs, cnt);
    }
    cnt.fold_dep();
}

// Enumerate every (tetrahedron, cell) pair of the records in S, 32 pairs per round (the
// warp-per-tetrahedron baseline): classify; deposit "cell inside" pairs; queue partial pairs,
// those of guarded tetrahedra apart, and clip them 32 at a time.
template <bool STATS, Acc A>
__device__ __forceinline__ void coop_cells(const DepositParams &P, WarpSmem *S, int lane, int npairs, Counters &cnt)
{
    const unsigned lt_mask = (1u << lane) - 1u;
    const int total = pair_prefix(S, lane, npairs);
    // one clip_round call site, so that the clip is inlined once (instruction-cache footprint)
    int qn = 0, gn = 0;
    for (int b0 = 0;; b0 += 32) {
        if (b0 < total) {
            const int idx = b0 + lane;
            bool partial = false, gpartial = false;
            unsigned long long ent = 0;
            if (idx < total) {
                const int t = pair_record(S, idx);
                const int local = idx - S->start[t];
                int ix, iy, iz;
                decompose(local, S->dim[0][t], S->dim[1][t], ix, iy, iz);
                const float cx = (float)(S->lo[0][t] + ix), cy = (float)(S->lo[1][t] + iy),
                            cz = (float)(S->lo[2][t] + iz);
                P3<float> n[4];
                float e[4], ps[4], ng[4];
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    n[f] = mk<float>(S->n[3 * f][t], S->n[3 * f + 1][t], S->n[3 * f + 2][t]);
                    e[f] = S->e[f][t];
                    ps[f] = S->pos[f][t];
                    ng[f] = S->neg[f][t];
                }
                const int cls = classify_cell<float>(n, e, ps, ng, cx, cy, cz);
                if (cls == CELL_INSIDE) {
                    const double m = (double)S->rho[t];
                    cnt.add_dep(m);
                    if (!deposit_pair<false, A>(P, S, t, S->lo[0][t] + ix, S->lo[1][t] + iy, S->lo[2][t] + iz, m) &&
                        STATS)
                        cnt.dropped += m;
                    if (STATS) { cnt.u[ST_INSIDE_CELLS]++; cnt.u[ST_OVERLAPPED]++; }
                } else if (cls == CELL_PARTIAL) {
                    ent = q_pack(t, ix, iy, iz);
                    if (S->axis[t] & kRecGuard) gpartial = true;
                    else partial = true;
                }
            }
            const unsigned bal = __ballot_sync(kFull, partial);
            if (partial) S->q[qn + __popc(bal & lt_mask)] = ent;
            qn += __popc(bal);
            const unsigned gbal = __ballot_sync(kFull, gpartial);
            if (gpartial) S->gq[gn + __popc(gbal & lt_mask)] = ent;
            gn += __popc(gbal);
            __syncwarp();
        }
        const bool last = b0 + 32 >= total;
        if (qn >= 32 || (last && qn > 0)) {
            const int take = qn >= 32 ? 32 : qn;
            clip_round<STATS, false, A>(P, S, take, lane, cnt);
            if (lane < qn - take) S->q[lane] = S->q[take + lane];
            qn -= take;
            __syncwarp();
        }
        if (gn >= 32 || (last && gn > 0)) {
            const int take = gn >= 32 ? 32 : gn;
            redo_round<STATS, false, A>(P, S, take, lane, cnt);
            if (lane < gn - take) S->gq[lane] = S->gq[take + lane];
            gn -= take;
            __syncwarp();
        }
        if (last && qn == 0 && gn == 0) break;
    }
    cnt.fold_dep();
}

// Each warp's shared memory is a WarpSmem; in the guarded pass a GuardSmem takes the place of
// its float slots (the struct's last member, which that pass never touches) and runs past the
// struct's end: 23 KB a warp, two 4-warp blocks an SM.
constexpr size_t kGuardWarpBytes = offsetof(WarpSmem, poly) + sizeof(GuardSmem);
static_assert(offsetof(WarpSmem, poly) % 16 == 0 && kGuardWarpBytes % 16 == 0 && sizeof(WarpSmem) % 16 == 0,
              "warp blocks of shared memory must keep 16-byte alignment");
PSE_HD constexpr size_t warp_stride(bool guard_slots) { return guard_slots ? kGuardWarpBytes : sizeof(WarpSmem); }

// this warp's block of dynamic shared memory
__device__ __forceinline__ WarpSmem *warp_smem(bool guard_slots)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<WarpSmem *>(smem_raw + (threadIdx.x >> 5) * warp_stride(guard_slots));
}

// Point S->vres at this warp's residual block (every lane writes the same value).
__device__ __forceinline__ void bind_residuals(const DepositParams &P, WarpSmem *S)
{
    S->vres = P.vres + ((size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (12 * 32);
    __syncwarp();
}

// dynamic shared memory of a warp kernel with `warps` warps
inline size_t warp_smem_bytes(int warps, bool guard_slots) { return warp_stride(guard_slots) * warps; }

inline int persistent_blocks(const void *kernel, int threads, size_t smem)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

}  // namespace
}  // namespace pse
