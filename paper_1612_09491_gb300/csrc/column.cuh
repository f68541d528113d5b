// column.cuh -- the column clip of the warp kernels: the overlap volumes of a tetrahedron
// with a run of cells stacked along its divergence axis, from one x/y clip per face
// (geom.cuh holds the per-cell clips it builds on).  Templated on the scalar type: float
// for the FP32 pass, double for guarded tetrahedra (from their exact vertices).
#pragma once

#include <cstring>
#include <type_traits>

#include "geom.cuh"

namespace pse {

// ---------------------------------------------------------------------------
// Column clip: the overlap volumes of a tetrahedron with a run of up to KW cells stacked
// along the divergence axis (one column of the clip frame), from one x/y clip per face.
//
// With the same field as overlap_volume, the volume of T below a level z = c inside the
// column is
//
//   B(c) = Σ_f  ∫∫_{Q_f} (min(z_f(x,y), c) - l(x,y)) dx dy          (signed per face)
//
// where Q_f is face f's projection clipped to the column; the reference plane l cancels
// over the closed surface for every c, so each level may be evaluated with it.  The cells
// of the column are the slabs between consecutive integer levels, vol_j = B(c_{j+1}) -
// B(c_j), so the x and y slab passes of a face are shared by all cells of the run and
// every interior level serves the two cells beside it.  Per face and level c:
//   * face entirely above c:   ∫(c - l)           = (3c X - Y)/6 with face sums X, Y;
//   * face entirely below c:   ∫(z - l)           = M/6, the face's own moment;
//   * face crossing c:         M/6 - ∫(z - c)_+, the last term a fan of triangles from a
//     point o_c of the face plane on the line z = c, over the parts of the polygon's
//     edges above c.  The fan's triangles along the cut line are degenerate (o_c lies on
//     it), so the cut edge need not be formed, and the sum is continuous in the vertices.
// o_c is the foot of the perpendicular from the local origin onto that line in the xy
// plane; the line crosses the face inside the tetrahedron's bounding box, so o_c stays
// within a few cells of the origin.
// ---------------------------------------------------------------------------
// The edge list of one clipped face polygon: up to 7 directed edges a -> b.  A float slot is one
// float4 (a.xyz, b.x) and one float2 (b.yz) on the device, so that a lane reads it with two
// loads; any other scalar type (and the host) keeps three two-scalar rows per slot.  Slots of
// neighbouring lanes are adjacent (a stride of 32 lanes), so accesses have no bank conflicts.
template <class T>
struct EdgeSlots {
    slot2_t<T> *e;
    PSE_HD void store(int k, const P3<T> &a, const P3<T> &b) const { slot_store<T>(e, k, a, b); }
    PSE_HD void load(int k, P3<T> &a, P3<T> &b) const { slot_load<T>(e, k, a, b); }
};
#ifdef __CUDACC__
// the float slots of one lane of a warp: h points into a [7][32] float4 block, l into a
// [7][32] float2 block
struct EdgeSlots4 {
    float4 *h;
    float2 *l;
    __device__ __forceinline__ void store(int k, const P3<float> &a, const P3<float> &b) const
    {
        h[32 * k] = make_float4(a.x, a.y, a.z, b.x);
        l[32 * k] = make_float2(b.y, b.z);
    }
    __device__ __forceinline__ void load(int k, P3<float> &a, P3<float> &b) const
    {
        const float4 u = h[32 * k];
        const float2 v = l[32 * k];
        a = mk<float>(u.x, u.y, u.z);
        b = mk<float>(u.w, v.x, v.y);
    }
};
#endif

template <class T>
struct FaceSums {
    T m6;          // 6 ∫ (z - l) over the clipped face polygon (signed by orientation)
    T x2;          // Σ cross_xy(a, b) over its edges (twice the signed projected area)
    T y6;          // Σ cross_xy(a, b) (l(0) + l(a) + l(b)): 6 ∫ l = y6, 6 ∫ c = 3 c x2
    T zmin, zmax;  // z range of the polygon's vertices
};

// 1 / x for the slab passes: the device's approximate reciprocal, whose result is only used
// clamped to an edge.  A difference of 0 (or one too small for it: flushed) gives an infinity,
// and the products with it 0, 1 or, clamped, 0 for NaN: a point of the edge all the same.
PSE_HD float slab_rcp(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.f / x;
#endif
}
template <class T>
PSE_HD T slab_rcp(T x)
{
    return fdiv(T(1), x);
}

// The sums below are written with explicit fused multiply-adds and separately rounded products,
// so that every kernel forms them alike, however the compiler would fuse them: a fan triangle's
// term and the integral of l over it (see fan_mid).
template <class T>
PSE_HD T fan_height(const P3<T> &a, const P3<T> &b, T fo, T l0, T lx, T ly)
{
    const T fa = a.z - fmaT(lx, a.x, fmaT(ly, a.y, l0));
    const T fb = b.z - fmaT(lx, b.x, fmaT(ly, b.y, l0));
    return fo + fa + fb;
}
template <class T>
PSE_HD T plane_sum(const P3<T> &a, const P3<T> &b, T l0, T lx, T ly)
{
    return fmaT(T(3), l0, fmaT(lx, a.x + b.x, mul_rn(ly, a.y + b.y)));
}

// x slab pass of the column clip: the triangle (a, b, c) clipped against lo <= x < hi, its
// surviving edges stored in order (the triangle's, then the new ones on lo and on hi); returns
// their number (0 to 5).  An edge is cut at its own parameters for the two planes, each end by
// the plane it lies beyond; an edge beyond one plane at both ends is left out (it would add
// exactly 0 to every sum).  ROLL keeps this loop and the one over the new y edges rolled, for the
// octree kernel, whose set-up code competes for the instruction cache (256^3: 3% less time; the
// uniform kernel loses 1% by it).
template <bool ROLL, class T, class Slots>
PSE_HD int xslab_triangle(const P3<T> &a, const P3<T> &b, const P3<T> &c, T lo, T hi, T tol, const Slots &E)
{
    const T lt = lo - tol, ht = hi - tol;
    P3<T> u = a, v = b, w = c;  // the edge u -> v, then v -> w, then w -> u
    // exit and entry points on the two planes (a triangle crosses each at most once each way)
    T xly = T(0), xlz = T(0), nly = T(0), nlz = T(0), xhy = T(0), xhz = T(0), nhy = T(0), nhz = T(0);
    bool cl = false, ch = false;
    int n = 0;
#pragma unroll (ROLL ? 1 : 3)
    for (int i = 0; i < 3; ++i) {
        const bool u_lo = u.x < lt, u_hi = u.x >= ht, v_lo = v.x < lt, v_hi = v.x >= ht;
        const bool inu = !u_lo && !u_hi, inv = !v_lo && !v_hi;
        const T pu = u_lo ? lo : hi, pv = v_lo ? lo : hi;  // the plane an end outside is cut by
        const T r = slab_rcp(v.x - u.x);
        const T tu = sat01((pu - u.x) * r), tv = sat01((pv - u.x) * r);
        const T dy = v.y - u.y, dz = v.z - u.z;
        const P3<T> nu = mk<T>(inu ? u.x : pu, inu ? u.y : fmaT(tu, dy, u.y), inu ? u.z : fmaT(tu, dz, u.z));
        const P3<T> nv = mk<T>(inv ? v.x : pv, inv ? v.y : fmaT(tv, dy, u.y), inv ? v.z : fmaT(tv, dz, u.z));
        const bool oxl = !u_lo && v_lo, onl = u_lo && !v_lo, oxh = !u_hi && v_hi, onh = u_hi && !v_hi;
        xly = oxl ? nv.y : xly;
        xlz = oxl ? nv.z : xlz;
        nly = onl ? nu.y : nly;
        nlz = onl ? nu.z : nlz;
        xhy = oxh ? nv.y : xhy;
        xhz = oxh ? nv.z : xhz;
        nhy = onh ? nu.y : nhy;
        nhz = onh ? nu.z : nhz;
        cl = cl || oxl;
        ch = ch || oxh;
        if (!(u_lo && v_lo) && !(u_hi && v_hi)) {
            E.store(n, nu, nv);
            ++n;
        }
        const P3<T> t = u;
        u = v;
        v = w;
        w = t;
    }
    if (cl) {
        E.store(n, mk<T>(lo, xly, xlz), mk<T>(lo, nly, nlz));
        ++n;
    }
    if (ch) {
        E.store(n, mk<T>(hi, xhy, xhz), mk<T>(hi, nhy, nhz));
        ++n;
    }
    return n;
}

// y slab pass of the column clip on the n edges in E, and the face sums of the clipped polygon
// (its surviving edges and the two new ones on the y planes).  The surviving edges of nonzero
// length are stored back in order, the new ones after them; returns their number (0 to 7).
template <bool ROLL, class T, class Slots>
PSE_HD int yslab_sums(const Slots &E, int n, T lo, T hi, T tol, const P3<T> &o, T fo, T l0, T lx, T ly, FaceSums<T> &I)
{
    const T lt = lo - tol, ht = hi - tol;
    P3<T> xl = mk<T>(T(0), lo, T(0)), nl = xl, xh = mk<T>(T(0), hi, T(0)), nh = xh;
    bool cl = false, ch = false;  // the polygon crosses lo / hi
    T m6 = T(0), x2 = T(0), y6 = T(0);
    T zmn = T(1e30), zmx = T(-1e30);  // an empty polygon keeps this range
    int m = 0;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        P3<T> ea, eb;
        E.load(k, ea, eb);
        const bool a_lo = ea.y < lt, b_lo = eb.y < lt;
        const bool a_hi = ea.y >= ht, b_hi = eb.y >= ht;
        const T inv = slab_rcp(eb.y - ea.y);
        const T pa = a_lo ? lo : hi, pb = b_lo ? lo : hi;  // the plane an end outside is cut by
        const T ta = sat01((pa - ea.y) * inv), tb = sat01((pb - ea.y) * inv);
        const T dx = eb.x - ea.x, dz = eb.z - ea.z;
        const bool ina = !a_lo && !a_hi, inb = !b_lo && !b_hi;
        const P3<T> na = mk<T>(ina ? ea.x : fmaT(ta, dx, ea.x), ina ? ea.y : pa, ina ? ea.z : fmaT(ta, dz, ea.z));
        const P3<T> nb = mk<T>(inb ? eb.x : fmaT(tb, dx, ea.x), inb ? eb.y : pb, inb ? eb.z : fmaT(tb, dz, ea.z));
        const bool oxl = !a_lo && b_lo, onl = a_lo && !b_lo, oxh = !a_hi && b_hi, onh = a_hi && !b_hi;
        xl.x = oxl ? nb.x : xl.x;
        xl.z = oxl ? nb.z : xl.z;
        nl.x = onl ? na.x : nl.x;
        nl.z = onl ? na.z : nl.z;
        xh.x = oxh ? nb.x : xh.x;
        xh.z = oxh ? nb.z : xh.z;
        nh.x = onh ? na.x : nh.x;
        nh.z = onh ? na.z : nh.z;
        cl = cl || oxl;
        ch = ch || oxh;
        // a dropped edge has zero length: it adds nothing to the sums
        const T cr = cross_xy(na, nb);
        m6 = fmaT(cross_xy(sub(na, o), sub(nb, o)), fan_height(na, nb, fo, l0, lx, ly), m6);
        x2 += cr;
        y6 = fmaT(cr, plane_sum(na, nb, l0, lx, ly), y6);
        // z range over edges of nonzero length (dropped edges carry no vertex of the polygon)
        const bool live = na.x != nb.x || na.y != nb.y || na.z != nb.z;
        if (live) {
            zmn = fmin(zmn, fmin(na.z, nb.z));
            zmx = fmax(zmx, fmax(na.z, nb.z));
            E.store(m, na, nb);
            ++m;
        }
    }
    // the new edges join points that already bound surviving edges: they change no z range.  (Their
    // terms are added up first, the lower one's as a product rounded on its own.)
    T am = T(0), ax = T(0), ay = T(0);
#pragma unroll (ROLL ? 1 : 2)
    for (int side = 0; side < 2; ++side) {
        const T cr = cross_xy(xl, nl);
        am = fmaT(cross_xy(sub(xl, o), sub(nl, o)), fan_height(xl, nl, fo, l0, lx, ly), am);
        ax += cr;
        ay = fmaT(cr, plane_sum(xl, nl, l0, lx, ly), ay);
        if (cl) {
            E.store(m, xl, nl);
            ++m;
        }
        xl = xh;
        nl = nh;
        cl = ch;
    }
    m6 += am;
    x2 += ax;
    y6 += ay;
    I.m6 = m6;
    I.x2 = x2;
    I.y6 = y6;
    I.zmin = zmn;
    I.zmax = zmx;
    return m;
}

// 6 ∫ (z - c)_+ over the polygon of the n edges in E: fan from s (nx, ny), a point of the face
// plane at height c, over the parts of the edges above c.  FUSED: the offsets from that point
// are formed with one rounding (the octree kernels) instead of from its rounded coordinates (the
// uniform ones); the two differ in the last bit only, and each kernel keeps to one of them.
template <bool FUSED, class T, class Slots>
PSE_HD T level_fan(const Slots &E, int n, T c, T s, T nx, T ny)
{
    const T ox = mul_rn(s, nx), oy = mul_rn(s, ny);
    T g = T(0);
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        P3<T> ea, eb;
        E.load(k, ea, eb);
        const bool a_up = ea.z > c, b_up = eb.z > c;
        const T t = (c - ea.z) * fdiv(T(1), eb.z - ea.z);
        const T px = fmaT(t, eb.x - ea.x, ea.x), py = fmaT(t, eb.y - ea.y, ea.y);
        const T ux = a_up ? ea.x : px, uy = a_up ? ea.y : py, vx = b_up ? eb.x : px, vy = b_up ? eb.y : py;
        const T ax = FUSED ? fmaT(-s, nx, ux) : ux - ox, ay = FUSED ? fmaT(-s, ny, uy) : uy - oy;
        const T bx = FUSED ? fmaT(-s, nx, vx) : vx - ox, by = FUSED ? fmaT(-s, ny, vy) : vy - oy;
        const T fa = a_up ? ea.z - c : T(0), fb = b_up ? eb.z - c : T(0);
        const T cr = mul_rn(ax, by) - mul_rn(ay, bx);
        g += (a_up || b_up) ? mul_rn(cr, fa + fb) : T(0);
    }
    return g;
}

// The tetrahedron of a run given as arrays (clip frame, relative to the run's first cell).
template <class T>
struct TetArrays {
    const P3<T> *p, *n;
    PSE_HD P3<T> vtx(int i) const { return p[i]; }
    PSE_HD P3<T> nrm(int f) const { return n[f]; }
};

// The local frame of one run: origin q (the centroid held in the run and rounded to 1/256,
// so the cell planes and the levels c_j = j - q.z stay exact), the reference plane l(x, y) =
// l0 + lx x + ly y held inside the run's z range at the column centre, the run length K and
// the first level evaluated, j0 (0 if the tetrahedron may reach below the run, else 1).
template <class T>
struct RunFrame {
    T qx, qy, qz, l0, lx, ly;
    int K, j0;
};

template <class T, class Src>
PSE_HD RunFrame<T> run_frame(const Src &src, T lx, T ly, int K, bool lo_open)
{
    const P3<T> p0 = src.vtx(0), p1 = src.vtx(1), p2 = src.vtx(2), p3 = src.vtx(3);
    const T cx = T(0.25) * ((p0.x + p1.x) + (p2.x + p3.x));
    const T cy = T(0.25) * ((p0.y + p1.y) + (p2.y + p3.y));
    const T cz = T(0.25) * ((p0.z + p1.z) + (p2.z + p3.z));
    const T kf = (T)K;
    RunFrame<T> F;
    F.qx = floor(fmin(fmax(cx, T(0)), T(1)) * T(256) + T(0.5)) * T(1.0 / 256);
    F.qy = floor(fmin(fmax(cy, T(0)), T(1)) * T(256) + T(0.5)) * T(1.0 / 256);
    F.qz = floor(fmin(fmax(cz, T(0)), kf) * T(256) + T(0.5)) * T(1.0 / 256);
    const T xc = T(0.5) - F.qx, yc = T(0.5) - F.qy;
    const T at = fmaT(ly, yc - (cy - F.qy), fmaT(lx, xc - (cx - F.qx), cz - F.qz));
    F.l0 = fmaT(-ly, yc, fmaT(-lx, xc, fmin(fmax(at, -F.qz), kf - F.qz)));
    F.lx = lx;
    F.ly = ly;
    F.K = K;
    F.j0 = lo_open ? 0 : 1;
    return F;
}

// Whether the face (a, b, c; local frame, normal z component nz) can reach the run's column: its
// projection's bounding box meets the column and it is not vertical.
template <class T>
PSE_HD bool face_meets_column(const P3<T> &a, const P3<T> &b, const P3<T> &c, T nz, const RunFrame<T> &F)
{
    const T mnx = fmin(a.x, fmin(b.x, c.x)), mxx = fmax(a.x, fmax(b.x, c.x));
    const T mny = fmin(a.y, fmin(b.y, c.y)), mxy = fmax(a.y, fmax(b.y, c.y));
    if (mxx < -F.qx || mnx >= T(1) - F.qx || mxy < -F.qy || mny >= T(1) - F.qy) return false;
    return nz != T(0);
}

// The faces of a run that can reach its column [0,1)^2 (bit f), from the projected vertices p
// (clip frame, relative to the run's first cell) and the signs of the normals' z components
// (up: bit f set if face f's is positive).  A face is left out when the square lies beyond its
// bounding box or beyond one of its edges by a margin far above the rounding of the clip, which
// would then find an empty polygon and add exactly 0, so leaving it out changes no bit: the
// margins are 2e-3 of a cell plus 4e-6 (m + 1)^2 on the edge functions (m: the largest
// coordinate), against errors of about 3e-6 m in positions and 1e-6 m^2 in the edge functions;
// beyond m = 500 every face is kept.  A face seen edge-on, whose sign is rounding, is a segment
// to within those errors, so either sign is safe.  On the headline workload's tetrahedra this
// leaves 2.8 of 4 faces a run (3.2 by the bounding boxes alone).
PSE_HD unsigned face_mask(const P3<float> (&p)[4], unsigned up)
{
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) m = ::fmaxf(m, ::fmaxf(::fmaxf(::fabsf(p[i].x), ::fabsf(p[i].y)), ::fabsf(p[i].z)));
    if (!(m <= 500.f)) return 15u;
    const float gap = 2e-3f;
    bool out[4];
    {
        const float lx = ::fminf(p[0].x, p[1].x), hx = ::fmaxf(p[0].x, p[1].x), lx2 = ::fminf(p[2].x, p[3].x),
                    hx2 = ::fmaxf(p[2].x, p[3].x);
        const float ly = ::fminf(p[0].y, p[1].y), hy = ::fmaxf(p[0].y, p[1].y), ly2 = ::fminf(p[2].y, p[3].y),
                    hy2 = ::fmaxf(p[2].y, p[3].y);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            // the face's vertices: the other one of f's pair, and the other pair
            const P3<float> s = p[f ^ 1];
            const bool lowpair = f < 2;
            const float mnx = ::fminf(s.x, lowpair ? lx2 : lx), mxx = ::fmaxf(s.x, lowpair ? hx2 : hx);
            const float mny = ::fminf(s.y, lowpair ? ly2 : ly), mxy = ::fmaxf(s.y, lowpair ? hy2 : hy);
            out[f] = mxx < -gap || mnx > 1.f + gap || mxy < -gap || mny > 1.f + gap;
        }
    }
    // edge i -> j: the square is wholly to its left (L) or right (R)
    const float eps = 4e-6f * (m + 1.f) * (m + 1.f);
    bool L[6], R[6];
    constexpr int ei[6] = {0, 0, 0, 1, 1, 2}, ej[6] = {1, 2, 3, 2, 3, 3};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const P3<float> a = p[ei[k]], b = p[ej[k]];
        const float dx = b.x - a.x, dy = b.y - a.y;
        const float c = dx * (0.5f - a.y) - dy * (0.5f - a.x);
        const float r = fmaf(0.5f + gap, ::fabsf(dx) + ::fabsf(dy), eps);
        L[k] = c > r;
        R[k] = c < -r;
    }
    // outward loops (face_vertices): 1-2-3, 0-3-2, 0-1-3, 0-2-1; counter-clockwise when up
    const bool s0 = (up & 1u) ? (R[3] || R[5] || L[4]) : (L[3] || L[5] || R[4]);
    const bool s1 = (up & 2u) ? (R[2] || L[5] || L[1]) : (L[2] || R[5] || R[1]);
    const bool s2 = (up & 4u) ? (R[0] || R[4] || L[2]) : (L[0] || L[4] || R[2]);
    const bool s3 = (up & 8u) ? (R[1] || L[3] || L[0]) : (L[1] || R[3] || R[0]);
    return (out[0] || s0 ? 0u : 1u) | (out[1] || s1 ? 0u : 2u) | (out[2] || s2 ? 0u : 4u) | (out[3] || s3 ? 0u : 8u);
}

// One face of a run: the x and y slab passes (the clipped polygon is left in the first n slots
// of E), then 6 x its term of B(c_j) for the levels j0 .. K by the closed forms (a level the
// face straddles gets the "below" form m6; the fan of its part above the level is subtracted
// afterwards, see level_fan), its z range, its moment, and the straddled levels jlo .. jhi
// (empty when jlo > jhi) with the plane data their fans need.
template <int KW, class T>
struct FaceRun {
    T k6[KW + 1];
    T zmin, zmax, m6;
    int jlo, jhi, n;
    T nx, ny, nz, ef;  // face plane n . x = ef in the local frame
};

// a face that adds nothing to the run
template <int KW, class T>
PSE_HD void face_none(FaceRun<KW, T> &R)
{
#pragma unroll
    for (int j = 0; j <= KW; ++j) R.k6[j] = T(0);
    R.zmin = T(1e30);
    R.zmax = T(-1e30);
    R.m6 = T(0);
    R.jlo = 0;
    R.jhi = -1;
    R.n = 0;
    R.nx = R.ny = R.nz = R.ef = T(0);
}

// (a, b, c): the face's vertices in the local frame, outward order; nf: its normal.
template <int KW, class T, bool ROLL = false, class Slots>
PSE_HD void face_run(const P3<T> &a, const P3<T> &b, const P3<T> &c, const P3<T> &nf, const RunFrame<T> &F,
                     const Slots &E, FaceRun<KW, T> &R)
{
    const T mnx = fmin(a.x, fmin(b.x, c.x)), mxx = fmax(a.x, fmax(b.x, c.x));
    const T mny = fmin(a.y, fmin(b.y, c.y)), mxy = fmax(a.y, fmax(b.y, c.y));
    const T mnz = fmin(a.z, fmin(b.z, c.z)), mxz = fmax(a.z, fmax(b.z, c.z));
    const T cmag = fmax(T(1), fmax(fmax(fmax(fabs(mnx), fabs(mxx)), fmax(fabs(mny), fabs(mxy))),
                                   fmax(fabs(mnz), fabs(mxz))));
    const T tol = T(8) * roundoff<T>() * cmag;
    const T ef = fmaT(nf.z, a.z, fmaT(nf.x, a.x, mul_rn(nf.y, a.y)));
    const T sc = fdiv(ef, fmaT(nf.z, nf.z, fmaT(nf.x, nf.x, mul_rn(nf.y, nf.y))));
    const P3<T> o = mk<T>(mul_rn(sc, nf.x), mul_rn(sc, nf.y), T(0));  // (its z enters fo only)
    const T fo = fmaT(sc, nf.z, -fmaT(F.lx, o.x, fmaT(F.ly, o.y, F.l0)));

    const int n3 = xslab_triangle<ROLL, T>(a, b, c, -F.qx, T(1) - F.qx, tol, E);
    FaceSums<T> I;
    R.n = yslab_sums<ROLL, T>(E, n3, -F.qy, T(1) - F.qy, tol, o, fo, F.l0, F.lx, F.ly, I);

    // levels the polygon straddles: jlo .. jhi (c_j - zmin > 0 and zmax - c_j > 0)
    const T kf = (T)F.K;
    const T flo = fmin(fmax(floor(I.zmin + F.qz) + T(1), T(F.j0)), kf + T(1));
    const T fhi = fmin(fmax(ceil(I.zmax + F.qz) - T(1), T(-1)), kf);
    R.jlo = (int)flo;
    R.jhi = (int)fhi;
    // closed forms: below jlo the face is above the level; from jlo on it is (at first taken
    // as) below it
#pragma unroll
    for (int j = 0; j <= KW; ++j) {
        const T cj = (T)j - F.qz;
        const T v = (j < R.jlo) ? fmaT(T(3) * cj, I.x2, -I.y6) : I.m6;
        R.k6[j] = (j >= F.j0 && j <= F.K) ? v : T(0);
    }
    R.zmin = I.zmin;
    R.zmax = I.zmax;
    R.m6 = I.m6;
    R.nx = nf.x;
    R.ny = nf.y;
    R.nz = nf.z;
    R.ef = ef;
}

// The anchor of a level fan, the point of the face plane at height c nearest the local origin in
// the xy plane, is s (nx, ny).
template <class T>
PSE_HD T fan_anchor(T nx, T ny, T nz, T ef, T c)
{
    return fmaT(-nz, c, ef) * fdiv(T(1), fmaT(nx, nx, mul_rn(ny, ny)));
}

// Volume of the cell between the levels c0 and c1 of a run, from the level sums s = 6 B(c) over
// its faces: a level at or below the tetrahedron's lowest point in the column (colmin) holds
// exactly 0, and one at or above its highest point (colmax) the column's whole volume (msum / 6),
// so they are set so rather than left to the rounding of terms that cancel.
template <class T>
PSE_HD T level_volume(T c0, T c1, T s0, T s1, T colmin, T colmax, T msum)
{
    const T b0 = (c0 <= colmin) ? T(0) : ((c0 >= colmax) ? msum : s0);
    const T b1 = (c1 <= colmin) ? T(0) : ((c1 >= colmax) ? msum : s1);
    return (b1 - b0) * T(1.0 / 6.0);
}

// ---------------------------------------------------------------------------
// The float64 column clip (guarded tetrahedra).  GB300's float64 pipe takes 16 cycles a warp
// instruction on each SM, 64 issue slots, so this version of the clip is written for few float64
// operations: 1 in 2.5 of the generic stages above.
//  * Comparisons, minima and clamps read the numbers' bits (ordered as integers) instead of
//    the float64 pipe.
//  * The reciprocal of an edge's extent starts from the float32 one and takes one step of
//    Chebyshev's iteration, r (1 + e + e^2) with e = 1 - x r (the error falls from 1e-7 to below rounding).
//  * All integrals of a polygon come from four moments, Σ C, Σ C (x_a + x_b), Σ C (y_a + y_b) and
//    Σ C (z_a + z_b), with C the cross product of an edge's ends about one of the polygon's own
//    vertices (in the cell, so nothing cancels).
//  * A level's fan starts from a crossing point of the level line itself, so that no face
//    plane enters, and whole-polygon bounds are kept as ordered integers.
// The clip's error stays a few 1e-16 of a cell (1e-12 is tested).  The shell-crossed 128^3 octree deposit,
// seven tenths of it this clip, takes 141 ms with the generic stages and 76 with these.  Ten warps an SM
// instead of eight change nothing: the pipe is 86% busy.
// ---------------------------------------------------------------------------
PSE_HD long long f64_bits(double x)
{
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    std::memcpy(&b, &x, sizeof(b));
    return b;
#endif
}
PSE_HD double f64_of(long long b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    std::memcpy(&x, &b, sizeof(x));
    return x;
#endif
}
// an integer that orders like the number
PSE_HD long long f64_key(double x)
{
    const long long b = f64_bits(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
// x > t for t > 0
PSE_HD bool f64_above(double x, double t) { return f64_bits(x) > f64_bits(t); }

// t held in [0, 1]
PSE_HD double f64_sat01(double t)
{
    const long long b = f64_bits(t);
    return b < 0 ? 0.0 : (b >= 0x3ff0000000000000ll ? 1.0 : t);
}

// float32 to float64 without a conversion instruction (those share the float64 pipe's rate);
// a float32 denormal is not kept (it becomes about 1e-38)
PSE_HD double f64_widen(float x)
{
#ifdef __CUDA_ARCH__
    const int b = __float_as_int(x), m = b & 0x7fffffff;
    const int hi = m == 0 ? 0 : (b & (int)0x80000000) | ((m >> 3) + 0x38000000);
    return __hiloint2double(hi, m == 0 ? 0 : b << 29);
#else
    return (double)x;
#endif
}

// 1 / x (0 for an x beyond 2^-100 .. 2^100: an edge that does not cross anything), within an ulp: the float32
// reciprocal of x cut to float32 (error e below 2^-21), then one step of Chebyshev's iteration for 1 / x
// (Altman's hyperpower method of order three), which leaves e^3
PSE_HD double f64_rcp(double x)
{
#ifdef __CUDA_ARCH__
    const int hi = __double2hiint(x), m = hi & 0x7fffffff;
    const bool ok = (unsigned)(m - ((1023 - 100) << 20)) < (200u << 20);
    const float f = __int_as_float((hi & (int)0x80000000) | (((m - 0x38000000) << 3) | (int)((unsigned)__double2loint(x) >> 29)));
    const int b = __float_as_int(slab_rcp(f));
    const double r = __hiloint2double((b & (int)0x80000000) | (((b & 0x7fffffff) >> 3) + 0x38000000), b << 29);
    const double e = fma(-x, r, 1.0);
    return ok ? fma(r, fma(e, e, e), r) : 0.0;
#else
    return x != 0.0 ? 1.0 / x : 0.0;
#endif
}

template <int KW>
struct FaceRun64 {
    double k6[KW + 1];
    double m6;
    long long kmin, kmax;  // z range of the polygon, as ordered integers
    int jlo, jhi, n;
};
constexpr long long kKeyMax = 0x7fffffffffffffffll, kKeyMin = -kKeyMax - 1;

template <int KW>
PSE_HD void face_none(FaceRun64<KW> &R)
{
#pragma unroll
    for (int j = 0; j <= KW; ++j) R.k6[j] = 0.0;
    R.m6 = 0.0;
    R.kmin = kKeyMax;
    R.kmax = kKeyMin;
    R.jlo = 0;
    R.jhi = -1;
    R.n = 0;
}

// Moments of a polygon, edge by edge: fan triangles from its vertex o.
struct Moments64 {
    double c, x, y, z;
    P3<double> o;
    PSE_HD void add(const P3<double> &a, const P3<double> &b, bool on)
    {
        const double ux = a.x - o.x, uy = a.y - o.y, wx = b.x - o.x, wy = b.y - o.y;
        const double cr = on ? fma(ux, wy, -(uy * wx)) : 0.0;
        c += cr;
        x = fma(cr, a.x + b.x, x);
        y = fma(cr, a.y + b.y, y);
        z = fma(cr, a.z + b.z, z);
    }
    // an edge on the plane y = h
    PSE_HD void add_at(const P3<double> &a, const P3<double> &b, double h, bool on)
    {
        const double cr = on ? (h - o.y) * (a.x - b.x) : 0.0;
        c += cr;
        x = fma(cr, a.x + b.x, x);
        y = fma(cr, h + h, y);
        z = fma(cr, a.z + b.z, z);
    }
};

// One face (a, b, c) of a run in the local frame: as face_run, tol the classification tolerance.
template <int KW, class Slots>
PSE_HD void face_run_f64(const P3<double> &a, const P3<double> &b, const P3<double> &c, const RunFrame<double> &F,
                         double tol, const Slots &E, FaceRun64<KW> &R)
{
    // ---- x slab: lo <= x < hi
    int n = 0;
    {
        const double lo = -F.qx, hi = 1.0 - F.qx;
        const P3<double> p[3] = {a, b, c};
        double dl[3], dh[3];
        bool below[3], above[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            dl[i] = lo - p[i].x;
            dh[i] = hi - p[i].x;
            below[i] = f64_above(dl[i], tol);
            above[i] = !f64_above(dh[i], tol);
        }
        double xly = 0.0, xlz = 0.0, nly = 0.0, nlz = 0.0, xhy = 0.0, xhz = 0.0, nhy = 0.0, nhz = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int j = i == 2 ? 0 : i + 1;
            const double inv = f64_rcp(p[j].x - p[i].x);
            const double ta = f64_sat01((below[i] ? dl[i] : dh[i]) * inv), tb = f64_sat01((below[j] ? dl[i] : dh[i]) * inv);
            const double dy = p[j].y - p[i].y, dz = p[j].z - p[i].z;
            const bool ina = !below[i] && !above[i], inb = !below[j] && !above[j];
            const double ay = ina ? p[i].y : fma(ta, dy, p[i].y), az = ina ? p[i].z : fma(ta, dz, p[i].z);
            const double by = inb ? p[j].y : fma(tb, dy, p[i].y), bz = inb ? p[j].z : fma(tb, dz, p[i].z);
            if (!below[i] && below[j]) { xly = by; xlz = bz; }
            if (below[i] && !below[j]) { nly = ay; nlz = az; }
            if (!above[i] && above[j]) { xhy = by; xhz = bz; }
            if (above[i] && !above[j]) { nhy = ay; nhz = az; }
            if (!(below[i] && below[j]) && !(above[i] && above[j])) {
                const double ax = ina ? p[i].x : (below[i] ? lo : hi), bx = inb ? p[j].x : (below[j] ? lo : hi);
                E.store(n, mk<double>(ax, ay, az), mk<double>(bx, by, bz));
                ++n;
            }
        }
        if ((below[0] || below[1] || below[2]) && !(below[0] && below[1] && below[2])) {
            E.store(n, mk<double>(lo, xly, xlz), mk<double>(lo, nly, nlz));
            ++n;
        }
        if ((above[0] || above[1] || above[2]) && !(above[0] && above[1] && above[2])) {
            E.store(n, mk<double>(hi, xhy, xhz), mk<double>(hi, nhy, nhz));
            ++n;
        }
    }
    // ---- y slab, and the polygon's moments and z range
    const double lo = -F.qy, hi = 1.0 - F.qy;
    const long long klo = f64_key(lo - tol), khi = f64_key(hi - tol);
    P3<double> xl = mk<double>(0.0, lo, 0.0), nl = xl, xh = mk<double>(0.0, hi, 0.0), nh = xh;
    bool cl = false, ch = false, any = false;
    Moments64 M;
    M.c = M.x = M.y = M.z = 0.0;
    M.o = mk<double>(0.0, 0.0, 0.0);
    long long kmin = kKeyMax, kmax = kKeyMin;
    int m = 0;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        P3<double> ea, eb;
        E.load(k, ea, eb);
        const long long kya = f64_key(ea.y), kyb = f64_key(eb.y);
        const bool a_lo = kya < klo, a_hi = kya >= khi, b_lo = kyb < klo, b_hi = kyb >= khi;
        const double dl = lo - ea.y, dh = hi - ea.y;
        const double inv = f64_rcp(eb.y - ea.y);
        const double ta = f64_sat01((a_lo ? dl : dh) * inv), tb = f64_sat01((b_lo ? dl : dh) * inv);
        const double dx = eb.x - ea.x, dz = eb.z - ea.z;
        const bool ina = !a_lo && !a_hi, inb = !b_lo && !b_hi;
        const P3<double> na = mk<double>(ina ? ea.x : fma(ta, dx, ea.x), ina ? ea.y : (a_lo ? lo : hi),
                                         ina ? ea.z : fma(ta, dz, ea.z));
        const P3<double> nb = mk<double>(inb ? eb.x : fma(tb, dx, ea.x), inb ? eb.y : (b_lo ? lo : hi),
                                         inb ? eb.z : fma(tb, dz, ea.z));
        if (!a_lo && b_lo) { xl = nb; cl = true; }
        if (a_lo && !b_lo) nl = na;
        if (!a_hi && b_hi) { xh = nb; ch = true; }
        if (a_hi && !b_hi) nh = na;
        const bool live = !(a_lo && b_lo) && !(a_hi && b_hi);
        if (live && !any) M.o = na;
        M.add(na, nb, live);
        if (live) {
            any = true;
            const long long ka = f64_key(na.z), kb = f64_key(nb.z);
            const long long kl = ka < kb ? ka : kb, kh = ka < kb ? kb : ka;
            kmin = kl < kmin ? kl : kmin;
            kmax = kh > kmax ? kh : kmax;
            E.store(m, na, nb);
            ++m;
        }
    }
    M.add_at(xl, nl, lo, cl);
    M.add_at(xh, nh, hi, ch);
    if (cl) {
        E.store(m, xl, nl);
        ++m;
    }
    if (ch) {
        E.store(m, xh, nh);
        ++m;
    }
    R.n = m;
    R.kmin = kmin;
    R.kmax = kmax;
    // 6 ∫ f of a linear f is Σ C (f(o) + f(a) + f(b)); l6: of the plane l; the face's own height less l;
    // a constant c less l is c a6 - l6
    const double a6 = 3.0 * M.c;
    const double l6 = fma(F.lx, fma(M.c, M.o.x, M.x), fma(F.ly, fma(M.c, M.o.y, M.y), a6 * F.l0));
    R.m6 = fma(M.c, M.o.z, M.z) - l6;
    int jlo = F.j0, jhi = -1;
#pragma unroll
    for (int j = 0; j <= KW; ++j) {
        const double cj = f64_widen((float)j) - F.qz;
        const long long kj = f64_key(cj);
        if (j <= F.K) {
            jlo += (j >= F.j0 && kj <= kmin) ? 1 : 0;
            jhi += kj < kmax ? 1 : 0;
        }
        // (levels below jlo: the face lies above them; kj <= kmin)
        R.k6[j] = (j >= F.j0 && j <= F.K) ? (kj <= kmin ? fma(a6, cj, -l6) : R.m6) : 0.0;
    }
    R.jlo = jlo;
    R.jhi = jhi;
}

// 6 ∫ (z - c)_+ over the polygon of the n edges in E, as level_fan.
template <class Slots>
PSE_HD double level_fan_f64(const Slots &E, int n, double c)
{
    const long long kc = f64_key(c);
    // the first edge that crosses the level
    int first = -1;
    P3<double> ea, eb;
#pragma unroll 1
    for (int k = 0; k < n && first < 0; ++k) {
        E.load(k, ea, eb);
        if ((f64_key(ea.z) > kc) != (f64_key(eb.z) > kc)) first = k;
    }
    if (first < 0) return 0.0;
    double t = (c - ea.z) * f64_rcp(eb.z - ea.z);
    const double ox = fma(t, eb.x - ea.x, ea.x), oy = fma(t, eb.y - ea.y, ea.y);
    double g = 0.0;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        E.load(k, ea, eb);
        const bool a_up = f64_key(ea.z) > kc, b_up = f64_key(eb.z) > kc;
        if (!a_up && !b_up) continue;
        double px = ox, py = oy;  // an edge wholly above does not use it
        const double fa = c - ea.z;
        if (a_up != b_up && k != first) {
            t = fa * f64_rcp(eb.z - ea.z);
            px = fma(t, eb.x - ea.x, ea.x);
            py = fma(t, eb.y - ea.y, ea.y);
        }
        const double ax = (a_up ? ea.x : px) - ox, ay = (a_up ? ea.y : py) - oy;
        const double bx = (b_up ? eb.x : px) - ox, by = (b_up ? eb.y : py) - oy;
        const double h = (a_up ? -fa : 0.0) + (b_up ? eb.z - c : 0.0);
        g = fma(fma(ax, by, -(ay * bx)), h, g);
    }
    return g;
}

// The volume between two levels, as level_volume, from the ordered z range.
PSE_HD double level_volume_f64(double c0, double c1, double s0, double s1, long long kmin, long long kmax, double msum)
{
    const long long k0 = f64_key(c0), k1 = f64_key(c1);
    const double b0 = k0 <= kmin ? 0.0 : (k0 >= kmax ? msum : s0);
    const double b1 = k1 <= kmin ? 0.0 : (k1 >= kmax ? msum : s1);
    return (b1 - b0) * (1.0 / 6.0);
}

// The classification tolerance for coordinates of up to `extent` cells.
PSE_HD double f64_tolerance(double extent) { return 8.0 * 2.220446049250313e-16 * (1.0 + extent); }

template <int KW, class Src>
PSE_HD void column_volumes_f64(const Src &src, double lx, double ly, int K, bool lo_open, double (&vol)[KW],
                               double2 *slots)
{
    const RunFrame<double> F = run_frame<double>(src, lx, ly, K, lo_open);
    const EdgeSlots<double> E{slots};
    const P3<double> q = mk<double>(F.qx, F.qy, F.qz);
    double extent = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const P3<double> v = src.vtx(i);
        extent = fmax(extent, fmax(fmax(fabs(v.x), fabs(v.y)), fabs(v.z)));
    }
    double S[KW + 1], msum = 0.0;
#pragma unroll
    for (int j = 0; j <= KW; ++j) S[j] = 0.0;
    long long kmin = kKeyMax, kmax = kKeyMin;
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
        int ia, ib, ic;
        face_vertices(f, ia, ib, ic);
        FaceRun64<KW> R;
        face_run_f64<KW>(sub(src.vtx(ia), q), sub(src.vtx(ib), q), sub(src.vtx(ic), q), F, f64_tolerance(extent), E, R);
#pragma unroll 1
        for (int j = R.jlo; j <= R.jhi; ++j) {
            const double g = level_fan_f64(E, R.n, (double)j - F.qz);
#pragma unroll
            for (int i = 0; i <= KW; ++i) R.k6[i] -= (i == j) ? g : 0.0;
        }
#pragma unroll
        for (int j = 0; j <= KW; ++j) S[j] += R.k6[j];
        kmin = R.kmin < kmin ? R.kmin : kmin;
        kmax = R.kmax > kmax ? R.kmax : kmax;
        msum += R.m6;
    }
#pragma unroll
    for (int j = 0; j < KW; ++j)
        vol[j] = level_volume_f64((double)j - F.qz, (double)(j + 1) - F.qz, S[j], S[j + 1], kmin, kmax, msum);
}

// Overlap volumes of a positively oriented tetrahedron (clip frame, relative to the first
// cell of the run: the run is [0,1)^2 x [0,K), K <= KW) with the K cells of the run.  src
// gives vertex i (src.vtx(i)) and the outward normal of face f (src.nrm(f)), read when
// needed; (lx, ly): reference slopes.  lo_open: the tetrahedron may reach below the run (a
// run that starts above its bounding box's first layer); otherwise B(0) is exactly 0.
// E: this lane's edge slots (two-scalar rows with a stride of 32).  This is the clip of one run
// by one thread; the warp kernels deal its faces and its level fans out to lanes (common.cuh)
// with the same stages and the same order of the sums.
template <int KW, class T, class Src>
PSE_HD void column_volumes(const Src &src, T lx, T ly, int K, bool lo_open, T (&vol)[KW], slot2_t<T> *slots)
{
    if constexpr (std::is_same<T, double>::value) {
        column_volumes_f64<KW>(src, lx, ly, K, lo_open, vol, slots);
        return;
    }
    const RunFrame<T> F = run_frame<T>(src, lx, ly, K, lo_open);
    const EdgeSlots<T> E{slots};
    const P3<T> q = mk<T>(F.qx, F.qy, F.qz);
    // S[j]: 6 B(c_j), c_j = j - q.z, j = 0 .. KW (levels past K are unused)
    T S[KW + 1];
#pragma unroll
    for (int j = 0; j <= KW; ++j) S[j] = T(0);
    // the tetrahedron's z range inside the column, and 6 x its volume there
    T colmin = T(1e30), colmax = T(-1e30), msum = T(0);
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
        int ia, ib, ic;
        face_vertices(f, ia, ib, ic);
        const P3<T> a = sub(src.vtx(ia), q), b = sub(src.vtx(ib), q), c = sub(src.vtx(ic), q);
        const P3<T> nf = src.nrm(f);
        if (!face_meets_column<T>(a, b, c, nf.z, F)) continue;
        FaceRun<KW, T> R;
        face_run<KW, T>(a, b, c, nf, F, E, R);
#pragma unroll 1
        for (int j = R.jlo; j <= R.jhi; ++j) {  // straddled levels: subtract the part above
            const T cj = (T)j - F.qz;
            const T g = level_fan<false, T>(E, R.n, cj, fan_anchor<T>(R.nx, R.ny, R.nz, R.ef, cj), R.nx, R.ny);
#pragma unroll
            for (int i = 0; i <= KW; ++i) R.k6[i] -= (i == j) ? g : T(0);
        }
#pragma unroll
        for (int j = 0; j <= KW; ++j) S[j] += R.k6[j];
        colmin = fmin(colmin, R.zmin);
        colmax = fmax(colmax, R.zmax);
        msum += R.m6;
    }
#pragma unroll
    for (int j = 0; j < KW; ++j)
        vol[j] = level_volume<T>((T)j - F.qz, (T)(j + 1) - F.qz, S[j], S[j + 1], colmin, colmax, msum);
}

}  // namespace pse
