// eses_edges.cu -- crossing edges, surface roots and normals, area and volume
// (the third and fourth ESES stages, Eq. 3-4).
//
// k_edge_count: per tile and axis, the edges (p, p + e_a) leaving the tile's
//   points whose end labels differ, and the edges with both ends inside.
// (exclusive scan of the counts -> every tile's output offset per axis; the
//   paper serialises this output step in a critical section, Algorithm 1)
// The root solve: the surface along an edge is made of pieces of van der
//   Waals spheres (convex), tori around pair circles (saddle) and probe
//   spheres around free triple points (concave).  Every root of every such
//   piece in [0, h] whose witness (projection on the expanded sphere /
//   nearest circle point / the triple point) is free, and whose witness
//   distance crosses r_p in the direction that leaves the end point's side
//   (falling from an inside end, rising from an outside end), is a candidate.
//   From an inside end point the first candidate is the first root; from an
//   outside end point the first candidate that is not strictly outside M is.
//   Seven launches linked by lists in HBM:
//   k_edge_stage: persistent CTAs take tiles from the work queue; per tile
//     the pieces are staged (shared memory, or the global-memory tier for a
//     tile that overflows it), the crossing edges listed, and written out:
//     the staged lists (the tile's slab), an edge record per edge, and the
//     (edge, piece) pairs that pass a prefilter (32 edges a warp, a lane each,
//     against the same pieces), spheres and tori in separate lists;
//   k_roots_sphere / k_roots_torus: one thread per pair, no block barrier:
//     sphere roots from the quadratic; torus roots of
//          (|y-o|^2 + rho^2 - r_p^2)^2 = 4 rho^2 (|y-o|^2 - ((y-o).u)^2)
//     on the near branch (|w| - rho)^2 + z^2 = r_p^2, isolated in FP32 on
//     eight sub-intervals with certified exclusion and monotonicity tests and
//     refined by Newton (undecided: the quartic on its derivative chain, then
//     FP64); every FP32 root carries an error bound; the accepted roots go to
//     the pair's slots;
//   k_roots_torus_exact: the tori's FP64 work that those leave, one thread each;
//   k_edge_pick: one thread per edge: the first root when the end point is
//     inside, the last one when it is outside and the first lies within r_p of
//     the last one's witness, where the FP32 bounds order the candidates; the
//     other edges are listed, with the candidates that are nearly tied;
//   k_edge_ties: FP64 roots of near ties, one thread each;
//   k_edge_hard: one warp per edge left: near ties broken on FP64 roots; at
//     an outside end point each earlier candidate tested first against the
//     later candidates' witnesses, then by the full witness search, whose
//     undecided items are re-tested in FP64.
//   The chosen piece and its FP32 root are recorded for the polish.
// k_edge_polish: one thread per crossing edge (full warps of FP64 work): the
//   FP64 root of the chosen piece next to the recorded one, the normal, the
//   outputs and the area/volume terms.
// k_reduce: per molecule, area = h^2 sum |n_a|, volume = h^2/3 sum of
//   inside lengths.
// Every tile kernel runs over the tiles of all molecules of a batch.
#include <math.h>

#include <algorithm>

#include "eses_kernels.h"
#include "eses_tile.cuh"

namespace eses {

constexpr int EDGE_THREADS = 256;
constexpr int EDGE_WARPS = EDGE_THREADS / 32;
constexpr int WCAND = 64;        // candidate roots of one edge in the selection buffer
constexpr int ROOT_THREADS_MAX = 256;  // per-candidate root kernels: threads per block (at most, the default)
constexpr int PICK_THREADS = 256;
constexpr int HARD_THREADS = 256;
constexpr int HMASK_WORDS = 1536;  // prefilter hit masks kept between the staging pass's two sweeps
constexpr int POLISH_THREADS = 256;

// --------------------------------------------------------------------------
// polynomial roots on an interval
// --------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ R root_eps();
template <>
__device__ __forceinline__ double root_eps<double>() { return 1e-15; }
template <>
__device__ __forceinline__ float root_eps<float>() { return 2e-7f; }

template <class R>
__device__ __forceinline__ R fp_eps();
template <>
__device__ __forceinline__ double fp_eps<double>() { return 2.3e-16; }
template <>
__device__ __forceinline__ float fp_eps<float>() { return 1.2e-7f; }

template <class R, int DEG>
__device__ __forceinline__ R horner(const R *c, R t)
{
    R v = c[DEG];
#pragma unroll
    for (int k = DEG - 1; k >= 0; --k) v = fma(v, t, c[k]);
    return v;
}

// root of c on [a, b], where c is monotone and f(a) (= fa) and f(b) differ in sign
template <class R, int DEG>
__device__ R mono_root(const R *c, R a, R b, R fa)
{
    R dc[DEG];
#pragma unroll
    for (int k = 0; k < DEG; ++k) dc[k] = (R)(k + 1) * c[k + 1];
    // rounding of c's value on [a, b]
    const R m = fmax(fabs(a), fabs(b));
    R noise = fabs(c[DEG]);
#pragma unroll
    for (int k = DEG - 1; k >= 0; --k) noise = noise * m + fabs(c[k]);
    noise *= fp_eps<R>();
    R t = R(0.5) * (a + b), step = INFINITY;
    for (int it = 0; it < 100; ++it) {
        R f = horner<R, DEG>(c, t);
        if (f == R(0)) return t;
        if ((f < R(0)) == (fa < R(0))) a = t;
        else b = t;
        R df = horner<R, DEG - 1>(dc, t);
        R tn = (df != R(0)) ? t - f / df : R(0.5) * (a + b);
        const bool out = !(tn > a && tn < b);
        // at its rounding f gives no better t once the steps leave the bracket
        // or no longer shrink (without this the search goes back to the middle of
        // the bracket, again and again until that has closed or for 100 steps)
        if (fabs(f) <= noise && (out || fabs(tn - t) >= R(0.75) * step)) return out ? t : tn;
        if (out) tn = R(0.5) * (a + b);
        const R d = fabs(tn - t);
        if (d <= root_eps<R>() * fmax(R(1), fabs(t))) return tn;
        step = d;
        t = tn;
        if (b - a <= root_eps<R>() * fmax(R(1), fabs(a))) return R(0.5) * (a + b);
    }
    return t;
}

// roots of c[0] + c[1] t + ... + c[DEG] t^DEG in [lo, hi], ascending: the
// derivative's roots split [lo, hi] into monotone pieces, each holding at most
// one root, found by safeguarded Newton-bisection
template <class R, int DEG>
struct PolyRoots {
    __device__ static __noinline__ int run(const R *c, R lo, R hi, R *out)
    {
        R dc[DEG];
#pragma unroll
        for (int k = 0; k < DEG; ++k) dc[k] = (R)(k + 1) * c[k + 1];
        R crit[DEG - 1];
        int ncr = PolyRoots<R, DEG - 1>::run(dc, lo, hi, crit);
        R pts[DEG + 1];
        int np = 0;
        pts[np++] = lo;
        for (int k = 0; k < ncr; ++k)
            if (crit[k] > pts[np - 1] && crit[k] < hi) pts[np++] = crit[k];
        pts[np++] = hi;
        int n = 0;
        R fprev = horner<R, DEG>(c, pts[0]);
        if (fprev == R(0)) out[n++] = pts[0];
        for (int k = 0; k + 1 < np; ++k) {
            R fnext = horner<R, DEG>(c, pts[k + 1]);
            if (fnext == R(0)) {
                if (n == 0 || out[n - 1] != pts[k + 1]) out[n++] = pts[k + 1];
            } else if (fprev != R(0) && ((fprev < R(0)) != (fnext < R(0)))) {
                out[n++] = mono_root<R, DEG>(c, pts[k], pts[k + 1], fprev);
            }
            fprev = fnext;
        }
        return n;
    }
};

template <class R>
struct PolyRoots<R, 1> {
    __device__ static int run(const R *c, R lo, R hi, R *out)
    {
        if (c[1] == R(0)) return 0;
        R t = -c[0] / c[1];
        if (t >= lo && t <= hi) {
            out[0] = t;
            return 1;
        }
        return 0;
    }
};

template <class R>
struct PolyRoots<R, 2> {
    __device__ static int run(const R *c, R lo, R hi, R *out)
    {
        R a = c[2], b = c[1], cc = c[0];
        if (a == R(0)) return PolyRoots<R, 1>::run(c, lo, hi, out);
        R disc = b * b - R(4) * a * cc;
        if (disc < R(0)) return 0;
        R sq = sqrt(disc);
        R q = R(-0.5) * (b + (b >= R(0) ? sq : -sq));
        R r1 = q / a;
        R r2 = (q != R(0)) ? cc / q : r1;
        if (r1 > r2) {
            R tmp = r1;
            r1 = r2;
            r2 = tmp;
        }
        int n = 0;
        if (r1 >= lo && r1 <= hi) out[n++] = r1;
        if (r2 >= lo && r2 <= hi && (n == 0 || r2 != out[0])) out[n++] = r2;
        return n;
    }
};

// --------------------------------------------------------------------------
// exact (FP64) roots and normals of one piece, any common frame
// --------------------------------------------------------------------------
// root of |s + t e_axis - c| = rad nearest t0 (t0 returned when none is real)
__device__ __forceinline__ double exact_root_sphere(const double *c, double rad, const double *s, int axis, double t0)
{
    double d[3] = {s[0] - c[0], s[1] - c[1], s[2] - c[2]};
    double b = d[axis];
    double cc = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] - rad * rad;
    double disc = b * b - cc;
    if (disc < 0.0) return t0;
    double sq = sqrt(disc);
    double q = -(b + (b >= 0.0 ? sq : -sq));
    double r1 = q, r2 = (q != 0.0) ? cc / q : q;
    return fabs(r1 - t0) <= fabs(r2 - t0) ? r1 : r2;
}

__device__ __forceinline__ void torus_coeffs(const double *o, const double *u, double rho, double rp, const double *s,
                                             int axis, double *co)
{
    double p0[3] = {s[0] - o[0], s[1] - o[1], s[2] - o[2]};
    double P = p0[0] * p0[0] + p0[1] * p0[1] + p0[2] * p0[2];
    double z0 = p0[0] * u[0] + p0[1] * u[1] + p0[2] * u[2];
    double pe = p0[axis], eu = u[axis];
    double K = P + rho * rho - rp * rp;
    double r2 = rho * rho;
    co[4] = 1.0;
    co[3] = 4.0 * pe;
    co[2] = 4.0 * pe * pe + 2.0 * K - 4.0 * r2 * (1.0 - eu * eu);
    co[1] = 4.0 * pe * K - 8.0 * r2 * (pe - z0 * eu);
    co[0] = K * K - 4.0 * r2 * (P - z0 * z0);
}

// FP64 Newton steps on the torus quartic from t0, at most four (the FP32 root
// is within 1e-3 A and the root simple, else the warp solve already took it in
// FP64): quadratic convergence, so the steps stop once one moves t by less
// than 1e-13 A (the next would move it by about the square of that)
// (`last`: the last step's length)
__device__ __noinline__ double exact_root_torus(const double *o, const double *u, double rho, double rp,
                                                   const double *s, int axis, double t0, double *last = nullptr)
{
    double co[5];
    torus_coeffs(o, u, rho, rp, s, axis, co);
    double dc[4] = {co[1], 2.0 * co[2], 3.0 * co[3], 4.0};
    double t = t0, dt = INFINITY;
    for (int it = 0; it < 4; ++it) {
        double f = horner<double, 4>(co, t);
        double df = horner<double, 3>(dc, t);
        if (df == 0.0) break;
        dt = f / df;
        t -= dt;
        if (fabs(dt) < 1e-13) break;
    }
    if (last) *last = fabs(dt);
    return t;
}

// The polish's form of the two, with the unit normal (towards the witness, i.e.
// into the solvent), in as few FP64 instructions as the same accuracy takes: a
// warp issues one in 16 cycles, a division or square root is about ten of them.
__device__ __forceinline__ void unit_of(double *n)
{
    const double vv = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
    const double iv = vv > 0.0 ? rsqrt(vv) : 0.0;
    n[0] *= iv;
    n[1] *= iv;
    n[2] *= iv;
}

__device__ __forceinline__ double into_edge(double t, double h) { return t > 0.0 ? (t < h ? t : h) : 0.0; }

// Sphere (`out`: 1 an atom's, its normal radial; -1 a probe's, towards its
// centre).  The root is -b +- sqrt(rad^2 - the distance^2 of the edge's line),
// without the b^2 that the quadratic's discriminant adds and takes off again
// and without a division: its largest and mean error against 80-bit arithmetic
// are at or below the quadratic formula's (mean 2.8e-16 and 3.3e-16 A at h 0.1).
__device__ __forceinline__ double polish_sphere(const double *c, double rad, double out, const double *s, int axis,
                                                double t0, double h, double *n)
{
    double d[3] = {s[0] - c[0], s[1] - c[1], s[2] - c[2]};
    const double b = d[axis];
    const double p = d[axis == 0 ? 1 : 0], q = d[axis == 2 ? 1 : 2];
    const double disc = (rad * rad - p * p) - q * q;
    double t;
    if (disc > 1e-4) {
        const double sq = sqrt(disc);
        t = t0 <= -b ? -b - sq : -b + sq;  // the root on t0's side of their middle
    } else {  // near a tangent a root moves by the square root of the rounding: the selection's form
        t = exact_root_sphere(c, rad, s, axis, t0);
    }
    t = into_edge(t, h);
    d[axis] += t;
    n[0] = out * d[0];
    n[1] = out * d[1];
    n[2] = out * d[2];
    unit_of(n);
    return t;
}

// Torus: Newton steps on the quartic as exact_root_torus, the slope's inverse
// in FP32 (the step's relative error, 1e-7, only multiplies the error that is
// left), ended once a step moves t by less than 1e-11 A (the next would move
// it by the square of that times the quartic's curvature over its slope, and
// by 1e-18 A for the slope's rounding); normal towards the nearest point of
// the circle.
__device__ __forceinline__ double polish_torus(const double *o, const double *u, double rho, double rp, const double *s,
                                               int axis, double t0, double h, double *n)
{
    double co[5];
    torus_coeffs(o, u, rho, rp, s, axis, co);
    const double dc[4] = {co[1], 2.0 * co[2], 3.0 * co[3], 4.0};
    double t = t0;
    for (int it = 0; it < 4; ++it) {
        const double f = horner<double, 4>(co, t);
        const float df = (float)horner<double, 3>(dc, t);
        if (fabsf(df) < 5e-2f) {  // nearly a double root: the selection's form, as for spheres
            t = exact_root_torus(o, u, rho, rp, s, axis, t0);
            break;
        }
        const double dt = f * (double)(1.0f / df);
        t -= dt;
        if (fabs(dt) < 1e-11) break;
    }
    t = into_edge(t, h);
    double y[3] = {s[0] - o[0], s[1] - o[1], s[2] - o[2]}, w[3];
    y[axis] += t;
    // the direction from the circle's axis to y, as axis_normal; y on the axis is left to it
    const double z = y[0] * u[0] + y[1] * u[1] + y[2] * u[2];
    for (int k = 0; k < 3; ++k) w[k] = y[k] - z * u[k];
    const double zr = w[0] * u[0] + w[1] * u[1] + w[2] * u[2];
    for (int k = 0; k < 3; ++k) w[k] -= zr * u[k];
    const double ww = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    if ((float)ww > 1e-12f * (1.0f + (float)z * (float)z)) {
        const double k = rho * rsqrt(ww);
        n[0] = k * w[0] - y[0];
        n[1] = k * w[1] - y[1];
        n[2] = k * w[2] - y[2];
    } else {
        axis_normal(y, u, w);
        n[0] = rho * w[0] - y[0];
        n[1] = rho * w[1] - y[1];
        n[2] = rho * w[2] - y[2];
    }
    unit_of(n);
    return t;
}

// exact root of a staged piece (tile frame, FP64 data from HBM) near t0
template <class XA>
__device__ __noinline__ double staged_exact_root(const XA &X, int kind, int slot, const double *s,
                                                    int axis, double rp, double t0)
{
    if (kind == 0) {
        P4<double> c = X.atom(slot);
        double cc[3] = {c.x, c.y, c.z};
        return exact_root_sphere(cc, c.w, s, axis, t0);
    }
    if (kind == 2) {
        P4<double> c = X.vq(slot);
        double cc[3] = {c.x, c.y, c.z};
        return exact_root_sphere(cc, rp, s, axis, t0);
    }
    P4<double> o = X.po(slot);
    P4<double> u = X.pu(slot);
    double oo[3] = {o.x, o.y, o.z}, uu[3] = {u.x, u.y, u.z};
    return exact_root_torus(oo, uu, o.w, rp, s, axis, t0);
}

// --------------------------------------------------------------------------
// the phased root solve: data between the launches
// --------------------------------------------------------------------------
// A candidate root of one crossing edge during the selection.
struct WCand {
    double t64;    // exact root once computed (NaN before)
    float t, err;  // FP32 root and its error bound (A)
    int kind, id;  // kind 0: van der Waals sphere (atom slot), 1: torus (pair slot), 2: probe sphere (vertex slot)
};

// A surface point on a grid point is a root at an end of its edges, which
// rounding leaves on either side of the end (Newton's limit from an exact tie
// is 1e-28 A off, a sphere's root an ulp); dropped there, the edge has no root
// or takes a later one.  Roots that far outside [0, h] are taken at the end;
// the crossing's direction keeps the neighbouring edge's root out.
constexpr double END_TOL = 1e-11;
__device__ __forceinline__ double at_end(double t, double h)
{
    if (t < 0.0 && t >= -END_TOL) return 0.0;
    return t > h && t <= h + END_TOL ? h : t;
}

// Accepted roots of one (edge, piece) candidate, written to the candidate's
// slots in HBM (at most SPH_SLOTS for a sphere, whose two roots cross in
// opposite directions; at most TOR_SLOTS, the quartic's degree, for a torus).
constexpr int SPH_SLOTS = 2;
constexpr int TOR_SLOTS = 4;
struct RootSink {
    RootRec *r;
    int n, cap;
    __device__ __forceinline__ void push(float t, float err, double t64)
    {
        if (n < cap) {
            RootRec q;
            q.t64 = t64;
            q.t = t;
            q.err = err;
            r[n] = q;
        }
        ++n;
    }
    // a slot kept for a root whose decision needs FP64 (err < 0: pending; the
    // FP32 root kept in t), settled by k_roots_torus_exact
    __device__ __forceinline__ void pend(float t) { push(t, -1.0f, __longlong_as_double(0x7ff8000000000000LL)); }
};
// a settled slot whose root was rejected
__device__ __forceinline__ RootRec no_root()
{
    RootRec q;
    q.t64 = __longlong_as_double(0x7ff8000000000000LL);
    q.t = INFINITY;
    q.err = 0.0f;
    return q;
}

// Lower point p (local index) of an edge in the tile frame, and the spacing,
// in T: for FP32 the molecule's table of k * h rounded to FP32 (the same
// values as rounding the FP64 products), so no FP64 arithmetic is spent.
template <class T>
__device__ __forceinline__ void edge_point(const Grid &G, int p, T *s, T &hT)
{
    if constexpr (sizeof(T) == sizeof(float)) {
        s[0] = G.hl[p >> 6];
        s[1] = G.hl[(p >> 3) & 7];
        s[2] = G.hl[p & 7];
        hT = G.hl[1];
    } else {
        s[0] = (double)(p >> 6) * G.h;
        s[1] = (double)((p >> 3) & 7) * G.h;
        s[2] = (double)(p & 7) * G.h;
        hT = G.h;
    }
}

// einfo[].y: lower point (local index), axis, end label, dropped (a buffer of
// the staging pass was full)
__host__ __device__ constexpr int edge_pack(int p, int axis, int lab, int dropped)
{
    return p | (axis << 9) | (lab << 11) | (dropped << 12);
}
__device__ __forceinline__ int pk_point(int pk) { return pk & 511; }
__device__ __forceinline__ int pk_axis(int pk) { return (pk >> 9) & 3; }
__device__ __forceinline__ int pk_label(int pk) { return (pk >> 11) & 1; }
__device__ __forceinline__ bool pk_dropped(int pk) { return ((pk >> 12) & 1) != 0; }

// A staged tile in HBM (its slab): this header, then the staged lists in the
// tile frame, each segment 16-byte aligned.  Written once by the staging pass
// and read (through L1/L2) by every root and selection thread of the tile.
struct alignas(16) SlabHdr {
    int na, np, nv, mol;
    double x0[3];  // tile frame origin (absolute)
    int t[3];      // tile coordinates in the run's grid
    int gt;        // batch tile
};

__host__ __device__ constexpr long long align16(long long b) { return (b + 15) & ~15LL; }

template <class T>
struct SlabLayout {
    long long atom, po, pu, vq, agid, pij, pidx, vidx, face, nbm, pslot, bytes;
    __host__ __device__ SlabLayout(int na, int np, int nv)
    {
        const long long nw = (na + 31) / 32;  // words of a set of staged atoms
        const long long P = (long long)sizeof(P4<T>);
        atom = (long long)sizeof(SlabHdr);
        po = atom + na * P;
        pu = po + np * P;
        vq = pu + np * P;
        agid = vq + nv * P;
        pij = align16(agid + 4LL * na);
        pidx = align16(pij + 8LL * np);
        vidx = align16(pidx + 4LL * np);
        face = align16(vidx + 4LL * nv);
        nbm = align16(face + na);
        pslot = align16(nbm + 4LL * na * nw);
        bytes = align16(pslot + 4LL * np);
    }
};

__device__ __forceinline__ P4<float> ldg4(const P4<float> *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return P4<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ P4<double> ldg4(const P4<double> *p)
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    return P4<double>{a.x, a.y, b.x, b.y};
}

// the staged lists of a slab (same interface as SmemAcc)
template <class T>
struct SlabAcc {
    using real = T;
    const P4<T> *a_, *po_, *pu_, *vq_;
    const int *agid_, *pidx_, *vidx_;
    const int2 *pij_;
    const uint8_t *face_;
    const unsigned *nbm_;
    const short2 *pslot_;
    int na_, np_, nv_, nw_;
    __device__ explicit SlabAcc(const unsigned char *s)
    {
        const int4 h = __ldg(reinterpret_cast<const int4 *>(s));
        na_ = h.x;
        np_ = h.y;
        nv_ = h.z;
        const SlabLayout<T> L(na_, np_, nv_);
        a_ = reinterpret_cast<const P4<T> *>(s + L.atom);
        po_ = reinterpret_cast<const P4<T> *>(s + L.po);
        pu_ = reinterpret_cast<const P4<T> *>(s + L.pu);
        vq_ = reinterpret_cast<const P4<T> *>(s + L.vq);
        agid_ = reinterpret_cast<const int *>(s + L.agid);
        pij_ = reinterpret_cast<const int2 *>(s + L.pij);
        pidx_ = reinterpret_cast<const int *>(s + L.pidx);
        vidx_ = reinterpret_cast<const int *>(s + L.vidx);
        face_ = reinterpret_cast<const uint8_t *>(s + L.face);
        nbm_ = reinterpret_cast<const unsigned *>(s + L.nbm);
        pslot_ = reinterpret_cast<const short2 *>(s + L.pslot);
        nw_ = (na_ + 31) >> 5;
    }
    __device__ int na() const { return na_; }
    __device__ int np() const { return np_; }
    __device__ int nv() const { return nv_; }
    __device__ P4<T> atom(int a) const { return ldg4(a_ + a); }
    __device__ int agid(int a) const { return __ldg(agid_ + a); }
    __device__ bool face(int a) const { return __ldg(face_ + a) != 0; }
    __device__ P4<T> po(int p) const { return ldg4(po_ + p); }
    __device__ P4<T> pu(int p) const { return ldg4(pu_ + p); }
    __device__ int2 pij(int p) const { return __ldg(pij_ + p); }
    __device__ P4<T> vq(int v) const { return ldg4(vq_ + v); }
    __device__ int pidx(int p) const { return __ldg(pidx_ + p); }
    __device__ int vidx(int v) const { return __ldg(vidx_ + v); }
    // neighbour set of staged atom a (staged atoms whose expanded spheres
    // come within 1e-3 A of meeting a's), ceil(na / 32) words
    __device__ const unsigned *nb(int a) const { return nbm_ + (size_t)a * nw_; }
    // staged slots of pair p's atoms (-1: not staged)
    __device__ short2 pslot(int p) const { return __ldg(pslot_ + p); }
    // model index of a staged piece (kind as in WCand)
    __device__ int model_index(int kind, int slot) const
    {
        return kind == 0 ? agid(slot) : (kind == 1 ? pidx(slot) : vidx(slot));
    }
};

// FP64 data of a slab's pieces from HBM, in the same tile frame (as ExactAcc)
template <class T>
struct SlabExact {
    using real = double;
    const SlabAcc<T> &S;
    const Model &M;
    double x0, y0, z0;
    float d0;  // bound of the tile frame's FP32 rounding
    __device__ SlabExact(const SlabAcc<T> &s, const Model &m, const double *o, float d)
        : S(s), M(m), x0(o[0]), y0(o[1]), z0(o[2]), d0(d) {}
    __device__ int na() const { return S.na(); }
    __device__ int np() const { return S.np(); }
    __device__ int nv() const { return S.nv(); }
    __device__ P4<double> atom(int a) const
    {
        const double4 g = M.atom[S.agid(a)];
        return P4<double>{g.x - x0, g.y - y0, g.z - z0, g.w};
    }
    __device__ int agid(int a) const { return S.agid(a); }
    __device__ bool face(int a) const { return S.face(a); }
    __device__ P4<double> po(int p) const
    {
        const double4 g = M.pair_o[S.pidx(p)];
        return P4<double>{g.x - x0, g.y - y0, g.z - z0, g.w};
    }
    __device__ P4<double> pu(int p) const
    {
        const double4 g = M.pair_u[S.pidx(p)];
        return P4<double>{g.x, g.y, g.z, 0.0};
    }
    __device__ int2 pij(int p) const { return S.pij(p); }
    __device__ P4<double> vq(int v) const
    {
        const double4 g = M.vert[S.vidx(v)];
        return P4<double>{g.x - x0, g.y - y0, g.z - z0, 0.0};
    }
    __device__ const unsigned *nb(int a) const { return S.nb(a); }
    __device__ short2 pslot(int p) const { return S.pslot(p); }
};

// Freeness of a witness on the expanded sphere of staged atom a (and, for a
// saddle witness, of staged atom b too): only the atoms whose expanded
// spheres meet a's (and b's) can cover it, so the neighbour sets decide the
// same as a test against every staged atom but a and b (free_set).  A pair
// whose atoms are not both staged is tested against every staged atom.
template <bool FILT, class Acc, class T>
__device__ __forceinline__ int free_witness(const Acc &A, T qx, T qy, T qz, int sa, int sb, int ga, int gb, T rp,
                                            T delta)
{
    int nt = 0;
    if (sa >= 0 && (gb < 0 || sb >= 0))
        return free_set<FILT>(A, qx, qy, qz, A.nb(sa), gb < 0 ? (const unsigned *)nullptr : A.nb(sb), rp, delta, nt);
    return free_pt<FILT>(A, qx, qy, qz, ga, gb, rp, delta);
}

// shared memory of the staging pass (beside the staged tile)
struct StageSmem {
    uint16_t rows[81];         // the tile's labels and the next layer's (tile_row)
    short eptr[3 * TILE_PTS];  // crossing edges of the tile (edge_pack), grouped by axis
    int cs[3 * TILE_PTS + 1];  // per edge: sphere candidates, then their offset in the tile's run
    int ct[3 * TILE_PTS + 1];  // the same for tori
    int estart[4];
    int gbase[3];  // global id of the tile's first edge per axis (all axes numbered in one run)
    int abase[3];  // its index in the axis' output
    int sh[EDGE_WARPS], sh2[EDGE_WARPS];
    long long slab;    // slab offset (16-byte units), -1 when the slab buffer is full
    long long sb, tb;  // the tile's first sphere / torus candidate, -1 when a buffer is full
    long long sb0, tb0;  // the same as reserved (also when a buffer is full)
    unsigned hmask[HMASK_WORDS];  // prefilter hits, ceil(items / 32) words per edge (when they fit), two halves a word
};

// Freeness of an FP64 saddle witness: free_witness<false>.
template <class Acc>
__device__ __forceinline__ bool exact_free(const Acc &A, const double *q, short2 sl, int2 ij, double rp)
{
    return free_witness<false>(A, q[0], q[1], q[2], (int)sl.x, (int)sl.y, ij.x, ij.y, rp, 0.0) == 1;
}

// The same answer where the staged copies are FP32: an atom whose FP32 distance
// is certain needs no FP64 one (2 d0 + 1e-6 A covers the rounding of q and of
// the atom).  One thread walks the atoms one after the other, so the latency of
// their loads is the time: four independent FP32 loads at once instead of an
// index and then an FP64 load for each (k_roots_torus_exact 116 -> 73 us on the
// packed box, 90 -> 66 us on 3,000 atoms).
__device__ __noinline__ bool exact_free(const SlabExact<float> &X, const double *q, short2 sl, int2 ij, double rp)
{
    const SlabAcc<float> &S = X.S;
    const float qx = (float)q[0], qy = (float)q[1], qz = (float)q[2], rpf = (float)rp;
    const float delta = 2.0f * X.d0 + 1e-6f;
    const bool sets = sl.x >= 0 && sl.y >= 0;
    const unsigned *m0 = sets ? S.nb(sl.x) : nullptr, *m1 = sets ? S.nb(sl.y) : nullptr;
    const int na = S.na();
    for (int w = 0; w * 32 < na; ++w) {
        unsigned bits = sets ? m0[w] & m1[w] : (na - w * 32 >= 32 ? 0xffffffffu : (1u << (na - w * 32)) - 1u);
        while (bits) {
            int k[4];
            P4<float> c[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                k[u] = bits ? (w << 5) + __ffs(bits) - 1 : -1;
                bits &= bits - 1;
                c[u] = S.atom(max(k[u], 0));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float dx = qx - c[u].x, dy = qy - c[u].y, dz = qz - c[u].z, R = c[u].w + rpf;
                const int t = lt_sq<true>(dx * dx + dy * dy + dz * dz, R * R, R, delta);
                if (k[u] < 0 || t == 0) continue;
                if (!sets) {
                    const int g = S.agid(k[u]);
                    if (g == ij.x || g == ij.y) continue;
                }
                if (t == 1) return false;
                const P4<double> e = X.atom(k[u]);
                const double ex = q[0] - e.x, ey = q[1] - e.y, ez = q[2] - e.z, R64 = e.w + rp;
                if (ex * ex + ey * ey + ez * ez < R64 * R64) return false;
            }
        }
    }
    return true;
}

// items [0, nsph) are spheres: the bits of 32-item word w that are spheres
__device__ __forceinline__ unsigned sphere_bits(int w, int nsph)
{
    const int r = nsph - 32 * w;
    return r >= 32 ? 0xffffffffu : (r <= 0 ? 0u : (1u << r) - 1u);
}

// axis, lower point (local index) and its label of crossing edge e of the tile
struct EdgeRef {
    int axis, p, lab;
};
__device__ __forceinline__ EdgeRef edge_ref(const StageSmem &E, int e)
{
    const int pk = E.eptr[e];
    return EdgeRef{pk_axis(pk), pk_point(pk), pk_label(pk)};
}

// index of the smallest key (ties: smaller index), -1 if every key is +inf
__device__ __forceinline__ int warp_argmin_key(float key, int k)
{
    float bt = key;
    int bk = (key < INFINITY) ? k : -1;
    for (int o = 16; o > 0; o >>= 1) {
        float ot = __shfl_xor_sync(0xffffffffu, bt, o);
        int ok = __shfl_xor_sync(0xffffffffu, bk, o);
        if (ok >= 0 && (bk < 0 || ot < bt || (ot == bt && ok < bk))) {
            bt = ot;
            bk = ok;
        }
    }
    return bk;
}

__device__ __forceinline__ int warp_argmin(const WCand *c, int n)
{
    const int lane = threadIdx.x & 31;
    float bt = INFINITY;
    int bk = -1;
    for (int k = lane; k < n; k += 32)
        if (c[k].t < bt) {
            bt = c[k].t;
            bk = k;
        }
    return warp_argmin_key(bt, bk);
}

// --------------------------------------------------------------------------
// torus pieces: near-branch roots of g(t) = D(t) - r_p, D the distance from
// y(t) = q0 + t e_axis to the circle (centre at the frame origin, axis u,
// radius rho).  These are the roots of the quartic whose nearest circle point
// is the witness.
// --------------------------------------------------------------------------
// D, dD/dt, the distance |w| to the circle's axis, |y|^2, z = y.u and w at t
__device__ __forceinline__ void circle_dist32(const float *q0, const float *u, float rho, int axis, float t, float &D,
                                              float &dD, float &nw, float &yy, float &z, float *w)
{
    float y0 = q0[0], y1 = q0[1], y2 = q0[2];
    if (axis == 0) y0 += t;
    else if (axis == 1) y1 += t;
    else y2 += t;
    z = y0 * u[0] + y1 * u[1] + y2 * u[2];
    yy = y0 * y0 + y1 * y1 + y2 * y2;
    w[0] = y0 - z * u[0];
    w[1] = y1 - z * u[1];
    w[2] = y2 - z * u[2];
    nw = sqrtf(fmaxf(yy - z * z, 0.0f));
    const float e = nw - rho;
    D = sqrtf(e * e + z * z);
    const float wa = axis == 0 ? w[0] : (axis == 1 ? w[1] : w[2]);
    dD = (nw > 0.0f && D > 0.0f) ? (e * wa / nw + z * u[axis]) / D : 0.0f;
}

// error bound of the FP32 D: staged positions (d0) and rounding of |y|^2 - z^2
// (relative 2^-24 per operation, amplified by |y|^2 / |w| in |w|)
__device__ __forceinline__ float circle_dist_err(float d0, float yy, float nw, float rho, float rp)
{
    return 2.0f * d0 + 4e-7f * (yy / fmaxf(nw, 1e-3f) + sqrtf(yy) + rho + rp);
}

// g along the edge from its quadratic pieces: |y|^2 = yy0 + 2 qa t + t^2 and
// z = z0 + ua t (qa, ua the edge-axis components of q0 and u)
struct LineCircle32 {
    float yy0, qa, z0, ua, rho, rp;
    __device__ __forceinline__ void eval(float t, float &g, float &dg, float &nw, float &yy) const
    {
        yy = fmaf(t, t + 2.0f * qa, yy0);
        const float z = fmaf(t, ua, z0);
        nw = sqrtf(fmaxf(yy - z * z, 0.0f));
        const float e = nw - rho;
        const float D = sqrtf(e * e + z * z);
        g = D - rp;
        const float wa = qa + t - z * ua;  // edge-axis component of w
        dg = (nw > 0.0f && D > 0.0f) ? __fdividef(e * __fdividef(wa, nw) + z * ua, D) : 0.0f;
    }
};

// Certified FP32 isolation of the roots of g on [lo, hi].  g is 1-Lipschitz
// and |g''| <= C = max(1/D, 1/|w|) (the distance to a circle has Hessian
// eigenvalues 0 and 1/D in the meridian plane and (dD/d|w|)/|w| around the
// axis; D and |w| are 1-Lipschitz too, so on a sub-interval of length l they
// stay above their smaller end value minus l/2).  On 8 sub-intervals: none
// holds a root when |g| at its ends adds up to more than its length; g' keeps
// its sign when g' has the same sign at both ends and |g'| there adds up to
// more than C l, and then the sub-interval holds one root if g changes sign,
// else none.  Each root is refined by Newton from the secant point inside its
// bracket.  Returns false when a sign or the monotonicity cannot be decided.
__device__ __noinline__ bool torus_roots32(const float *q0, const float *u, float rho, float rp, int axis, float lo,
                                           float hi, float d0, float *rt, int &nr)
{
    constexpr int K = 8;
    const float dl = (hi - lo) / (float)K;
    LineCircle32 L;
    L.yy0 = q0[0] * q0[0] + q0[1] * q0[1] + q0[2] * q0[2];
    L.qa = q0[axis];
    L.z0 = q0[0] * u[0] + q0[1] * u[1] + q0[2] * u[2];
    L.ua = u[axis];
    L.rho = rho;
    L.rp = rp;
    unsigned rootmask = 0;
    float gp = 0.0f, dgp = 0.0f, egp = 0.0f, mwp = 0.0f;
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        const float t = k == K ? hi : lo + (float)k * dl;
        float g, dg, nw, yy;
        L.eval(t, g, dg, nw, yy);
        const float eg = circle_dist_err(d0, yy, nw, rho, rp);
        const float mw = fminf(g + rp, nw);
        if (k > 0) {
            const bool sc = (gp <= 0.0f) != (g <= 0.0f);
            if (sc || fabsf(gp) + fabsf(g) <= dl + egp + eg) {
                if (fabsf(gp) <= egp || fabsf(g) <= eg) return false;
                const float low = fminf(mwp, mw) - 0.5f * dl;
                if (!(low > 1e-2f)) return false;
                if (!((dgp > 0.0f) == (dg > 0.0f) && fabsf(dgp) + fabsf(dg) > dl / low + 2e-4f)) return false;
                if (sc) rootmask |= 1u << (k - 1);
            }
        }
        gp = g;
        dgp = dg;
        egp = eg;
        mwp = mw;
    }
    nr = 0;
    while (rootmask) {
        const int k = __ffs(rootmask) - 1;
        rootmask &= rootmask - 1;
        if (nr == 4) return false;
        float a = lo + (float)k * dl, b = k + 1 == K ? hi : lo + (float)(k + 1) * dl;
        float ga, gb, dga, dgb, nwa, yya;
        L.eval(a, ga, dga, nwa, yya);
        L.eval(b, gb, dgb, nwa, yya);
        const bool neg_a = ga <= 0.0f;
        float t = a + (b - a) * __fdividef(ga, ga - gb);
        for (int itn = 0; itn < 5; ++itn) {  // Newton, bisection when it leaves the bracket
            float f, df, nw, yy;
            L.eval(t, f, df, nw, yy);
            if (f == 0.0f) break;
            if ((f <= 0.0f) == neg_a) a = t;
            else b = t;
            float tn = df != 0.0f ? t - __fdividef(f, df) : 0.5f * (a + b);
            if (!(tn > a && tn < b)) tn = 0.5f * (a + b);
            t = tn;
        }
        rt[nr++] = t;
    }
    return true;
}

// One FP64 root t64 of a torus piece: kept if it lies on the near branch in
// [0, h], its witness distance crosses r_p in the direction that leaves the
// end point's side, and its witness (nearest circle point) is free.
template <class Acc>
__device__ __noinline__ void torus_root_exact(const Acc &X, RootSink &out, int pi, const double *s64, int axis,
                                              double h, double rp, bool inside, double t64)
{
    t64 = at_end(t64, h);
    if (!(t64 >= 0.0 && t64 <= h)) return;
    const P4<double> oe = X.po(pi);
    const P4<double> ue = X.pu(pi);
    const double oo[3] = {oe.x, oe.y, oe.z}, u64[3] = {ue.x, ue.y, ue.z};
    double yd[3] = {s64[0] - oo[0], s64[1] - oo[1], s64[2] - oo[2]};
    yd[axis] += t64;
    const double Ad = yd[0] * yd[0] + yd[1] * yd[1] + yd[2] * yd[2] + oe.w * oe.w - rp * rp;
    const double zd = yd[0] * u64[0] + yd[1] * u64[1] + yd[2] * u64[2];
    double wd[3];
    const double nwd = axis_normal(yd, u64, wd);  // unit direction
    const double near2 = (nwd - oe.w) * (nwd - oe.w) + zd * zd;
    if (fabs(near2 - rp * rp) > 1e-7 * rp * rp || !(nwd > 0.0) || !(Ad >= 0.0)) return;
    const double rd = ((nwd - oe.w) * wd[axis] + zd * u64[axis]) / rp;
    const double rate = fabs(rd) <= 1e-9 ? 0.0 : rd;
    if (inside ? rate > 0.0 : rate < 0.0) return;
    const int2 ij = X.pij(pi);
    const short2 sl = X.pslot(pi);
    const double q[3] = {oo[0] + oe.w * wd[0], oo[1] + oe.w * wd[1], oo[2] + oe.w * wd[2]};
    if (exact_free(X, q, sl, ij, rp)) out.push((float)t64, 0.0f, t64);
}

// Every root of a torus piece in [0, h] (or END_TOL past an end) from the
// quartic, each decided in FP64.
template <class Acc>
__device__ __noinline__ void torus_piece_exact(const Acc &X, RootSink &out, int pi, const double *s64, int axis,
                                               double h, double rp, bool inside)
{
    const P4<double> oe = X.po(pi);
    const P4<double> ue = X.pu(pi);
    const double oo[3] = {oe.x, oe.y, oe.z}, u64[3] = {ue.x, ue.y, ue.z};
    double co[5], r64[4];
    torus_coeffs(oo, u64, oe.w, rp, s64, axis, co);
    const int n = PolyRoots<double, 4>::run(co, 0.0, h, r64);
    for (int k = 0; k < n; ++k) torus_root_exact(X, out, pi, s64, axis, h, rp, inside, r64[k]);
    // a simple root just past an end
    const double dc[4] = {co[1], 2.0 * co[2], 3.0 * co[3], 4.0};
    for (int e = 0; e < 2; ++e) {
        const double t = e == 0 ? 0.0 : h, f = horner<double, 4>(co, t), df = horner<double, 3>(dc, t);
        if (f == 0.0 || !(fabs(f) <= END_TOL * fabs(df))) continue;
        if (e == 0 ? (f > 0.0) == (df > 0.0) : (f > 0.0) != (df > 0.0))  // t - f / df lies outside
            torus_root_exact(X, out, pi, s64, axis, h, rp, inside, t);
    }
}

// Can item `it` (staged atom, vertex or pair, in that order) put an accepted
// root on the edge from s along axis (`inside`: the label at s)?
// Spheres |y - c| = rad: the segment comes within rad of c, and its far end
// (for a root where the line leaves the ball) or near end (where it enters)
// is not inside the ball.  The line must leave a van der Waals ball and enter
// a probe ball after an inside end, the other way round after an outside one;
// an atom whose expanded sphere keeps no free face has no free witness.
// Tori, D the distance to the circle along the edge, g = D - r_p: D is
// 1-Lipschitz, so |g| at the midpoint is at most h/2; and where the circle and
// its axis stay away (|g''| <= C = 1 / min(D, |w|) over the edge) |g| is at
// most |g'| h/2 + C h^2/8, and g' keeps its sign when |g'| > C h/2, which must
// be falling after an inside end, rising after an outside one.
// The test is FP32 in either form and a superset of the pieces with roots at
// any scale: every length is compared with a margin mg = 2e-3 A + 12 d0, d0 the
// bound of a staged difference's rounding, which grows with the molecule's
// lengths.  Squares are formed from components across the edge or the axis, never as
// differences of squares, so a length is off by 4 d0 at most, and g' by
// 5 d0 over the smaller of D and |w| (2e-3 A alone and differences of squares
// lost roots on balls of 1e5, and tests that were given up on edges above
// 4 A took every piece there).  (The Lipschitz test alone, and spheres by
// their distance range only, left 1.50 M sphere and 4.31 M torus candidates on
// 1.14 M edges of the 5,000-atom globule, 1.0 M and 1.6 M now.)
struct CandItem {  // one staged piece, held by a lane over many edges
    float x, y, z, r;  // sphere: centre, radius; circle: centre, rho
    float ux, uy, uz;  // circle: axis
    int kind;          // 0 van der Waals sphere, 1 probe sphere, 2 circle, -1 none
};

template <class T, class CP>
__device__ __forceinline__ CandItem cand_item(const TileS<T, CP> &S, int it, int nitem, float rp)
{
    const int na = S.na, nsph = S.na + S.nv;
    CandItem c{0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, -1};
    if (it >= nitem) return c;
    const P4<T> o = it < na ? S.atom[it] : (it < nsph ? S.vq[it - na] : S.po[it - nsph]);
    c.x = (float)o.x;
    c.y = (float)o.y;
    c.z = (float)o.z;
    c.r = it < na || it >= nsph ? (float)o.w : rp;
    c.kind = it < na ? (S.aface[it] != 0 ? 0 : -1) : (it < nsph ? 1 : 2);
    if (it >= nsph) {
        const P4<T> u = S.pu[it - nsph];
        c.ux = (float)u.x;
        c.uy = (float)u.y;
        c.uz = (float)u.z;
    }
    return c;
}

// m: the edge's middle, half: half its length
__device__ __forceinline__ bool cand_test(const CandItem &c, const float *m, int axis, bool inside, float half,
                                          float rp, float mg)
{
    const float d0 = m[0] - c.x, d1 = m[1] - c.y, d2 = m[2] - c.z;
    if (c.kind < 2) {
        const float a = axis == 0 ? d0 : (axis == 1 ? d1 : d2), p = axis == 0 ? d1 : d0, q = axis == 2 ? d1 : d2;
        const float pp = p * p + q * q;
        const float vn = a + fminf(fmaxf(-a, -half), half);         // nearest point of the segment
        const float ve = (c.kind == 0) == inside ? a + half : a - half;
        const float rhi = c.r + mg, rlo = fmaxf(c.r - mg, 0.0f);
        return c.kind >= 0 && pp + vn * vn <= rhi * rhi && pp + ve * ve >= rlo * rlo;
    }
    const float zc = d0 * c.ux + d1 * c.uy + d2 * c.uz;
    const float w0 = d0 - zc * c.ux, w1 = d1 - zc * c.uy, w2 = d2 - zc * c.uz;
    const float nw = sqrtf(w0 * w0 + w1 * w1 + w2 * w2), e1 = nw - c.r;
    const float D = sqrtf(e1 * e1 + zc * zc), gm = fabsf(D - rp), H = half + mg;
    if (gm > H) return false;
    const float low = fminf(D, nw) - H;
    if (low < 50.0f * mg) return true;
    const float ua = axis == 0 ? c.ux : (axis == 1 ? c.uy : c.uz), wa = axis == 0 ? w0 : (axis == 1 ? w1 : w2);
    const float bend = __fdividef(H, low);  // C h/2: g' moves by at most this over the edge
    const float dg = __fdividef(e1 * __fdividef(wa, nw) + zc * ua, D);
    if (gm > fabsf(dg) * H + 0.5f * bend * H + mg) return false;
    return !((inside ? dg : -dg) > bend + 1e-2f);
}

// Prefilter of the lane's edge (middle m, axis, label) against 16 staged
// items from i0 on, the same items on every lane: bit b for item i0 + b.  The
// warp's edges are neighbours, so an item is mostly near to all of them or to
// none and the lanes stay together (lanes over items, a warp per edge, ran the
// sphere and the torus test for every word that held both: 24,000 cycles a tile
// of 75 edges and 60 items on the globule, half of the staging pass with the
// writing of the pairs).  Whole warp.
template <class T, class CP>
__device__ __forceinline__ unsigned cand_bits(const TileS<T, CP> &S, int i0, int nitem, const float *m, int axis,
                                              bool inside, float half, float rp, float mg)
{
    unsigned bits = 0u;
    const int n = min(16, nitem - i0);
    CandItem mine;
    if constexpr (sizeof(T) == sizeof(double)) mine = cand_item<T, CP>(S, i0 + (threadIdx.x & 15), nitem, rp);
    for (int b = 0; b < n; ++b) {
        CandItem c;
        if constexpr (sizeof(T) == sizeof(double)) {  // converted once, by a lane each
            c.x = __shfl_sync(0xffffffffu, mine.x, b);
            c.y = __shfl_sync(0xffffffffu, mine.y, b);
            c.z = __shfl_sync(0xffffffffu, mine.z, b);
            c.r = __shfl_sync(0xffffffffu, mine.r, b);
            c.ux = __shfl_sync(0xffffffffu, mine.ux, b);
            c.uy = __shfl_sync(0xffffffffu, mine.uy, b);
            c.uz = __shfl_sync(0xffffffffu, mine.uz, b);
            c.kind = __shfl_sync(0xffffffffu, mine.kind, b);
        } else {
            c = cand_item<T, CP>(S, i0 + b, nitem, rp);
        }
        if (c.kind >= 0 && cand_test(c, m, axis, inside, half, rp, mg)) bits |= 1u << b;
    }
    return bits;
}

// Roots of one (edge, piece) candidate that can be the surface on that edge:
// every root in [0, h] of the piece whose witness distance crosses r_p in the
// direction that leaves the end point's side (falling from an inside end,
// rising from an outside end) and whose witness is free.  FP32 roots carry an
// error bound; a decision the bound cannot make goes to FP64.  A: the staged
// lists (tile frame), X: the same pieces in FP64; s64 the edge's lower point
// in the tile frame.
//
// Spheres (item < na: van der Waals sphere of staged atom `item`, convex,
// witness = projection on the expanded sphere; else the probe sphere of staged
// triple point item - na, concave, witness = the triple point).
template <class T, bool FILT, class AccT, class AccX>
__device__ void sphere_roots(const AccT &A, const AccX &X, int item, const T *s, const double *s64, int axis,
                             bool inside, T hT, T rpT, double h, double rp, T d0, RootSink &out)
{
    const int na = A.na();
    const T past = FILT ? T(1e-4) : T(END_TOL);
    const T lo = -past, hi = hT + past;
    const T tmax = T(1e-3);  // FP32 root error beyond which FP64 decides (grazing pieces)
    const double NaN = __longlong_as_double(0x7ff8000000000000LL);
    const bool vdw = item < na;
    const int slot = vdw ? item : item - na;
    const P4<T> c = vdw ? A.atom(slot) : A.vq(slot);
    const T rad = vdw ? c.w : rpT;
    const T d[3] = {s[0] - c.x, s[1] - c.y, s[2] - c.z};
    const T dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const T b = d[axis], disc = b * b - (dd - rad * rad);
    const T co32[3] = {dd - rad * rad, T(2) * b, T(1)};
    T rt32[2];
    int nr = PolyRoots<T, 2>::run(co32, lo, hi, rt32);
    if (FILT && nr == 0 && disc < T(2e-3)) {  // grazing: let FP64 decide
        rt32[0] = -b;
        nr = (-b >= lo && -b <= hi) ? 1 : 0;
    }
    for (int k = 0; k < nr; ++k) {
        T t = FILT ? rt32[k] : (T)at_end((double)rt32[k], h);
        T vA = d[axis] + t;  // +-sqrt(disc) at a root: the rate of |y - c|
        T terr = T(0);
        if (FILT) {
            const T derr = T(2) * (fabs(b) + sqrt(dd)) * d0 + T(2e-6) * (dd + rad * rad);
            terr = d0 + derr / (T(2) * fmax(fabs(vA), T(1e-20)));
        }
        double t64 = NaN;
        const bool exact = FILT && (terr > tmax || t < terr + T(1e-6) || t > hT - terr - T(1e-6));
        if (exact) {
            const P4<double> ce = vdw ? X.atom(slot) : X.vq(slot);
            const double cc[3] = {ce.x, ce.y, ce.z};
            const double r64 = vdw ? ce.w : rp;
            t64 = at_end(exact_root_sphere(cc, r64, s64, axis, (double)t), h);
            double dv[3] = {s64[0] - cc[0], s64[1] - cc[1], s64[2] - cc[2]};
            dv[axis] += t64;
            const double f = dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2] - r64 * r64;
            if (!(t64 >= 0.0 && t64 <= h) || fabs(f) > 1e-9 * r64) continue;
            vA = (T)dv[axis];
            if (fabs(dv[axis]) <= 1e-9 * r64) vA = T(0);  // tangent: either way
            t = (T)t64;
            terr = T(0);
        }
        // witness distance: R - |y - c| (convex) falls iff vA > 0; |y - v| (concave) rises iff vA > 0
        const bool rises = vdw ? (vA < T(0)) : (vA > T(0));
        const bool falls = vdw ? (vA > T(0)) : (vA < T(0));
        if (inside ? rises : falls) continue;
        if (vdw) {
            T v32[3] = {d[0], d[1], d[2]};
            v32[axis] += t;
            const T nvv = sqrt(v32[0] * v32[0] + v32[1] * v32[1] + v32[2] * v32[2]);
            const T Rr = c.w + rpT;
            const T sc = Rr / nvv;
            int f = -1;
            if (FILT) {
                const T delta = d0 + terr * (T(1) + sc) + T(2e-6);
                f = free_witness<true>(A, c.x + sc * v32[0], c.y + sc * v32[1], c.z + sc * v32[2], slot, -1,
                                       A.agid(slot), -1, rpT, delta);
            }
            if (f < 0) {
                const P4<double> ce = X.atom(slot);
                const double cc[3] = {ce.x, ce.y, ce.z};
                if (t64 != t64) t64 = exact_root_sphere(cc, ce.w, s64, axis, (double)t);
                double v[3] = {s64[0] - cc[0], s64[1] - cc[1], s64[2] - cc[2]};
                v[axis] += t64;
                const double nv64 = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
                const double R64 = ce.w + rp;
                f = free_witness<false>(X, cc[0] + R64 * v[0] / nv64, cc[1] + R64 * v[1] / nv64,
                                        cc[2] + R64 * v[2] / nv64, slot, -1, A.agid(slot), -1, rp, 0.0);
            }
            if (f != 1) continue;
        }
        out.push((float)t, (float)terr, t64);
    }
}

// Tori (saddle pieces) around the free-arc circle of staged pair pi: roots on
// the near branch, isolated in FP32 (certified) with the quartic on its
// derivative chain and FP64 where that cannot decide.
template <class AccT, class AccX>
__device__ void torus_roots(const AccT &A, const AccX &X, int pi, const double *s64, int axis, bool inside, double h,
                            double rp, float d0, RootSink &out)
{
    const float s[3] = {(float)s64[0], (float)s64[1], (float)s64[2]};
    const float hT = (float)h, rpT = (float)rp;
    const float lo = -1e-4f, hi = hT + 1e-4f;
    const float tmax = 1e-3f;
    const double NaN = __longlong_as_double(0x7ff8000000000000LL);
    const P4<float> o = A.po(pi);
    const P4<float> u = A.pu(pi);
    const float q0[3] = {s[0] - o.x, s[1] - o.y, s[2] - o.z};
    const float uu[3] = {u.x, u.y, u.z};
    float rt[4];
    int nr = 0;
    if (!torus_roots32(q0, uu, o.w, rpT, axis, lo, hi, d0, rt, nr)) {
        // sampling undecided (near-tangent line, or close to the circle's axis): the
        // quartic's roots on the derivative chain
        const float P = q0[0] * q0[0] + q0[1] * q0[1] + q0[2] * q0[2];
        const float z0 = q0[0] * uu[0] + q0[1] * uu[1] + q0[2] * uu[2];
        const float pe = q0[axis], eu = uu[axis];
        const float K = P + o.w * o.w - rpT * rpT, r2 = o.w * o.w;
        const float co32[5] = {K * K - 4.0f * r2 * (P - z0 * z0), 4.0f * pe * K - 8.0f * r2 * (pe - z0 * eu),
                               4.0f * pe * pe + 2.0f * K - 4.0f * r2 * (1.0f - eu * eu), 4.0f * pe, 1.0f};
        float rq[4];
        const int nq = PolyRoots<float, 4>::run(co32, lo, hi, rq);
        nr = 0;
        for (int k = 0; k < nq; ++k) {
            float D, dD, nw, yy, zy, wv[3];
            circle_dist32(q0, uu, o.w, axis, rq[k], D, dD, nw, yy, zy, wv);
            // near branch: A = |y|^2 + rho^2 - r_p^2 >= 0; undecided signs go to FP64
            const float Ay = yy + r2 - rpT * rpT;
            if (fabsf(Ay) < 1e-3f * (yy + r2 + rpT * rpT)) nr = -1;
            else if (Ay > 0.0f && nr >= 0) rt[nr++] = rq[k];
        }
        if (nr < 0) {
            torus_piece_exact(X, out, pi, s64, axis, h, rp, inside);
            return;
        }
    }
    const int2 ij = A.pij(pi);
    const short2 sl = A.pslot(pi);
    for (int k = 0; k < nr; ++k) {
        const float t = rt[k];
        float D, rate, nw, yy, zy, wv[3];
        circle_dist32(q0, uu, o.w, axis, t, D, rate, nw, yy, zy, wv);
        // root error: residual plus rounding of g over |g'| (g' varies little within terr)
        const float terr =
            (fabsf(D - rpT) + circle_dist_err(d0, yy, nw, o.w, rpT)) / fmax(fabs(rate), 1e-20f) + d0;
        if (terr > tmax || t < terr + 1e-6f || t > hT - terr - 1e-6f || fabs(rate) < 1e-3f ||
            nw < 1e-3f) {  // grazing or at an end point: the FP64 root decides
            const P4<double> oe = X.po(pi);
            const P4<double> ue = X.pu(pi);
            const double oo[3] = {oe.x, oe.y, oe.z}, u64[3] = {ue.x, ue.y, ue.z};
            const double t64 = exact_root_torus(oo, u64, oe.w, rp, s64, axis, (double)t);
            torus_root_exact(X, out, pi, s64, axis, h, rp, inside, t64);
            continue;
        }
        if (inside ? rate > 0.0f : rate < 0.0f) continue;
        const float kk = o.w / nw;
        const float delta = d0 + terr * (1.0f + 2.0f * o.w / nw) + 2e-6f;
        const int f = free_witness<true>(A, o.x + kk * wv[0], o.y + kk * wv[1], o.z + kk * wv[2], (int)sl.x,
                                         (int)sl.y, ij.x, ij.y, rpT, delta);
        if (f == 1) {
            out.push(t, terr, NaN);
        } else if (f < 0) {
            const P4<double> oe = X.po(pi);
            const P4<double> ue = X.pu(pi);
            const double oo[3] = {oe.x, oe.y, oe.z}, u64[3] = {ue.x, ue.y, ue.z};
            const double t64 = exact_root_torus(oo, u64, oe.w, rp, s64, axis, (double)t);
            torus_root_exact(X, out, pi, s64, axis, h, rp, inside, t64);
        }
    }
}

// First root of one crossing edge from its candidates c[0, n) (whole warp; c
// in shared memory, updated in place).  Returns 0 with the chosen piece (kind,
// staged slot) and its root, 1 when no root is found, 2 when the candidates
// overflowed the buffer (the first WCAND are used).
template <class T, bool FILT, class AccT, class AccX>
__device__ int warp_select(const AccT &A, const AccX &X, WCand *c, int n, const T *s, const double *s64, int axis,
                           bool inside, float hf, T rpT, double rp, T d0, float &t_out, int &kind_out, int &slot_out)
{
    const int lane = threadIdx.x & 31;
    const float tie = 1e-6f * hf;  // FP32 rounding of a root
    int status = n > WCAND ? 2 : 0;
    if (n > WCAND) n = WCAND;
    int pick = -1;
    for (int iter = 0; iter <= n; ++iter) {
        int k = warp_argmin(c, n);
        if (k < 0) break;
        // candidates that the FP32 bounds cannot order against k: settle with FP64 roots
        const float tk = c[k].t, ek = c[k].err;
        bool tied = false;
        for (int j = lane; j < n; j += 32)
            if (j != k && c[j].t < INFINITY && c[j].t - tk <= c[j].err + ek + tie) tied = true;
        if (__any_sync(0xffffffffu, tied)) {
            for (int j = lane; j < n; j += 32)
                if (c[j].t < INFINITY && c[j].t - tk <= c[j].err + ek + tie && c[j].t64 != c[j].t64)
                    c[j].t64 = staged_exact_root(X, c[j].kind, c[j].id, s64, axis, rp, (double)c[j].t);
            __syncwarp();
            double bt = INFINITY;
            int bk = -1;
            for (int j = lane; j < n; j += 32)
                if (c[j].t < INFINITY && c[j].t - tk <= c[j].err + ek + tie && c[j].t64 < bt) {
                    bt = c[j].t64;
                    bk = j;
                }
            for (int o = 16; o > 0; o >>= 1) {
                double ot = __shfl_xor_sync(0xffffffffu, bt, o);
                int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                if (ok >= 0 && (bk < 0 || ot < bt || (ot == bt && ok < bk))) {
                    bt = ot;
                    bk = ok;
                }
            }
            k = bk;
        }
        if (inside) {
            pick = k;
            break;
        }
        // outside end point: the root must not be strictly outside M.  The
        // surface crossing is always a candidate (the nearest free point at
        // it is a piece's free witness) and every candidate before it lies
        // strictly outside, so the last candidate left needs no test.
        bool others = false;
        for (int j = lane; j < n; j += 32)
            if (j != k && c[j].t < INFINITY) others = true;
        if (!__any_sync(0xffffffffu, others)) {
            pick = k;
            break;
        }
        int r;
        unsigned um_prop = 0u, um_vert = 0u;
        if (FILT) {
            // FP32 position: the FP32 root and its bound, or the exact root
            // rounded (its rounding and that of the sum within 2e-7 A)
            const bool ex = c[k].t64 == c[k].t64;
            T y0 = s[0], y1 = s[1], y2 = s[2];
            T tt = ex ? (T)c[k].t64 : (T)c[k].t;
            if (axis == 0) y0 += tt;
            else if (axis == 1) y1 += tt;
            else y2 += tt;
            const T dk = d0 + (ex ? T(2e-7) : (T)c[k].err);
            // First the witnesses of the other remaining candidates' pieces at
            // y_k: the crossing is a later candidate, whose witness at y_k is
            // usually free and closer than r_p (then y_k is strictly outside M).
            // Only a certain answer counts; otherwise the full search decides.
            T qx = T(0), qy = T(0), qz = T(0), dq = T(0);
            int e0 = -1, e1 = -1, tw = 0;
            bool vnear = false;
            if (lane < n && lane != k && c[lane].t < INFINITY &&
                !(c[lane].kind == c[k].kind && c[lane].id == c[k].id)) {
                const int id = c[lane].id;
                if (c[lane].kind == 0) {
                    tw = face_proposal<true>(A, id, y0, y1, y2, rpT, rpT, dk, qx, qy, qz, dq, e0, e1);
                } else if (c[lane].kind == 1) {
                    tw = saddle_proposal<true>(A, id, y0, y1, y2, rpT, rpT, dk, qx, qy, qz, dq, e0, e1);
                } else {  // a free triple point closer than r_p
                    const P4<T> v = A.vq(id);
                    const T dx = y0 - v.x, dy = y1 - v.y, dz = y2 - v.z;
                    vnear = lt_sq<true>(dx * dx + dy * dy + dz * dz, rpT * rpT, rpT, dk) == 1;
                }
            }
            bool und = false, mine = false;
            if (__any_sync(0xffffffffu, vnear) ||
                warp_test_proposals<true>(A, __ballot_sync(0xffffffffu, tw == 1), tw, qx, qy, qz, dq, e0, e1, rpT,
                                          dk, und, mine) == 1)
                r = 1;
            else
                r = warp_witness<true>(A, y0, y1, y2, rpT, rpT, dk, c[k].kind, c[k].id, um_prop, um_vert);
        } else {
            r = -2;
        }
        if (r < 0) {  // FP64 at the exact root: the undecided items only, or the whole search
            double t64 = c[k].t64;
            if (t64 != t64) t64 = staged_exact_root(X, c[k].kind, c[k].id, s64, axis, rp, (double)c[k].t);
            double y[3] = {s64[0], s64[1], s64[2]};
            y[axis] += t64;
            if (r == -1)
                r = warp_witness_retest(X, y[0], y[1], y[2], rp, rp - 1e-11, um_prop, um_vert);
            else
                r = warp_witness<false>(X, y[0], y[1], y[2], rp, rp - 1e-11, 0.0, -1, -1, um_prop, um_vert);
        }
        if (r == 0) {
            pick = k;
            break;
        }
        __syncwarp();
        if (lane == 0) c[k].t = INFINITY;  // strictly outside M: not the root
        __syncwarp();
    }
    if (pick < 0) return 1;
    t_out = c[pick].t64 == c[pick].t64 ? (float)c[pick].t64 : c[pick].t;
    kind_out = c[pick].kind;
    slot_out = c[pick].id;
    return status;
}

// Per tile and axis: crossing edges (end labels differ) and inside edges (both
// ends inside) leaving the tile's points in + direction, and the tile's inside
// points.  One warp per tile.  Bound by the label reads: a row of 8 + 1 labels
// is read as three aligned words (byte by byte where those would pass the
// molecule's end) and kept as 9 bits, bit 15 set for a row on the grid; the
// counts are then popcounts of rows against their neighbours.  Byte loads per
// point and axis took 153 us on 38 M points (250 GB/s) and 939 us on 198 M; 45 and 243 us now.
constexpr int COUNT_WARPS = 8;

__global__ void __launch_bounds__(COUNT_WARPS * 32) k_edge_count(Batch B, const int8_t *__restrict__ labels_all,
                                                                int *__restrict__ tile_edges,
                                                                int *__restrict__ tile_inside,
                                                                int *__restrict__ etiles)
{
    __shared__ uint16_t rows[COUNT_WARPS][81];
    const int lane = threadIdx.x & 31;
    uint16_t *row = rows[threadIdx.x >> 5];
    const long long nt = B.n_tiles;
    const long long nw = (long long)gridDim.x * COUNT_WARPS;
    for (long long gt = (long long)blockIdx.x * COUNT_WARPS + (threadIdx.x >> 5); gt < nt; gt += nw) {
        const Grid &G = B.grid[mol_of_tile(B, gt)];
        const long long d2 = G.dims[2];
        int t[3];
        tile_coords(G, gt - G.tile0, t);
        const long long gk = (long long)TILE * t[2];
        tile_rows(G, labels_all, t, row);
        // (points past the grid hold the next row's labels: masked by the row lengths)
        const int n_on = (int)min(9LL, d2 - gk), n_own = (int)max(0LL, min(8LL, G.own[2] - gk));
        const unsigned own = (1u << n_own) - 1u, ownz = own & ((1u << (n_on - 1)) - 1u);
        unsigned c[3] = {0u, 0u, 0u}, npin = 0u;  // crossing | inside edges << 16
        for (int q = 0; q < 2; ++q) {
            const int i = (2 * lane + q) >> 3, j = (2 * lane + q) & 7, r = 9 * i + j;
            if ((long long)TILE * t[0] + i >= G.own[0] || (long long)TILE * t[1] + j >= G.own[1]) continue;
            const unsigned m = row[r], x = row[r + 9], y = row[r + 1], z = (m & 0x1ffu) >> 1;
            const unsigned ox = (x & 0x8000u) ? own : 0u, oy = (y & 0x8000u) ? own : 0u;
            c[0] += __popc((m ^ x) & ox) | (__popc(m & x & ox) << 16);
            c[1] += __popc((m ^ y) & oy) | (__popc(m & y & oy) << 16);
            c[2] += __popc((m ^ z) & ownz) | (__popc(m & z & ownz) << 16);
            npin += __popc(m & own);
        }
        for (int a = 0; a < 3; ++a) c[a] = __reduce_add_sync(0xffffffffu, c[a]);
        npin = __reduce_add_sync(0xffffffffu, npin);
        if (lane < 3) {
            const unsigned v = lane == 0 ? c[0] : (lane == 1 ? c[1] : c[2]);
            tile_edges[lane * nt + gt] = (int)(v & 0xffffu);
            tile_inside[lane * nt + gt] = (int)(v >> 16);
        } else if (lane == 3) {
            tile_inside[3 * nt + gt] = (int)npin;
        } else if (lane == 4 && ((c[0] | c[1] | c[2]) & 0xffffu)) {
            etiles[1 + atomicAdd(&etiles[0], 1)] = (int)gt;  // the staging pass' tiles, any order
        }
        __syncwarp();
    }
}

// per axis, the first crossing edge of every molecule in the axis' output
// (medge[a * (n_mol + 1) + m]; m = n_mol gives the axis total)
__global__ void k_mol_edges(Batch B, const int *__restrict__ edge_start, long long *__restrict__ medge)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 3 * (B.n_mol + 1)) return;
    const int a = k / (B.n_mol + 1), m = k % (B.n_mol + 1);
    const long long nt = B.n_tiles;
    medge[k] = (long long)edge_start[a * nt + B.tile_off[m]] - edge_start[a * nt];
}

__device__ __forceinline__ int block_excl_scan_e(int v, int *sh, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    int base = 0, tot = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
        if (k < wid) base += sh[k];
        tot += sh[k];
    }
    __syncthreads();
    *total = tot;
    return base + inc - v;
}

template <class T, class CP>
__host__ __device__ constexpr size_t edge_tile_bytes()  // rounded to 256: aligned slices in global memory
{
    return (sizeof(TileS<T, CP>) + 255) & ~(size_t)255;
}

// exclusive prefix sums of v[0..n) and w[0..n) in place (whole block), the
// totals at v[n] and w[n]; each thread sums a contiguous run of entries
__device__ __forceinline__ void block_scan_runs(int *v, int *w, int n, int *sh, int *sh2)
{
    const int per = (n + EDGE_THREADS - 1) / EDGE_THREADS;
    const int b = threadIdx.x * per, e = min(n, b + per);
    int sv = 0, sw = 0;
    for (int k = b; k < e; ++k) {
        sv += v[k];
        sw += w[k];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int iv = sv, iw = sw;
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, iv, o);
        const int c = __shfl_up_sync(0xffffffffu, iw, o);
        if (lane >= o) {
            iv += a;
            iw += c;
        }
    }
    if (lane == 31) {
        sh[wid] = iv;
        sh2[wid] = iw;
    }
    __syncthreads();
    int bv = 0, bw = 0, tv = 0, tw = 0;
    for (int k = 0; k < EDGE_WARPS; ++k) {
        if (k < wid) {
            bv += sh[k];
            bw += sh2[k];
        }
        tv += sh[k];
        tw += sh2[k];
    }
    int rv = bv + iv - sv, rw = bw + iw - sw;
    for (int k = b; k < e; ++k) {
        const int a = v[k], c = w[k];
        v[k] = rv;
        w[k] = rw;
        rv += a;
        rw += c;
    }
    if (threadIdx.x == 0) {
        v[n] = tv;
        w[n] = tw;
    }
    __syncthreads();
}

// 1. Staging pass.  Persistent CTAs take tiles from the work queue, which holds
// the tiles with crossing edges only (a pop and a look at the counts of every
// tile cost 0.25 ms on 76,516 tiles, of which 16,000 have any).  Per tile: the
// pieces are staged (CP = CapMid: in shared memory,
// a tile that overflows it goes to ovf; CP = CapBig (BIG): the tiles listed in
// ovf, staged in this CTA's slice of the global scratch `big`, lists cut at
// capacity with the error bit set), the crossing edges listed per axis in
// point order, and written to HBM: the staged lists (the tile's slab), per
// edge its output point index and its record (einfo, ecnt), and the (edge,
// piece) pairs that pass the prefilter, spheres and tori in separate lists,
// each edge's run in item order.  A buffer that is full drops the tile's
// edges (flagged); the counters still add up what was needed.
template <class T, bool FILT, class CP, bool BIG>
__global__ void __launch_bounds__(EDGE_THREADS) k_edge_stage(Model M, Batch B, TileSched Q,
                                                             const int8_t *__restrict__ labels_all,
                                                             const int *__restrict__ edge_start, EdgeOut out,
                                                             int *__restrict__ err, int *__restrict__ ovf,
                                                             unsigned char *__restrict__ big, RootWork W)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileS<T, CP> &S = *reinterpret_cast<TileS<T, CP> *>(BIG ? big + (size_t)blockIdx.x * edge_tile_bytes<T, CP>()
                                                             : smem_raw);
    StageSmem &E = *reinterpret_cast<StageSmem *>(BIG ? smem_raw : smem_raw + edge_tile_bytes<T, CP>());
    __shared__ long long q_base;
    __shared__ Grid sG;
    const long long nt = B.n_tiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T rpT = (T)M.rp;
    long long iter = 0;
    const long long npos = sched_count(Q, nt);
    for (;;) {
      const long long base = next_tiles(Q, iter, &q_base);
      if (base >= npos) break;
      const long long bend = min(base + (long long)Q.per, npos);
      for (long long pos = base; pos < bend; ++pos) {
        const long long gt = sched_tile(Q, pos);
        const int mol = mol_of_tile(B, gt);
        load_grid(B, mol, sG);
        const Grid &G = sG;
        const long long tile = gt - G.tile0;
        const int8_t *__restrict__ labels = labels_all + G.lab0;
        const long long st1 = G.dims[2], st0 = G.dims[1] * G.dims[2];
        const long long fst1 = G.full[2], fst0 = G.full[1] * G.full[2];  // strides of the output indices
        double x0[3];
        stage_tile<T>(M, G, mol, tile, S, x0);
        if (!BIG && (S.flags & ERR_CAP_ANY)) {  // uniform: set before stage_tile's last barrier
            if (threadIdx.x == 0) {  // to the global-memory tier (ovf: run total, stage count, tiles)
                atomicAdd(&ovf[0], 1);
                const int k = atomicAdd(&ovf[1], 1);
                ovf[2 + k] = (int)gt;
            }
            __syncthreads();
            continue;
        }
        if (threadIdx.x == 0 && S.flags) atomicOr(err, S.flags);
        int t[3];
        tile_coords(G, tile, t);
        if (threadIdx.x < 81) E.rows[threadIdx.x] = tile_row(G, labels_all, t, threadIdx.x);
        if (threadIdx.x >= 96 && threadIdx.x < 99) {
            const int a = threadIdx.x - 96;
            E.gbase[a] = edge_start[a * nt + gt];
            E.abase[a] = E.gbase[a] - edge_start[a * nt];
        }
        __syncthreads();
        // the tile's crossing edges, axis by axis, in point order: one thread per
        // axis and row of 8 points, one scan over all of them
        {
            static_assert(EDGE_THREADS >= 192, "a thread per axis and row");
            const int a = threadIdx.x >> 6, row = threadIdx.x & 63, i = row >> 3, j = row & 7, r = 9 * i + j;
            unsigned m = 0u, cross = 0u;
            if (a < 3 && TILE * t[0] + i < G.own[0] && TILE * t[1] + j < G.own[1]) {
                const long long gk = (long long)TILE * t[2];
                const int n_on = (int)min(9LL, G.dims[2] - gk), n_own = (int)max(0LL, min(8LL, G.own[2] - gk));
                unsigned on = (1u << n_own) - 1u;
                m = E.rows[r];
                const unsigned x = a == 0 ? E.rows[r + 9] : (a == 1 ? E.rows[r + 1] : (m >> 1) | 0x8000u);
                if (a == 2) on &= (1u << (n_on - 1)) - 1u;
                cross = (x & 0x8000u) ? (m ^ x) & on : 0u;
            }
            int tot;
            int rank = block_excl_scan_e(__popc(cross), E.sh, &tot);
            if (row == 0 && a < 3) E.estart[a] = rank;
            if (threadIdx.x == 0) E.estart[3] = tot;
            for (; cross; cross &= cross - 1) {
                const int k = __ffs(cross) - 1;
                E.eptr[rank++] = (short)edge_pack(8 * row + k, a, (m >> k) & 1, 0);
            }
            __syncthreads();
        }
        const int ne = E.estart[3];
        const int na = S.na, np = S.np, nv = S.nv, nsph = na + nv, nitem = nsph + np;
        if (threadIdx.x == 0) {  // the tile's slab
            const unsigned long long bytes = (unsigned long long)SlabLayout<T>(na, np, nv).bytes;
            const unsigned long long off = atomicAdd(W.ctr, bytes);
            E.slab = off + bytes <= (unsigned long long)W.cap_slab ? (long long)(off >> 4) : -1LL;
        }
        // output point index of every edge (full grid)
        for (int e = threadIdx.x; e < ne; e += EDGE_THREADS) {
            const EdgeRef R = edge_ref(E, e);
            const int li = R.p >> 6, lj = (R.p >> 3) & 7, lk = R.p & 7;
            out.idx[R.axis][E.abase[R.axis] + (e - E.estart[R.axis])] =
                (long long)(TILE * (t[0] + G.toff[0]) + li) * fst0 + (long long)(TILE * (t[1] + G.toff[1]) + lj) * fst1 +
                (TILE * (t[2] + G.toff[2]) + lk);
        }
        // (edge, item) pairs that pass the prefilter, counted: a warp takes 32
        // edges and 16 items at a time; the hit masks kept when they fit
        const int nwd = (nitem + 31) >> 5, ngrp = (ne + 31) >> 5;
        const bool keep = (long long)ne * nwd <= HMASK_WORDS;
        const float rpf = (float)M.rp;
        uint16_t *half = reinterpret_cast<uint16_t *>(E.hmask);
        auto test16 = [&](int e, int i0) -> unsigned {  // whole warp, one edge per lane
            const EdgeRef R = edge_ref(E, e < ne ? e : 0);
            float s[3], hs;
            edge_point<float>(G, R.p, s, hs);
            const float half = 0.5f * hs;
            for (int a = 0; a < 3; ++a) s[a] += a == R.axis ? half : 0.0f;
            const unsigned m = cand_bits<T, CP>(S, i0, nitem, s, R.axis, R.lab == LABEL_IN, half, rpf, G.mg);
            return e < ne ? m : 0u;
        };
        auto word = [&](int e, int w) -> unsigned {  // the hits of edge e among items 32 w ..
            return keep ? (e < ne ? E.hmask[e * nwd + w] : 0u) : test16(e, 32 * w) | (test16(e, 32 * w + 16) << 16);
        };
        if (keep) {
            for (int k = warp; k < ngrp * 2 * nwd; k += EDGE_WARPS) {
                const int hw = k / ngrp, e = 32 * (k - hw * ngrp) + lane;
                const unsigned m = test16(e, 16 * hw);
                if (e < ne) half[2 * nwd * e + hw] = (uint16_t)m;
            }
            __syncthreads();
        }
        for (int e0 = 32 * warp; e0 < ne; e0 += EDGE_THREADS) {
            const int e = e0 + lane;
            int cs = 0, ct = 0;
            for (int w = 0; w < nwd; ++w) {
                const unsigned m = word(e, w), sm = sphere_bits(w, nsph);
                cs += __popc(m & sm);
                ct += __popc(m & ~sm);
            }
            if (e < ne) {
                E.cs[e] = cs;
                E.ct[e] = ct;
            }
        }
        __syncthreads();
        block_scan_runs(E.cs, E.ct, ne, E.sh, E.sh2);
        if (threadIdx.x == 0) {
            const unsigned long long ns = (unsigned long long)E.cs[ne], nq = (unsigned long long)E.ct[ne];
            const unsigned long long sb = atomicAdd(W.ctr + 1, ns);
            const unsigned long long tb = atomicAdd(W.ctr + 2, nq);
            const bool ok = E.slab >= 0 && sb + ns <= (unsigned long long)W.cap_sph &&
                            tb + nq <= (unsigned long long)W.cap_tor;
            E.sb = ok ? (long long)sb : -1LL;
            E.tb = ok ? (long long)tb : -1LL;
            E.sb0 = (long long)sb;
            E.tb0 = (long long)tb;
        }
        __syncthreads();
        const bool ok = E.sb >= 0;
        if (ok) {  // the slab: header and staged lists
            unsigned char *sl = W.slab + ((size_t)E.slab << 4);
            const SlabLayout<T> L(na, np, nv);
            if (threadIdx.x == 0) {
                SlabHdr hd;
                hd.na = na;
                hd.np = np;
                hd.nv = nv;
                hd.mol = mol;
                for (int a = 0; a < 3; ++a) {
                    hd.x0[a] = x0[a];
                    hd.t[a] = t[a];
                }
                hd.gt = (int)gt;
                *reinterpret_cast<SlabHdr *>(sl) = hd;
            }
            P4<T> *pa = reinterpret_cast<P4<T> *>(sl + L.atom);
            P4<T> *po = reinterpret_cast<P4<T> *>(sl + L.po);
            P4<T> *pu = reinterpret_cast<P4<T> *>(sl + L.pu);
            P4<T> *pv = reinterpret_cast<P4<T> *>(sl + L.vq);
            int *ag = reinterpret_cast<int *>(sl + L.agid);
            int2 *pj = reinterpret_cast<int2 *>(sl + L.pij);
            int *px = reinterpret_cast<int *>(sl + L.pidx);
            int *vx = reinterpret_cast<int *>(sl + L.vidx);
            uint8_t *fc = reinterpret_cast<uint8_t *>(sl + L.face);
            for (int k = threadIdx.x; k < na; k += EDGE_THREADS) {
                pa[k] = S.atom[k];
                ag[k] = S.agid[k];
                fc[k] = S.aface[k];
            }
            for (int k = threadIdx.x; k < np; k += EDGE_THREADS) {
                po[k] = S.po[k];
                pu[k] = S.pu[k];
                pj[k] = S.pij[k];
                px[k] = S.pidx[k];
            }
            for (int k = threadIdx.x; k < nv; k += EDGE_THREADS) {
                pv[k] = S.vq[k];
                vx[k] = S.vidx[k];
            }
            // neighbour sets (expanded spheres within 1e-3 A of meeting; the
            // margin covers the rounding of the staged FP32 positions)
            unsigned *nbm = reinterpret_cast<unsigned *>(sl + L.nbm);
            const int nw = (na + 31) >> 5;
            for (int it = warp; it < na * nw; it += EDGE_WARPS) {
                const int a = it / nw, b = ((it - a * nw) << 5) + lane;
                const P4<T> ca = S.atom[a];
                bool meet = false;
                if (b < na && b != a) {
                    const P4<T> cb = S.atom[b];
                    const T dx = ca.x - cb.x, dy = ca.y - cb.y, dz = ca.z - cb.z;
                    const T reach = ca.w + rpT + T(1e-3) + cb.w + rpT;
                    meet = dx * dx + dy * dy + dz * dz < reach * reach;
                }
                const unsigned bits = __ballot_sync(0xffffffffu, meet);
                if (lane == 0) nbm[it] = bits;
            }
            // staged slots of every pair's atoms
            short2 *ps = reinterpret_cast<short2 *>(sl + L.pslot);
            for (int k = threadIdx.x; k < np; k += EDGE_THREADS) {
                const int2 ij = S.pij[k];
                int si = -1, sj = -1;
                for (int a = 0; a < na; ++a) {
                    const int g = S.agid[a];
                    si = g == ij.x ? a : si;
                    sj = g == ij.y ? a : sj;
                }
                ps[k] = make_short2((short)si, (short)sj);
            }
        }
        // edge records
        for (int e = threadIdx.x; e < ne; e += EDGE_THREADS) {
            const EdgeRef R = edge_ref(E, e);
            const long long g = (long long)E.gbase[R.axis] + (e - E.estart[R.axis]);
            W.einfo[g] = make_int4(ok ? (int)E.slab : 0, edge_pack(R.p, R.axis, R.lab, ok ? 0 : 1),
                                   ok ? (int)(E.sb + E.cs[e]) : 0, ok ? (int)(E.tb + E.ct[e]) : 0);
            W.ecnt[g] = ok ? ((E.cs[e + 1] - E.cs[e]) | ((E.ct[e + 1] - E.ct[e]) << 16)) : 0;
        }
        // the pairs themselves, in item order.  Every slot of the reserved runs
        // below the capacities is written: a slot no pair fills (a dropped tile,
        // or a second prefilter pass that disagreed with the count) gets a dead
        // record (edge -1), so the root kernels never read an unwritten slot.
        if (ok) {
            for (int e0 = 32 * warp; e0 < ne; e0 += EDGE_THREADS) {
                const int e = e0 + lane;
                const bool on = e < ne;
                long long ps = 0, pt = 0, ps1 = 0, pt1 = 0;
                int g = 0;
                if (on) {
                    const EdgeRef R = edge_ref(E, e);
                    g = E.gbase[R.axis] + (e - E.estart[R.axis]);
                    ps = E.sb + E.cs[e];
                    pt = E.tb + E.ct[e];
                    ps1 = E.sb + E.cs[e + 1];
                    pt1 = E.tb + E.ct[e + 1];
                }
                for (int w = 0; w < nwd; ++w)
                    for (unsigned m = word(e, w); m; m &= m - 1) {
                        const int it = 32 * w + __ffs(m) - 1;
                        if (it < nsph) {
                            if (ps < ps1) W.csph[ps++] = make_int2(g, it);
                        } else if (pt < pt1) {
                            W.ctor[pt++] = make_int2(g, it - nsph);
                        }
                    }
                for (; ps < ps1; ++ps) W.csph[ps] = make_int2(-1, 0);
                for (; pt < pt1; ++pt) W.ctor[pt] = make_int2(-1, 0);
            }
        } else {
            const long long s1 = min(E.sb0 + E.cs[ne], W.cap_sph), t1 = min(E.tb0 + E.ct[ne], W.cap_tor);
            for (long long q = E.sb0 + threadIdx.x; q < s1; q += EDGE_THREADS) W.csph[q] = make_int2(-1, 0);
            for (long long q = E.tb0 + threadIdx.x; q < t1; q += EDGE_THREADS) W.ctor[q] = make_int2(-1, 0);
        }
        __syncthreads();
      }
    }
}

// 2. Roots of the sphere candidates, one thread each (grid-stride).
template <class T, bool FILT>
__global__ void __launch_bounds__(ROOT_THREADS_MAX) k_roots_sphere(Model M, Batch B, RootWork W,
                                                                   int *__restrict__ err)
{
    const long long n = min((long long)W.ctr[1], W.cap_sph);
    const double rp = M.rp;
    const T rpT = (T)rp;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int2 c = W.csph[k];
        if (c.x < 0 || c.x >= W.n_edges) {  // dead record
            W.nsph[k] = 0;
            continue;
        }
        const int4 inf = W.einfo[c.x];
        const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
        const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
        const int mol = __ldg(&hd->mol);
        const double x0[3] = {__ldg(&hd->x0[0]), __ldg(&hd->x0[1]), __ldg(&hd->x0[2])};
        const double h = B.grid[mol].h;
        const T d0 = FILT ? (T)B.grid[mol].d0 : T(0);
        const int pk = inf.y, p = pk_point(pk);
        const double s64[3] = {(double)(p >> 6) * h, (double)((p >> 3) & 7) * h, (double)(p & 7) * h};
        T s[3], hT;
        edge_point<T>(B.grid[mol], p, s, hT);
        const SlabAcc<T> A(sl);
        const SlabExact<T> X(A, M, x0, B.grid[mol].d0);
        RootSink out{W.rsph + (size_t)SPH_SLOTS * k, 0, SPH_SLOTS};
        sphere_roots<T, FILT>(A, X, c.y, s, s64, pk_axis(pk), pk_label(pk) == LABEL_IN, hT, rpT, h, rp, d0, out);
        if (out.n > SPH_SLOTS) atomicOr(err, ERR_CAP_CAND);
        W.nsph[k] = (uint8_t)min(out.n, SPH_SLOTS);
    }
}

// The FP32 part of torus_roots (FILT): the certified isolation and, per
// root, the FP32 decisions.  A root whose decision needs FP64 keeps a pending
// slot; a candidate whose isolation is undecided is left whole to the exact
// kernel.  Returns 0 (done), 1 (pending slots) or 2 (whole candidate).
template <class AccT>
__device__ int torus_roots_fp32(const AccT &A, int pi, const float *s, int axis, bool inside, float hT, float rpT,
                                float d0, RootSink &out)
{
    const float lo = -1e-4f, hi = hT + 1e-4f;
    const float tmax = 1e-3f;
    const double NaN = __longlong_as_double(0x7ff8000000000000LL);
    const P4<float> o = A.po(pi);
    const P4<float> u = A.pu(pi);
    const float q0[3] = {s[0] - o.x, s[1] - o.y, s[2] - o.z};
    const float uu[3] = {u.x, u.y, u.z};
    float rt[4];
    int nr = 0;
    if (!torus_roots32(q0, uu, o.w, rpT, axis, lo, hi, d0, rt, nr)) return 2;
    int job = 0;
    const int2 ij = A.pij(pi);
    const short2 sl = A.pslot(pi);
    for (int k = 0; k < nr; ++k) {
        const float t = rt[k];
        float D, rate, nw, yy, zy, wv[3];
        circle_dist32(q0, uu, o.w, axis, t, D, rate, nw, yy, zy, wv);
        const float terr = (fabsf(D - rpT) + circle_dist_err(d0, yy, nw, o.w, rpT)) / fmax(fabs(rate), 1e-20f) + d0;
        if (terr > tmax || t < terr + 1e-6f || t > hT - terr - 1e-6f || fabs(rate) < 1e-3f || nw < 1e-3f) {
            out.pend(t);  // grazing or at an end point: the FP64 root decides
            job = 1;
            continue;
        }
        if (inside ? rate > 0.0f : rate < 0.0f) continue;
        const float kk = o.w / nw;
        const float delta = d0 + terr * (1.0f + 2.0f * o.w / nw) + 2e-6f;
        const int f = free_witness<true>(A, o.x + kk * wv[0], o.y + kk * wv[1], o.z + kk * wv[2], (int)sl.x,
                                         (int)sl.y, ij.x, ij.y, rpT, delta);
        if (f == 1) {
            out.push(t, terr, NaN);
        } else if (f < 0) {
            out.pend(t);
            job = 1;
        }
    }
    return job;
}

// 3. Roots of the torus candidates, one thread each (grid-stride, the lanes
// of a warp together).  FP32 form: torus_roots_fp32, and the candidates with
// FP64 work listed for k_roots_torus_exact (one warp-aggregated append per
// iteration); FP64 form: every root in FP64 here.
template <class T, bool FILT>
__global__ void __launch_bounds__(ROOT_THREADS_MAX) k_roots_torus(Model M, Batch B, RootWork W,
                                                                  int *__restrict__ err)
{
    const long long n = min((long long)W.ctr[2], W.cap_tor);
    const double rp = M.rp;
    const float rpf = (float)rp;
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long k0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); k0 < n; k0 += stride) {
        const long long k = k0 + lane;
        int job = 0;
        if (k < n) {
        const int2 c = W.ctor[k];
        if (c.x < 0 || c.x >= W.n_edges) {  // dead record
            W.ntor[k] = 0;
        } else {
        const int4 inf = W.einfo[c.x];
        const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
        const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
        const int mol = __ldg(&hd->mol);
        const double x0[3] = {__ldg(&hd->x0[0]), __ldg(&hd->x0[1]), __ldg(&hd->x0[2])};
        const double h = B.grid[mol].h;
        const T d0 = FILT ? (T)B.grid[mol].d0 : T(0);
        const int pk = inf.y, p = pk_point(pk);
        const SlabAcc<T> A(sl);
        RootSink out{W.rtor + (size_t)TOR_SLOTS * k, 0, TOR_SLOTS};
        if constexpr (FILT) {
            float s[3], hT;
            edge_point<float>(B.grid[mol], p, s, hT);
            job = torus_roots_fp32(A, c.y, s, pk_axis(pk), pk_label(pk) == LABEL_IN, hT, rpf, (float)d0, out);
        } else {
            const double s64[3] = {(double)(p >> 6) * h, (double)((p >> 3) & 7) * h, (double)(p & 7) * h};
            // The certified isolation leaves the edge's roots as single ones: Newton steps in
            // FP64 from there, and every decision in FP64 (47 k candidates of 200 atoms: the quartic
            // on its derivative chain for each 472 us, 282 us so, 126 us with mono_root's stop).  The quartic where the
            // isolation is undecided or the steps do not settle.
            const int axis = pk_axis(pk);
            const bool inside = pk_label(pk) == LABEL_IN;
            const P4<T> o = A.po(c.y), u = A.pu(c.y);
            const float q0[3] = {(float)(s64[0] - o.x), (float)(s64[1] - o.y), (float)(s64[2] - o.z)};
            const float uu[3] = {(float)u.x, (float)u.y, (float)u.z};
            const double oo[3] = {o.x, o.y, o.z}, u64[3] = {u.x, u.y, u.z};
            float rt[4];
            int nr = 0;
            bool whole = !torus_roots32(q0, uu, (float)o.w, rpf, axis, -1e-4f, (float)h + 1e-4f, B.grid[mol].d0, rt, nr);
            for (int j = 0; j < nr && !whole; ++j) {
                double last = 0.0;
                const double t64 = exact_root_torus(oo, u64, o.w, rp, s64, axis, (double)rt[j], &last);
                if (last < 1e-10) torus_root_exact(A, out, c.y, s64, axis, h, rp, inside, t64);
                else whole = true;
            }
            if (whole) {
                out.n = 0;
                torus_piece_exact(A, out, c.y, s64, axis, h, rp, inside);
            }
        }
        if (out.n > TOR_SLOTS) atomicOr(err, ERR_CAP_CAND);
        W.ntor[k] = (uint8_t)min(out.n, TOR_SLOTS);
        }
        }
        if constexpr (FILT) {  // list the candidates with FP64 work: (candidate, whole)
            const unsigned m = __ballot_sync(0xffffffffu, job != 0);
            if (m) {
                unsigned long long b = 0;
                if (lane == 0) b = atomicAdd(W.ctr + 4, (unsigned long long)__popc(m));
                b = __shfl_sync(0xffffffffu, b, 0);
                if (job != 0) {
                    const unsigned long long q = b + __popc(m & ((1u << lane) - 1));
                    // (a full list is reported by the run from the count)
                    if (q < (unsigned long long)W.cap_jobs) W.jobs[q] = make_int2((int)k, job);
                }
            }
        }
    }
}

// 3b. The listed torus candidates' FP64 work, one thread each (FP32 form
// only): job 1 settles the pending slots (the FP64 root next to the FP32 one,
// kept or rejected as torus_roots does), job 2 solves the whole candidate
// with torus_roots (the quartic on its derivative chain, FP64 where needed).
// Bound by the latency of its chains of loads and FP64 instructions: three
// blocks on an SM rather than the two of its 126 registers (178 -> 157 us on the
// 20,000-atom globule).
__global__ void __launch_bounds__(ROOT_THREADS_MAX, 3) k_roots_torus_exact(Model M, Batch B, RootWork W,
                                                                           int *__restrict__ err)
{
    const long long n = min((long long)W.ctr[4], W.cap_jobs);
    const double rp = M.rp;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const int2 jb = W.jobs[q];
        const long long k = jb.x;
        const int2 c = W.ctor[k];
        const int4 inf = W.einfo[c.x];
        const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
        const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
        const int mol = __ldg(&hd->mol);
        const double x0[3] = {__ldg(&hd->x0[0]), __ldg(&hd->x0[1]), __ldg(&hd->x0[2])};
        const double h = B.grid[mol].h;
        const float d0 = B.grid[mol].d0;
        const int pk = inf.y, p = pk_point(pk), axis = pk_axis(pk);
        const bool inside = pk_label(pk) == LABEL_IN;
        const double s64[3] = {(double)(p >> 6) * h, (double)((p >> 3) & 7) * h, (double)(p & 7) * h};
        const SlabAcc<float> A(sl);
        const SlabExact<float> X(A, M, x0, d0);
        RootRec *slots = W.rtor + (size_t)TOR_SLOTS * k;
        if (jb.y == 2) {
            RootSink out{slots, 0, TOR_SLOTS};
            torus_roots(A, X, c.y, s64, axis, inside, h, rp, d0, out);
            if (out.n > TOR_SLOTS) atomicOr(err, ERR_CAP_CAND);
            W.ntor[k] = (uint8_t)min(out.n, TOR_SLOTS);
        } else {
            const P4<double> oe = X.po(c.y);
            const P4<double> ue = X.pu(c.y);
            const double oo[3] = {oe.x, oe.y, oe.z}, u64[3] = {ue.x, ue.y, ue.z};
            const int nr = W.ntor[k];
            for (int j = 0; j < nr; ++j) {
                const RootRec r = slots[j];
                if (!(r.err < 0.0f)) continue;
                const double t64 = exact_root_torus(oo, u64, oe.w, rp, s64, axis, (double)r.t);
                RootSink one{slots + j, 0, 1};
                torus_root_exact(X, one, c.y, s64, axis, h, rp, inside, t64);
                if (one.n == 0) slots[j] = no_root();
            }
        }
    }
}

// chosen piece of an edge for the FP64 polish: FP32 root, kind, model index,
// end label, failure
__device__ __forceinline__ void code_out(EdgeOut &out, int axis, long long o, int failed, float tr, int kind, int mid,
                                         int lab)
{
    out.code[axis][o] = make_int2(__float_as_int(tr), (kind << 29) | (lab << 28) | (failed << 27) | mid);
}

// Witness of the accepted root at y of a staged piece (kind as in WCand) and a
// bound of its error, dy bounding y's; false where it is ill-conditioned.  An
// accepted root's witness is free.
template <class T>
__device__ __forceinline__ bool root_witness(const SlabAcc<T> &A, int kind, int slot, const T *y, T rp, T d0, T dy,
                                             T *w, T &dw)
{
    if (kind == 2) {
        const P4<T> v = A.vq(slot);
        w[0] = v.x;
        w[1] = v.y;
        w[2] = v.z;
        dw = d0;
        return true;
    }
    if (kind == 0) {
        const P4<T> c = A.atom(slot);
        const T v[3] = {y[0] - c.x, y[1] - c.y, y[2] - c.z}, R = c.w + rp;
        const T sc = R / sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        w[0] = c.x + sc * v[0];
        w[1] = c.y + sc * v[1];
        w[2] = c.z + sc * v[2];
        dw = d0 + (d0 + dy) * (T(1) + T(2) * sc);
        return true;
    }
    const P4<T> o = A.po(slot), u = A.pu(slot);
    const T v[3] = {y[0] - o.x, y[1] - o.y, y[2] - o.z};
    const T z = v[0] * u.x + v[1] * u.y + v[2] * u.z;
    const T p[3] = {v[0] - z * u.x, v[1] - z * u.y, v[2] - z * u.z};
    const T nw = sqrt(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
    if (!(nw > T(1e-2))) return false;
    const T k = o.w / nw;
    w[0] = o.x + k * p[0];
    w[1] = o.y + k * p[1];
    w[2] = o.z + k * p[2];
    dw = d0 + T(2) * k * (d0 + dy + (sizeof(T) == sizeof(float) ? T(2e-6) * (nw + fabs(z)) : T(0)));
    return true;
}

// 4. The first root of every edge whose choice needs neither a witness test
// nor an FP64 tie break, with no candidate the FP32 bounds cannot order: one
// thread per edge, candidates in order (spheres by item, then tori).
// From an inside end point it is the first candidate.  From an outside one it
// is the last if the first lies closer than r_p to the last one's witness: that
// is a free probe centre, the edge between the two lies in the ball of r_p
// around it, so every candidate before the last is strictly outside M.  (A
// single candidate is the last.)  The other edges are listed for the selections:
// without the rule for several candidates 266 k of 1.2 M edges on the
// 5,000-atom globule, 23 k with it.  A dropped edge is recorded as failed (and
// the run as over capacity).
template <class T>
__global__ void __launch_bounds__(PICK_THREADS) k_edge_pick(Model M, Batch B, RootWork W,
                                                            const int *__restrict__ edge_start,
                                                            long long ne_all, EdgeOut out, int *__restrict__ err)
{
    const long long nt = B.n_tiles;
    const int lane = threadIdx.x & 31;
    const long long nwarp = (long long)gridDim.x * (PICK_THREADS / 32);
    for (long long w0 = ((long long)blockIdx.x * (PICK_THREADS / 32) + (threadIdx.x >> 5)) * 32; w0 < ne_all;
         w0 += nwarp * 32) {
        const long long g = w0 + lane;
        bool hard = false;
        if (g < ne_all) {
            const int4 inf = W.einfo[g];
            const int cnt = W.ecnt[g];
            const int ns = cnt & 0xffff, nq = (cnt >> 16) & 0xffff;
            // the axis from the edge's place in the output (all axes in one run)
            const int axis = g < edge_start[nt] ? 0 : (g < edge_start[2 * nt] ? 1 : 2);
            const int pk = inf.y, lab = pk_label(pk);
            const long long o = g - edge_start[axis * nt];
            // a record that is not the staging pass's (never expected) counts as dropped
            const bool bad = pk_axis(pk) != axis || inf.x < 0 || 16LL * inf.x >= W.cap_slab || inf.z < 0 ||
                             inf.w < 0 || (long long)inf.z + ns > W.cap_sph || (long long)inf.w + nq > W.cap_tor;
            if (pk_dropped(pk) || bad) {
                atomicOr(err, ERR_CAP_CAND);
                code_out(out, axis, o, 1, 0.0f, 0, 0, lab);
            } else {
                const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
                const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
                const int na = __ldg(&hd->na);
                // smallest FP32 root (ties to the first) and largest, their records, and the count
                struct Root {
                    float t, err;
                    double t64;
                    int kind, slot, n;
                } first{INFINITY, 0.0f, 0.0, -1, 0, -1}, last{-INFINITY, 0.0f, 0.0, -1, 0, -1};
                int n = 0;
                auto roots = [&](auto f) {  // every accepted root in order: f(root, torus?, record, slot, place)
                    int k = 0;
                    for (int j = 0; j < ns; ++j) {
                        const int nr = W.nsph[inf.z + j];
                        for (int r = 0; r < nr; ++r) {
                            const RootRec q = W.rsph[(size_t)SPH_SLOTS * (inf.z + j) + r];
                            if (q.t < INFINITY) f(q, false, j, r, k++);
                        }
                    }
                    for (int j = 0; j < nq; ++j) {
                        const int nr = W.ntor[inf.w + j];
                        for (int r = 0; r < nr; ++r) {
                            const RootRec q = W.rtor[(size_t)TOR_SLOTS * (inf.w + j) + r];
                            if (q.t < INFINITY && !(q.err < 0.0f)) f(q, true, j, r, k++);  // (else rejected or never settled)
                        }
                    }
                    return k;
                };
                n = roots([&](const RootRec &q, bool tor, int j, int, int k) {
                    if (q.t < first.t) first = Root{q.t, q.err, q.t64, tor ? 1 : 0, j, k};
                    if (q.t > last.t) last = Root{q.t, q.err, q.t64, tor ? 1 : 0, j, k};
                });
                const Grid &G = B.grid[__ldg(&hd->mol)];
                const float tie = 1e-6f * G.hl[1];
                const bool in = lab == LABEL_IN || n == 1;
                hard = !(n >= 1 && n <= WCAND && first.n >= 0);
                Root &pick = in ? first : last;
                if (!hard && n > 1) {  // every other candidate certainly after the first, or before the last
                    roots([&](const RootRec &q, bool, int, int, int k) {
                        if (k != pick.n && (in ? q.t - pick.t : pick.t - q.t) <= q.err + pick.err + tie) hard = true;
                    });
                }
                const SlabAcc<T> A(sl);
                if (!hard) {  // the piece: spheres are numbered atoms first, then triple points
                    if (pick.kind == 0) {
                        const int it = W.csph[inf.z + pick.slot].y;
                        pick.kind = it < na ? 0 : 2;
                        pick.slot = it < na ? it : it - na;
                    } else {
                        pick.slot = W.ctor[inf.w + pick.slot].y;
                    }
                    if (!in) {
                        const bool e0 = first.t64 == first.t64, e1 = last.t64 == last.t64;  // exact roots
                        const T d0 = sizeof(T) == sizeof(float) ? (T)G.d0 : T(0);
                        T s[3], hT, y0[3], y1[3], w[3], dw;
                        edge_point<T>(G, pk_point(pk), s, hT);
                        const T rp = (T)M.rp;
                        const T t0 = e0 ? (T)first.t64 : (T)first.t, t1 = e1 ? (T)last.t64 : (T)last.t;
                        for (int a = 0; a < 3; ++a) {
                            y0[a] = s[a] + (a == axis ? t0 : T(0));
                            y1[a] = s[a] + (a == axis ? t1 : T(0));
                        }
                        const T f0 = (e0 ? T(2e-7) : (T)first.err) + d0, f1 = e1 ? T(2e-7) : (T)last.err;
                        hard = true;
                        if (root_witness<T>(A, last.kind, last.slot, y1, rp, d0, f1, w, dw)) {
                            const T dx = y0[0] - w[0], dy = y0[1] - w[1], dz = y0[2] - w[2];
                            hard = lt_sq<true>(dx * dx + dy * dy + dz * dz, rp * rp, rp, f0 + dw + T(2e-6)) != 1;
                        }
                    }
                }
                if constexpr (sizeof(T) == sizeof(float)) {
                    // a hard edge's candidates that the bounds cannot order against the first or the last one: their
                    // FP64 roots are made before the selection
                    if (hard && n > 1) {
                        auto near = [&](const Root &e, const RootRec &q, int k) {
                            return k != e.n && fabsf(q.t - e.t) <= q.err + e.err + tie;
                        };
                        bool near_first = false, near_last = false;
                        roots([&](const RootRec &q, bool, int, int, int k) {
                            near_first = near_first || near(first, q, k);
                            near_last = near_last || near(last, q, k);
                        });
                        roots([&](const RootRec &q, bool tor, int j, int r, int k) {
                            const bool tied = near(first, q, k) || near(last, q, k) || (k == first.n && near_first) ||
                                              (k == last.n && near_last);
                            if (!tied || q.t64 == q.t64) return;
                            const unsigned long long z = atomicAdd(W.ctr + 5, 1ull);
                            if (z >= (unsigned long long)W.cap_ties) return;
                            const int rec = (tor ? inf.w : inf.z) + j, it = tor ? W.ctor[rec].y : W.csph[rec].y;
                            W.ties[z] = make_int4((int)g, rec, r | ((tor ? 1 : (it < na ? 0 : 2)) << 4),
                                                  !tor && it >= na ? it - na : it);
                        });
                    }
                }
                if (!hard) {
                    const float tr = pick.t64 == pick.t64 ? (float)pick.t64 : pick.t;
                    code_out(out, axis, o, 0, tr, pick.kind, A.model_index(pick.kind, pick.slot), lab);
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, hard);
        int base = 0;
        if (lane == 0 && m) base = (int)atomicAdd(W.ctr + 3, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (hard) W.hard[base + __popc(m & ((1u << lane) - 1))] = (int)g;
    }
}

// 4b. FP32 form only: FP64 roots of the listed tied candidates, one thread each, into their records.
__global__ void __launch_bounds__(128) k_edge_ties(Model M, Batch B, RootWork W)
{
    const long long n = min((long long)W.ctr[5], W.cap_ties);
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const int4 jb = W.ties[q];
        const int4 inf = W.einfo[jb.x];
        const int kind = jb.z >> 4, r = jb.z & 15, p = pk_point(inf.y);
        const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
        const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
        const double x0[3] = {__ldg(&hd->x0[0]), __ldg(&hd->x0[1]), __ldg(&hd->x0[2])};
        const double h = B.grid[__ldg(&hd->mol)].h;
        const double s64[3] = {(double)(p >> 6) * h, (double)((p >> 3) & 7) * h, (double)(p & 7) * h};
        const SlabAcc<float> A(sl);
        const SlabExact<float> X(A, M, x0, B.grid[hd->mol].d0);
        RootRec *rec = kind == 1 ? W.rtor + (size_t)TOR_SLOTS * jb.y + r : W.rsph + (size_t)SPH_SLOTS * jb.y + r;
        rec->t64 = staged_exact_root(X, kind, jb.w, s64, pk_axis(inf.y), M.rp, (double)rec->t);
    }
}

// 5. The listed edges: one warp per edge (grid-stride over the list).  The
// edge's accepted roots are gathered in candidate order into the warp's
// buffer in shared memory (at most WCAND; more is a capacity error), then
// chosen by warp_select.  A failure is logged with its candidates.
// Bound by latency (a warp's witness searches, one after the other): three
// blocks on an SM rather than two at 118 registers, 422 -> 390 us on 38 k edges.
template <class T, bool FILT>
__global__ void __launch_bounds__(HARD_THREADS, FILT ? 3 : 1) k_edge_hard(Model M, Batch B, RootWork W,
                                                            const int *__restrict__ edge_start, EdgeOut out,
                                                            int *__restrict__ n_fail, int *__restrict__ err,
                                                            long long *__restrict__ fail_log)
{
    __shared__ WCand cand[HARD_THREADS / 32][WCAND];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long nt = B.n_tiles;
    const long long nh = (long long)W.ctr[3];
    const double rp = M.rp;
    const T rpT = (T)rp;
    WCand *c = cand[warp];
    for (long long q = (long long)blockIdx.x * (HARD_THREADS / 32) + warp; q < nh;
         q += (long long)gridDim.x * (HARD_THREADS / 32)) {
        const int g = W.hard[q];
        const int4 inf = W.einfo[g];
        const int cnt = W.ecnt[g];
        const int ns = cnt & 0xffff, nq = (cnt >> 16) & 0xffff;
        const int pk = inf.y, axis = pk_axis(pk), lab = pk_label(pk), p = pk_point(pk);
        const long long o = (long long)g - edge_start[axis * nt];
        const unsigned char *sl = W.slab + ((size_t)(unsigned)inf.x << 4);
        const SlabHdr *hd = reinterpret_cast<const SlabHdr *>(sl);
        const int mol = __ldg(&hd->mol);
        const double x0[3] = {__ldg(&hd->x0[0]), __ldg(&hd->x0[1]), __ldg(&hd->x0[2])};
        const double h = B.grid[mol].h;
        const T d0 = FILT ? (T)B.grid[mol].d0 : T(0);
        const double s64[3] = {(double)(p >> 6) * h, (double)((p >> 3) & 7) * h, (double)(p & 7) * h};
        T s[3], hT;
        edge_point<T>(B.grid[mol], p, s, hT);
        const SlabAcc<T> A(sl);
        const SlabExact<T> X(A, M, x0, B.grid[mol].d0);
        const int na = A.na();
        // gather: lanes over candidates, each lane's roots at its prefix of the counts
        int n = 0;
        for (int j0 = 0; j0 < ns + nq; j0 += 32) {
            const int j = j0 + lane;
            const bool sph = j < ns;
            int nr = 0;
            if (j < ns + nq) nr = sph ? W.nsph[inf.z + j] : W.ntor[inf.w + (j - ns)];
            int inc = nr;
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += u;
            }
            const int at = n + inc - nr;
            if (nr > 0) {
                int kind, slot;
                if (sph) {
                    const int it = W.csph[inf.z + j].y;
                    kind = it < na ? 0 : 2;
                    slot = it < na ? it : it - na;
                } else {
                    kind = 1;
                    slot = W.ctor[inf.w + (j - ns)].y;
                }
                for (int r = 0; r < nr; ++r) {
                    if (at + r >= WCAND) break;
                    const RootRec qr = sph ? W.rsph[(size_t)SPH_SLOTS * (inf.z + j) + r]
                                           : W.rtor[(size_t)TOR_SLOTS * (inf.w + (j - ns)) + r];
                    WCand &w = c[at + r];
                    w.t64 = qr.t64;
                    w.t = qr.err < 0.0f ? INFINITY : qr.t;  // a rejected (or unsettled) slot: no candidate
                    w.err = qr.err;
                    w.kind = kind;
                    w.id = slot;
                }
            }
            n += __shfl_sync(0xffffffffu, inc, 31);
        }
        __syncwarp();
        float tr = 0.5f * (float)h;
        int kind = 0, slot = 0;
        int status = pk_dropped(pk) ? 2 : warp_select<T, FILT>(A, X, c, n, s, s64, axis, lab == LABEL_IN, (float)hT, rpT, rp, d0, tr,
                                                               kind, slot);
        if (lane == 0) {
            const int mid = status == 1 || pk_dropped(pk) ? 0 : A.model_index(kind, slot);
            if (status != 0) atomicOr(err, status == 1 ? ERR_ROOT : ERR_CAP_CAND);
            if (status == 1) {
                const int fs = atomicAdd(n_fail, 1);
                if (fs < FAIL_LOG) {
                    long long *rec = fail_log + FAIL_REC * fs;
                    for (int z = 0; z < FAIL_REC; ++z) rec[z] = 0;
                    rec[0] = axis;
                    rec[1] = (long long)TILE * __ldg(&hd->t[0]) + (p >> 6);
                    rec[2] = (long long)TILE * __ldg(&hd->t[1]) + ((p >> 3) & 7);
                    rec[3] = (long long)TILE * __ldg(&hd->t[2]) + (p & 7);
                    rec[4] = lab;
                    rec[5] = na;
                    rec[6] = A.np();
                    rec[7] = A.nv();
                    rec[8] = n;
                    for (int z = 0; z < 7 && z < n && z < WCAND; ++z) {
                        rec[9 + z] = (long long)((double)c[z].t * 1e9);
                        rec[16 + z] = c[z].kind;
                    }
                    rec[23] = mol;
                }
            }
            code_out(out, axis, o, status == 1 || pk_dropped(pk) ? 1 : 0, tr, kind, mid, lab);
        }
        __syncwarp();
    }
}

// One thread per crossing edge, over the three axes: FP64 root of the chosen
// piece next to the recorded FP32 root, normal, outputs, area/volume terms.
// Bound by FP64 issue (one warp instruction per 16 cycles per SM, 83 % of the
// time).  The block's edges are first ordered by kind, tori before spheres, so
// nearly every warp runs one of the two paths instead of both (513 -> 326 us
// on 1.2 M edges), four blocks stay on an SM (285 us; 82 -> 68 us on 0.1 M
// edges), and the two paths spend few FP64 divisions and square roots
// (polish_sphere, polish_torus): 443 -> 305 us on 1.9 M edges, 58 -> 42 us on 0.18 M.
__global__ void __launch_bounds__(POLISH_THREADS, 4) k_edge_polish(Model M, Batch B, EdgeOut out,
                                                                const long long *__restrict__ medge,
                                                                double2 *__restrict__ term)
{
    __shared__ short order[POLISH_THREADS];
    __shared__ int n_tor[POLISH_THREADS / 32];
    const long long e0 = (long long)blockIdx.x * POLISH_THREADS;
    const int nm = B.n_mol;
    const long long n0 = medge[nm], n1 = medge[2 * nm + 1], n2 = medge[3 * nm + 2];
    const double rp = M.rp;
    {
        const long long e = e0 + threadIdx.x;
        const int a = e < n0 ? 0 : (e < n0 + n1 ? 1 : 2);
        const long long o = e - (a == 0 ? 0 : (a == 1 ? n0 : n0 + n1));
        const bool tor = e < n0 + n1 + n2 && ((out.code[a][o].y >> 29) & 3) == 1;
        const unsigned m = __ballot_sync(0xffffffffu, tor);
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane == 0) n_tor[warp] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < POLISH_THREADS / 32; ++w) {
            if (w < warp) before += n_tor[w];
            all += n_tor[w];
        }
        before += __popc(m & ((1u << lane) - 1));
        order[tor ? before : all + (int)threadIdx.x - before] = (short)threadIdx.x;
        __syncthreads();
    }
    const long long e = e0 + order[threadIdx.x];
    if (e < n0 + n1 + n2) {
        const int a = e < n0 ? 0 : (e < n0 + n1 ? 1 : 2);
        const long long o = e - (a == 0 ? 0 : (a == 1 ? n0 : n0 + n1));
        // molecule of the edge: its axis output is molecule-major
        const long long *me = medge + a * (nm + 1);
        int lo = 0, hi = nm;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (me[mid] <= o) lo = mid;
            else hi = mid;
        }
        const Grid &G = B.grid[lo];
        const double h = G.h;
        const long long idx = out.idx[a][o];
        const int2 code = out.code[a][o];
        const float t32 = __int_as_float(code.x);
        const int kind = (code.y >> 29) & 3, lab_s = (code.y >> 28) & 1, failed = (code.y >> 27) & 1;
        const int mid = code.y & ((1 << 27) - 1);
        // the recorded piece must exist (a kind and index out of range is treated as a failed root)
        const bool bad = kind == 3 || (kind == 0 && mid >= M.n_atoms) || (kind == 1 && mid >= M.n_pairs) ||
                         (kind == 2 && mid >= M.n_verts);
        double s[3];  // full-grid point of the lower index
        if (idx < (1LL << 32) && G.full[1] * G.full[2] < (1LL << 32)) {  // 32-bit division where it fits
            const unsigned i32 = (unsigned)idx, d2 = (unsigned)G.full[2], d1 = (unsigned)G.full[1];
            const unsigned q = i32 / d2;
            s[0] = G.lo[0] + h * (double)(q / d1);
            s[1] = G.lo[1] + h * (double)(q % d1);
            s[2] = G.lo[2] + h * (double)(i32 - q * d2);
        } else {
            s[0] = G.lo[0] + h * (double)(idx / (G.full[1] * G.full[2]));
            s[1] = G.lo[1] + h * (double)((idx / G.full[2]) % G.full[1]);
            s[2] = G.lo[2] + h * (double)(idx % G.full[2]);
        }
        double t = 0.5 * h, n[3] = {0.0, 0.0, 0.0};
        if (!failed && !bad) {
            if (kind != 1) {
                const double4 g = kind == 0 ? M.atom[mid] : M.vert[mid];
                const double c[3] = {g.x, g.y, g.z};
                t = polish_sphere(c, kind == 0 ? g.w : rp, kind == 0 ? 1.0 : -1.0, s, a, (double)t32, h, n);
            } else {
                const double4 g = M.pair_o[mid], q = M.pair_u[mid];
                const double c[3] = {g.x, g.y, g.z}, u[3] = {q.x, q.y, q.z};
                t = polish_torus(c, u, g.w, rp, s, a, (double)t32, h, n);
            }
        }
        const double tau = t * G.ih;
        out.tau[a][o] = tau;
        out.nrm[a][3 * o + 0] = n[0];
        out.nrm[a][3 * o + 1] = n[1];
        out.nrm[a][3 * o + 2] = n[2];
        out.tau32[a][o] = (float)tau;
        out.nrm32[a][3 * o + 0] = (float)n[0];
        out.nrm32[a][3 * o + 1] = (float)n[1];
        out.nrm32[a][3 * o + 2] = (float)n[2];
        // Crofton area term and the inside length of the edge (C9)
        term[e] = make_double2(h * h * fabs(n[a]), lab_s ? t : h - t);
    }
}

// Area/volume reduction in two fixed-order levels (deterministic): block
// (m, g) of k_reduce_part sums the terms of molecule m whose index within the
// molecule's range is g (mod parts * blockDim), in a fixed tree, for the
// molecule's number of parts (red_parts; the blocks past it return);
// k_reduce_final adds those partials of each molecule in a fixed tree.
constexpr int RED_PARTS = 64;  // at most (16 parts: 192 us on one molecule's 4.9 M terms, 53 us on 1.2 M; 58 and 17 now)
constexpr int RED_THREADS = 512;

// parts of a molecule: its own size decides (a batch's molecule is summed as it
// is alone), a part for every 8,192 terms and tiles
__device__ __forceinline__ int red_parts(const Batch &B, const long long *medge, int m)
{
    const int nm = B.n_mol;
    long long n = B.tile_off[m + 1] - B.tile_off[m];
    for (int a = 0; a < 3; ++a) n += medge[a * (nm + 1) + m + 1] - medge[a * (nm + 1) + m];
    return (int)max(1LL, min((long long)RED_PARTS, n / 8192));
}

__global__ void __launch_bounds__(RED_THREADS) k_reduce_part(Batch B, const double2 *__restrict__ term,
                                                             const long long *__restrict__ medge,
                                                             const int *__restrict__ tile_inside,
                                                             double *__restrict__ part_d,
                                                             long long *__restrict__ part_i)
{
    __shared__ double sa[32], sv[32];
    __shared__ long long si[32], sp[32];
    const int m = blockIdx.x / RED_PARTS, g = blockIdx.x % RED_PARTS, nm = B.n_mol;
    const int parts = red_parts(B, medge, m);
    if (g >= parts) return;
    const long long nt = B.n_tiles;
    const long long stride = (long long)parts * RED_THREADS;
    const long long first = (long long)g * RED_THREADS + threadIdx.x;
    double a = 0.0, v = 0.0;
    long long ie = 0, pin = 0;
    long long axis_base = 0;
    for (int ax = 0; ax < 3; ++ax) {
        const long long *me = medge + ax * (nm + 1);
        for (long long k = me[m] + first; k < me[m + 1]; k += stride) {
            const double2 w = term[axis_base + k];
            a += w.x;
            v += w.y;
        }
        axis_base += me[nm];
    }
    for (long long k = B.tile_off[m] + first; k < B.tile_off[m + 1]; k += stride) {
        ie += (long long)tile_inside[k] + tile_inside[nt + k] + tile_inside[2 * nt + k];
        pin += tile_inside[3 * nt + k];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        v += __shfl_down_sync(0xffffffffu, v, o);
        ie += __shfl_down_sync(0xffffffffu, ie, o);
        pin += __shfl_down_sync(0xffffffffu, pin, o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sa[wid] = a;
        sv[wid] = v;
        si[wid] = ie;
        sp[wid] = pin;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double A = 0.0, V = 0.0;
        long long IE = 0, P = 0;
        for (int k = 0; k < RED_THREADS / 32; ++k) {
            A += sa[k];
            V += sv[k];
            IE += si[k];
            P += sp[k];
        }
        part_d[2 * blockIdx.x] = A;
        part_d[2 * blockIdx.x + 1] = V;
        part_i[2 * blockIdx.x] = P;
        part_i[2 * blockIdx.x + 1] = IE;
    }
}

// out2[2m..] = {area, volume}; counts[2m..] = {inside points, inside edges (all axes)}: a warp per molecule,
// its parts over the lanes, then a fixed tree
__global__ void k_reduce_final(Batch B, const long long *__restrict__ medge, const double *__restrict__ part_d, const long long *__restrict__ part_i,
                               double *__restrict__ out2, long long *__restrict__ counts)
{
    const int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (m >= B.n_mol) return;
    double A = 0.0, V = 0.0;
    long long P = 0, IE = 0;
    const int parts = red_parts(B, medge, m);
    for (int g = lane; g < parts; g += 32) {
        const int k = m * RED_PARTS + g;
        A += part_d[2 * k];
        V += part_d[2 * k + 1];
        P += part_i[2 * k];
        IE += part_i[2 * k + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        A += __shfl_xor_sync(0xffffffffu, A, o);
        V += __shfl_xor_sync(0xffffffffu, V, o);
        P += __shfl_xor_sync(0xffffffffu, P, o);
        IE += __shfl_xor_sync(0xffffffffu, IE, o);
    }
    if (lane == 0) {
        const double h = B.grid[m].h;
        out2[2 * m] = A;
        out2[2 * m + 1] = h * h * (V + h * (double)IE) / 3.0;
        counts[2 * m] = P;
        counts[2 * m + 1] = IE;
    }
}

static int grid_tiles(long long n)
{
    long long g = n < 1 ? 1 : n;
    return (int)(g > 2147483647LL ? 2147483647LL : g);
}

int launch_edge_count(const Batch &B, const int8_t *labels, int *tile_edges, int *tile_inside, int *etiles,
                      cudaStream_t st)
{
    cudaMemsetAsync(etiles, 0, sizeof(int), st);
    k_edge_count<<<grid_tiles((B.n_tiles + COUNT_WARPS - 1) / COUNT_WARPS), COUNT_WARPS * 32, 0, st>>>(
        B, labels, tile_edges, tile_inside, etiles);
    return 1;
}

int launch_mol_edges(const Batch &B, const int *edge_start, long long *medge, cudaStream_t st)
{
    const int n = 3 * (B.n_mol + 1);
    k_mol_edges<<<(n + 255) / 256, 256, 0, st>>>(B, edge_start, medge);
    return 1;
}

template <class T>
static size_t stage_smem()
{
    return edge_tile_bytes<T, CapMid>() + sizeof(StageSmem);
}

static int g_edge_n_sm = 1;  // SMs: the grid of the global-memory tier and of the persistent root kernels
// resident blocks per SM: [FP64, FP32][sphere roots, torus roots][64, 128, 256 threads]; hard selection
static int g_occ_roots[2][2][3];
static int g_occ_hard[2];
static int g_occ_exact;

static int threads_slot(int threads) { return threads <= 64 ? 0 : (threads <= 128 ? 1 : 2); }

// dynamic shared memory limits and occupancies (once per device, before any launch or capture)
void edges_init()
{
    cudaFuncSetAttribute(k_edge_stage<double, false, CapMid, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)stage_smem<double>());
    cudaFuncSetAttribute(k_edge_stage<float, true, CapMid, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)stage_smem<float>());
    cudaFuncSetAttribute(k_edge_stage<double, false, CapBig, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(StageSmem));
    cudaFuncSetAttribute(k_edge_stage<float, true, CapBig, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(StageSmem));
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    g_edge_n_sm = n_sm > 0 ? n_sm : 1;
    const int tb[3] = {64, 128, 256};
    for (int k = 0; k < 3; ++k) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_roots[0][0][k], k_roots_sphere<double, false>, tb[k], 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_roots[0][1][k], k_roots_torus<double, false>, tb[k], 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_roots[1][0][k], k_roots_sphere<float, true>, tb[k], 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_roots[1][1][k], k_roots_torus<float, true>, tb[k], 0);
    }
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_exact, k_roots_torus_exact, 256, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_hard[0], k_edge_hard<double, false>, HARD_THREADS, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_occ_hard[1], k_edge_hard<float, true>, HARD_THREADS, 0);
}

// bytes of global scratch the staging pass's global-memory tier needs
size_t edges_big_bytes()
{
    size_t per = edge_tile_bytes<double, CapBig>();
    if (edge_tile_bytes<float, CapBig>() > per) per = edge_tile_bytes<float, CapBig>();
    return per * (size_t)g_edge_n_sm;
}

int edge_ctas_per_sm(int precision)
{
    int n = 0;
    if (precision == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_edge_stage<double, false, CapMid, false>, EDGE_THREADS,
                                                      stage_smem<double>());
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_edge_stage<float, true, CapMid, false>, EDGE_THREADS,
                                                      stage_smem<float>());
    return n > 0 ? n : 1;
}

bool root_threads_valid(int threads) { return threads == 0 || threads == 64 || threads == 128 || threads == 256; }

long long slab_bytes_max(int precision)
{
    return precision == 0 ? SlabLayout<double>(CapBig::A, CapBig::P, CapBig::V).bytes
                          : SlabLayout<float>(CapBig::A, CapBig::P, CapBig::V).bytes;
}

template <class T, bool FILT>
static void stage_launch(const Model &M, const Batch &B, const TileSched &Q, int grid, const int8_t *labels,
                         const int *edge_start, EdgeOut out, int *err, int *ovf, unsigned char *big,
                         const RootWork &W, cudaStream_t st)
{
    cudaMemsetAsync(W.ctr, 0, 8 * sizeof(unsigned long long), st);
    if (Q.head) cudaMemsetAsync(Q.head, 0, sizeof(unsigned long long), st);
    cudaMemsetAsync(ovf + 1, 0, sizeof(int), st);
    k_edge_stage<T, FILT, CapMid, false><<<grid, EDGE_THREADS, stage_smem<T>(), st>>>(M, B, Q, labels, edge_start,
                                                                                       out, err, ovf, nullptr, W);
    TileSched QB{nullptr, 1, ovf + 2, ovf + 1};
    if (!big) return;
    k_edge_stage<T, FILT, CapBig, true><<<g_edge_n_sm, EDGE_THREADS, sizeof(StageSmem), st>>>(
        M, B, QB, labels, edge_start, out, err, ovf, big, W);
}

template <class T, bool FILT>
static void roots_launch(const Model &M, const Batch &B, int threads, EdgeOut out, const int *edge_start,
                         long long ne_all, int *n_fail, int *err, long long *fail_log, const RootWork &W,
                         cudaStream_t st)
{
    const int P = FILT ? 1 : 0, ts = threads_slot(threads), tb = 64 << ts;
    const int gs = std::max(g_occ_roots[P][0][ts], 1) * g_edge_n_sm;
    const int gq = std::max(g_occ_roots[P][1][ts], 1) * g_edge_n_sm;
    k_roots_sphere<T, FILT><<<gs, tb, 0, st>>>(M, B, W, err);
    cudaMemsetAsync(W.ctr + 3, 0, 3 * sizeof(unsigned long long), st);  // listed edges, FP64 jobs, ties
    k_roots_torus<T, FILT><<<gq, tb, 0, st>>>(M, B, W, err);
    if (FILT)
        k_roots_torus_exact<<<std::max(g_occ_exact, 1) * g_edge_n_sm, tb, 0, st>>>(M, B, W, err);
    const long long pb = std::min<long long>(std::max<long long>(ceil_div_ll(ne_all, PICK_THREADS), 1),
                                             8LL * g_edge_n_sm);
    k_edge_pick<T><<<(unsigned)pb, PICK_THREADS, 0, st>>>(M, B, W, edge_start, ne_all, out, err);
    if (FILT)
        k_edge_ties<<<(unsigned)std::min<long long>(std::max<long long>(ceil_div_ll(ne_all, 1024), 1), 8LL * g_edge_n_sm),
                      128, 0, st>>>(M, B, W);
    k_edge_hard<T, FILT><<<std::max(g_occ_hard[P], 1) * g_edge_n_sm, HARD_THREADS, 0, st>>>(
        M, B, W, edge_start, out, n_fail, err, fail_log);
}

int launch_edge_stage(const Model &M, const Batch &B, int precision, const TileSched &Q, int grid,
                      const int8_t *labels, const int *edge_start, EdgeOut out, int *err, int *ovf,
                      unsigned char *big, const RootWork &W, cudaStream_t st)
{
    if (grid < 1) grid = 1;
    if (precision == 0)
        stage_launch<double, false>(M, B, Q, grid, labels, edge_start, out, err, ovf, big, W, st);
    else
        stage_launch<float, true>(M, B, Q, grid, labels, edge_start, out, err, ovf, big, W, st);
    return big ? 2 : 1;
}

int launch_edge_roots(const Model &M, const Batch &B, int precision, int threads, EdgeOut out,
                      const int *edge_start, long long ne_all, int *n_fail, int *err, long long *fail_log,
                      const RootWork &W, cudaStream_t st)
{
    if (!root_threads_valid(threads) || threads == 0) threads = ROOT_THREADS_MAX;
    // the failures of these launches only: planning runs them again when the FP64 job list was full, and what
    // it lacked then counted as failed edges
    cudaMemsetAsync(n_fail, 0, sizeof(int), st);
    if (precision == 0)
        roots_launch<double, false>(M, B, threads, out, edge_start, ne_all, n_fail, err, fail_log, W, st);
    else
        roots_launch<float, true>(M, B, threads, out, edge_start, ne_all, n_fail, err, fail_log, W, st);
    return precision == 0 ? 4 : 6;
}

long long polish_blocks(long long n_edges) { return n_edges > 0 ? ceil_div_ll(n_edges, POLISH_THREADS) : 0; }

int launch_edge_polish(const Model &M, const Batch &B, EdgeOut out, long long n_edges_total,
                       const long long *medge, double2 *term, cudaStream_t st)
{
    long long nb = polish_blocks(n_edges_total);
    if (nb > 0) k_edge_polish<<<(unsigned)nb, POLISH_THREADS, 0, st>>>(M, B, out, medge, term);
    return nb > 0 ? 1 : 0;
}

long long reduce_scratch(int n_mol) { return 2LL * RED_PARTS * n_mol; }

int launch_reduce(const Batch &B, const double2 *term, const long long *medge, const int *tile_inside, double *part_d,
                  long long *part_i, double *out2, long long *counts, cudaStream_t st)
{
    k_reduce_part<<<B.n_mol * RED_PARTS, RED_THREADS, 0, st>>>(B, term, medge, tile_inside, part_d, part_i);
    k_reduce_final<<<(B.n_mol + 3) / 4, 128, 0, st>>>(B, medge, part_d, part_i, out2, counts);
    return 2;
}

}  // namespace eses
