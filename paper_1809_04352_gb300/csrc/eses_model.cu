// eses_model.cu -- analytic patch construction (the first ESES stage, §2.2).
//
// From the atoms this builds, in FP64:
//   1. a counting sort of the atoms into uniform cells (cell edge 2 R_max, so
//      every overlapping pair of expanded balls sits in adjacent cells);
//   2. neighbour lists: j with |c_i - c_j| < R_i + R_j;
//   3. circle pairs: i < j whose expanded spheres meet in a circle
//      (|R_i - R_j| < D < R_i + R_j), carrier of the saddle (toroidal) patch;
//   4. for every circle, the arcs covered by the other expanded balls: a ball k
//      covers the arc where cos(phi - psi_k) > T_k; the circle keeps a free
//      arc unless one ball covers it whole or every covered-arc end point is
//      itself covered.  A free end point lies on three expanded spheres and in
//      no other ball: it is a free triple point (concave patch centre; the
//      probe-clash test of the north-star is this freeness test, in FP64);
//   5. a per-atom flag "the expanded sphere keeps a free face";
//   6. free-arc pairs and free triple points binned into the cells.
// The paper builds patches from all atom pairs under a distance threshold
// (§5) -- the same set as step 3.
#include <math.h>

#include <algorithm>

#include "eses_kernels.h"

namespace eses {

// double-float split of a grid-frame coordinate
__device__ __forceinline__ void split_df(double v, float &hi, float &lo)
{
    hi = (float)v;
    lo = (float)(v - (double)hi);
}

__device__ __forceinline__ int cell_coord(double v, double lo, double cell, int n)
{
    int k = (int)floor((v - lo) / cell);
    return k < 0 ? 0 : (k >= n ? n - 1 : k);
}

// cell id of a point of molecule m
__device__ __forceinline__ int cell_of(const CellGrid &g, double cell, double x, double y, double z)
{
    int a = cell_coord(x, g.clo[0], cell, g.cn[0]);
    int b = cell_coord(y, g.clo[1], cell, g.cn[1]);
    int c = cell_coord(z, g.clo[2], cell, g.cn[2]);
    return g.coff + (a * g.cn[1] + b) * g.cn[2] + c;
}

__global__ void k_cell_count(const double *__restrict__ xyz, const int *__restrict__ in_mol, int n,
                             const CellGrid *__restrict__ cg, double cell, int *__restrict__ cell_id,
                             int *__restrict__ cell_count)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int id = cell_of(cg[in_mol[i]], cell, xyz[3 * i + 0], xyz[3 * i + 1], xyz[3 * i + 2]);
    cell_id[i] = id;
    atomicAdd(&cell_count[id], 1);
}

int launch_cell_count(const double *xyz, const int *in_mol, int n, const CellGrid *cg, double cell, int *cell_id,
                      int *cell_count, cudaStream_t st)
{
    if (n <= 0) return 0;
    k_cell_count<<<(n + 255) / 256, 256, 0, st>>>(xyz, in_mol, n, cg, cell, cell_id, cell_count);
    return 1;
}

__global__ void k_cell_scatter(int n, const int *__restrict__ cell_id, const int *__restrict__ cell_start,
                               int *__restrict__ cursor, int *__restrict__ sorted_orig)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int id = cell_id[i];
    sorted_orig[cell_start[id] + atomicAdd(&cursor[id], 1)] = i;
}

int launch_cell_scatter(const double *, const double *, int n, const int *cell_id, const int *cell_start, int *cursor,
                         int *sorted_orig, cudaStream_t st)
{
    if (n <= 0) return 0;
    k_cell_scatter<<<(n + 255) / 256, 256, 0, st>>>(n, cell_id, cell_start, cursor, sorted_orig);
    return 1;
}

// Every cell's atoms ordered by original atom index (deterministic layout),
// gathered with their FP32 copies.  One warp per cell, an atom's place its rank
// among the cell's indices (one thread's insertion sort in global memory held
// the launch to 85 us on 26 atoms a cell; 6 us now).
constexpr int CELL_WARPS = 4;

__global__ void __launch_bounds__(CELL_WARPS * 32) k_cell_finish(
    const double *__restrict__ xyz, const double *__restrict__ r, const int *__restrict__ in_mol, int ncell,
    const int *__restrict__ cell_start, const int *__restrict__ scattered, const Grid *__restrict__ grids,
    int *__restrict__ sorted_orig, double4 *__restrict__ atom, int *__restrict__ atom_mol,
    int *__restrict__ atom_cell, float4 *__restrict__ hi, float4 *__restrict__ lo)
{
    const int lane = threadIdx.x & 31;
    for (long long c = (long long)blockIdx.x * CELL_WARPS + (threadIdx.x >> 5); c < ncell;
         c += (long long)gridDim.x * CELL_WARPS) {
        const int s = cell_start[c], e = cell_start[c + 1];
        for (int a = s + lane; a < e; a += 32) {
            const int o = scattered[a];
            int rank = 0;
            for (int b = s; b < e; ++b) rank += scattered[b] < o ? 1 : 0;
            const int k = s + rank, mol = in_mol[o];
            const double4 at = make_double4(xyz[3 * o], xyz[3 * o + 1], xyz[3 * o + 2], r[o]);
            sorted_orig[k] = o;
            atom[k] = at;
            atom_mol[k] = mol;
            atom_cell[k] = (int)c;
            const double *L = grids[mol].lo;
            float hx, hy, hz, ex, ey, ez;
            split_df(at.x - L[0], hx, ex);
            split_df(at.y - L[1], hy, ey);
            split_df(at.z - L[2], hz, ez);
            hi[k] = make_float4(hx, hy, hz, (float)at.w);
            lo[k] = make_float4(ex, ey, ez, 0.0f);
        }
    }
}

int launch_cell_finish(const double *xyz, const double *r, const int *in_mol, int ncell, const int *cell_start,
                       const int *scattered, const Grid *grids, int *sorted_orig, double4 *atom, int *atom_mol,
                       int *atom_cell, float4 *hi, float4 *lo, cudaStream_t st)
{
    const int nb = (ncell + CELL_WARPS - 1) / CELL_WARPS;
    k_cell_finish<<<nb < 65536 ? nb : 65536, CELL_WARPS * 32, 0, st>>>(xyz, r, in_mol, ncell, cell_start, scattered,
                                                                       grids, sorted_orig, atom, atom_mol, atom_cell,
                                                                       hi, lo);
    return 1;
}

// --------------------------------------------------------------------------
// The atoms of the 27 cells around sorted atom i (in the cells of its own
// molecule) in cell order, one warp: f(j, valid) on every lane, 32 atoms at a
// time.  The three cells along the last axis hold consecutive atoms, so the
// walk is over 9 runs laid end to end (a cell of the globules holds 3 atoms:
// cell by cell, 27 steps of 3 lanes).
// --------------------------------------------------------------------------
template <class F>
__device__ __forceinline__ void warp_neighbour_cells(const Model &M, int i, F f)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const CellGrid &g = M.cg[M.atom_mol[i]];
    const int c = M.atom_cell[i] - g.coff, n1 = g.cn[1], n2 = g.cn[2];
    const int cc = c % n2, cb = (c / n2) % n1, ca = c / (n2 * n1);
    int start = 0, len = 0;
    if (lane < 9) {
        const int a = ca - 1 + lane / 3, b = cb - 1 + lane % 3;
        if (a >= 0 && b >= 0 && a < g.cn[0] && b < n1) {
            const int row = g.coff + (a * n1 + b) * n2;
            start = M.cell_start[row + max(cc - 1, 0)];
            len = M.cell_start[row + min(cc + 1, n2 - 1) + 1] - start;
        }
    }
    int end = len;  // inclusive prefix over the runs
    for (int o = 1; o < 16; o <<= 1) {
        const int v = __shfl_up_sync(full, end, o);
        if (lane >= o) end += v;
    }
    const int total = __shfl_sync(full, end, 8);
    start -= end - len;  // atom of position t in run r: start[r] + t
    for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = t0 + lane;
        int r = 0;
        for (int q = 0; q < 8; ++q) r += t >= __shfl_sync(full, end, q) ? 1 : 0;
        f(__shfl_sync(full, start, r) + t, t < total);
    }
}

constexpr int NB_WARPS = 4;  // warps (atoms) per block of the neighbour and pair kernels

// the circle where expanded spheres (ci, Ri) and (cj, Rj) meet, if any.  Every
// operation is an explicit round-to-nearest intrinsic, so no multiply-add is
// contracted and every inlined copy (count and fill kernels, any path)
// computes the same bits: counts and fills agree, and a circle's bits do not
// depend on where it was computed.  frame_of and cover_of are kept out of
// line for the same reason.
__device__ __forceinline__ bool circle_of(double4 ci, double Ri, double4 cj, double Rj, double3 &o, double3 &u,
                                          double &rho)
{
    const double dx = __dsub_rn(cj.x, ci.x), dy = __dsub_rn(cj.y, ci.y), dz = __dsub_rn(cj.z, ci.z);
    const double D2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double S = __dadd_rn(Ri, Rj);
    if (!(D2 < __dmul_rn(S, S))) return false;
    const double D = __dsqrt_rn(D2);
    if (!(D > fabs(__dsub_rn(Ri, Rj)))) return false;
    const double a = __ddiv_rn(__dsub_rn(__dadd_rn(D2, __dmul_rn(Ri, Ri)), __dmul_rn(Rj, Rj)), __dmul_rn(2.0, D));
    const double rho2 = __dsub_rn(__dmul_rn(Ri, Ri), __dmul_rn(a, a));
    if (!(rho2 > 0.0)) return false;
    u = make_double3(__ddiv_rn(dx, D), __ddiv_rn(dy, D), __ddiv_rn(dz, D));
    o = make_double3(__dadd_rn(ci.x, __dmul_rn(a, u.x)), __dadd_rn(ci.y, __dmul_rn(a, u.y)),
                     __dadd_rn(ci.z, __dmul_rn(a, u.z)));
    rho = __dsqrt_rn(rho2);
    return true;
}

// The circle of atoms i and j, computed from the one with the smaller input
// index (axis from it to the other): the same bits whatever the atoms' places
// in the cell sort, so any model holding both atoms -- a subset of the atoms
// on the same grid included -- has the same circle.
__device__ __forceinline__ bool circle_canon(const Model &M, int i, int j, const double4 &ci, double Ri,
                                             const double4 &cj, double Rj, double3 &o, double3 &u, double &rho)
{
    const bool sw = M.atom_orig[i] > M.atom_orig[j];
    return circle_of(sw ? cj : ci, sw ? Rj : Ri, sw ? ci : cj, sw ? Ri : Rj, o, u, rho);
}

// Sorted atom j next to atom i: 0 the expanded spheres do not overlap, 1 they
// do without meeting in a circle (`within`: ball i lies inside ball j), 2 they
// meet in a circle.  Taken in FP32 from the double-float copies when the
// distance clears every limit by 1e-3 A + 1e-5 S (the copies' difference is
// good to 1e-6 A and the radii to 6e-8 S), else in FP64 with the circle's own
// arithmetic -- FP64 here costs an SM one warp instruction per 16 cycles.
__device__ __forceinline__ int nb_class(const Model &M, int i, int j, const float4 &ih, const float4 &il, bool &within)
{
    const float4 jh = M.atom_hi[j], jl = M.atom_lo[j];
    const float dx = (jh.x - ih.x) + (jl.x - il.x), dy = (jh.y - ih.y) + (jl.y - il.y),
                dz = (jh.z - ih.z) + (jl.z - il.z);
    const float rpf = (float)M.rp, Ri = ih.w + rpf, Rj = jh.w + rpf;
    const float d2 = dx * dx + dy * dy + dz * dz, S = Ri + Rj, m = 1e-3f + 1e-5f * S;
    if (d2 > (S + m) * (S + m)) return 0;
    const float inner = fabsf(Ri - Rj) + m;
    if (S > m && d2 < (S - m) * (S - m) && d2 > inner * inner) return 2;
    const double4 ci = M.atom[i], cj = M.atom[j];
    const double Rd = ci.w + M.rp, Re = cj.w + M.rp;
    const double ex = cj.x - ci.x, ey = cj.y - ci.y, ez = cj.z - ci.z;
    const double D2 = ex * ex + ey * ey + ez * ez, Sd = Rd + Re;
    if (!(D2 < Sd * Sd)) return 0;
    double3 o, u;
    double rho;
    if (circle_canon(M, i, j, ci, Rd, cj, Re, o, u, rho)) return 2;
    if (Re >= Rd && sqrt(D2) <= Re - Rd) within = true;
    return 1;
}

// One warp per atom: neighbours (expanded spheres that overlap), circles,
// circles with later atoms (the atom's pairs), and whether the expanded ball
// lies inside another one.
__global__ void __launch_bounds__(NB_WARPS * 32) k_nb_count(Model M, int *__restrict__ nb_count,
                                                           int *__restrict__ circle_count,
                                                           int *__restrict__ pair_count,
                                                           uint8_t *__restrict__ contained)
{
    const int i = blockIdx.x * NB_WARPS + (threadIdx.x >> 5);
    if (i >= M.n_atoms) return;  // uniform per warp
    const float4 ih = M.atom_hi[i], il = M.atom_lo[i];
    int nb = 0, nc = 0, np = 0;
    bool inside = false;
    warp_neighbour_cells(M, i, [&](int j, bool valid) {
        if (!valid || j == i) return;
        const int k = nb_class(M, i, j, ih, il, inside);
        nb += k > 0 ? 1 : 0;
        nc += k == 2 ? 1 : 0;
        np += k == 2 && j > i ? 1 : 0;
    });
    nb = __reduce_add_sync(0xffffffffu, nb);
    nc = __reduce_add_sync(0xffffffffu, nc);
    np = __reduce_add_sync(0xffffffffu, np);
    inside = __any_sync(0xffffffffu, inside);
    if ((threadIdx.x & 31) == 0) {
        nb_count[i] = nb;
        circle_count[i] = nc;
        pair_count[i] = np;
        contained[i] = inside ? 1 : 0;
    }
}

int launch_nb_count(const Model &M, int *nb_count, int *circle_count, int *pair_count, uint8_t *contained,
                    cudaStream_t st)
{
    if (M.n_atoms <= 0) return 0;
    k_nb_count<<<(M.n_atoms + NB_WARPS - 1) / NB_WARPS, NB_WARPS * 32, 0, st>>>(M, nb_count, circle_count, pair_count,
                                                                              contained);
    return 1;
}

// One warp per atom i: the neighbour list in cell order (the same order as a
// serial walk over the 27 cells), and its pairs -- the circles with neighbours
// j > i -- in that order.
__global__ void __launch_bounds__(NB_WARPS * 32) k_nb_fill(Model M, int *__restrict__ nb_list,
                                                          const int *__restrict__ pair_start,
                                                          int2 *__restrict__ pair_ij)
{
    const int i = blockIdx.x * NB_WARPS + (threadIdx.x >> 5);
    if (i >= M.n_atoms) return;
    const unsigned full = 0xffffffffu, below = (1u << (threadIdx.x & 31)) - 1;
    const float4 ih = M.atom_hi[i], il = M.atom_lo[i];
    int w = M.nb_start[i], wp = pair_start[i];
    warp_neighbour_cells(M, i, [&](int j, bool valid) {
        bool within = false;
        const int k = valid && j != i ? nb_class(M, i, j, ih, il, within) : 0;
        const unsigned m = __ballot_sync(full, k > 0), mp = __ballot_sync(full, k == 2 && j > i);
        if (k > 0) nb_list[w + __popc(m & below)] = j;
        if (k == 2 && j > i) pair_ij[wp + __popc(mp & below)] = make_int2(i, j);
        w += __popc(m);
        wp += __popc(mp);
    });
}

int launch_nb_fill(const Model &M, int *nb_list, const int *pair_start, int2 *pair_ij, cudaStream_t st)
{
    if (M.n_atoms <= 0) return 0;
    k_nb_fill<<<(M.n_atoms + NB_WARPS - 1) / NB_WARPS, NB_WARPS * 32, 0, st>>>(M, nb_list, pair_start, pair_ij);
    return 1;
}

// One thread per pair (full warps of FP64 work): its circle, and the FP32 copies.
__global__ void k_pair_geom(Model M, const Grid *__restrict__ grids, double4 *__restrict__ pair_o,
                            double4 *__restrict__ pair_u, float4 *__restrict__ hi, float4 *__restrict__ lo,
                            float4 *__restrict__ u32)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M.n_pairs) return;
    const int2 ij = M.pair_ij[k];
    const double4 ci = M.atom[ij.x], cj = M.atom[ij.y];
    double3 o = make_double3(0.0, 0.0, 0.0), u = o;
    double rho = 0.0;
    circle_canon(M, ij.x, ij.y, ci, ci.w + M.rp, cj, cj.w + M.rp, o, u, rho);
    pair_o[k] = make_double4(o.x, o.y, o.z, rho);
    pair_u[k] = make_double4(u.x, u.y, u.z, 0.0);
    const double *L = grids[M.atom_mol[ij.x]].lo;
    float hx, hy, hz, ex, ey, ez;
    split_df(o.x - L[0], hx, ex);
    split_df(o.y - L[1], hy, ey);
    split_df(o.z - L[2], hz, ez);
    hi[k] = make_float4(hx, hy, hz, (float)rho);
    lo[k] = make_float4(ex, ey, ez, 0.0f);
    u32[k] = make_float4((float)u.x, (float)u.y, (float)u.z, 0.0f);
}

int launch_pair_geom(const Model &M, const Grid *grids, double4 *pair_o, double4 *pair_u, float4 *hi, float4 *lo,
                     float4 *u32, cudaStream_t st)
{
    if (M.n_pairs <= 0) return 0;
    k_pair_geom<<<(M.n_pairs + 127) / 128, 128, 0, st>>>(M, grids, pair_o, pair_u, hi, lo, u32);
    return 1;
}

// --------------------------------------------------------------------------
// free arcs and free triple points
// --------------------------------------------------------------------------
struct CircleFrame {
    double3 o, u, v1, v2;
    double rho;
};

__device__ __noinline__ CircleFrame frame_of(double4 po, double4 pu)
{
    CircleFrame f;
    f.o = make_double3(po.x, po.y, po.z);
    f.u = make_double3(pu.x, pu.y, pu.z);
    f.rho = po.w;
    // a unit vector normal to u
    double3 t = fabs(f.u.x) > 0.6 ? make_double3(0.0, 1.0, 0.0) : make_double3(1.0, 0.0, 0.0);
    double3 v = make_double3(f.u.y * t.z - f.u.z * t.y, f.u.z * t.x - f.u.x * t.z, f.u.x * t.y - f.u.y * t.x);
    double nv = sqrt(v.x * v.x + v.y * v.y + v.z * v.z);
    f.v1 = make_double3(v.x / nv, v.y / nv, v.z / nv);
    f.v2 = make_double3(f.u.y * f.v1.z - f.u.z * f.v1.y, f.u.z * f.v1.x - f.u.x * f.v1.z,
                        f.u.x * f.v1.y - f.u.y * f.v1.x);
    return f;
}

// Coverage of the circle by ball (ck, Rk): 0 none, 1 partial (end points
// qa, qb returned), 2 the whole circle.
__device__ __noinline__ int cover_of(const CircleFrame &f, double4 ck, double Rk, double3 &qa, double3 &qb)
{
    double dx = ck.x - f.o.x, dy = ck.y - f.o.y, dz = ck.z - f.o.z;
    double d1 = dx * f.v1.x + dy * f.v1.y + dz * f.v1.z;
    double d2 = dx * f.v2.x + dy * f.v2.y + dz * f.v2.z;
    double dd = dx * dx + dy * dy + dz * dz;
    double A = sqrt(d1 * d1 + d2 * d2);
    // |q(phi) - c_k|^2 = rho^2 + |d|^2 - 2 rho A cos(phi - psi); covered iff < R_k^2
    double num = f.rho * f.rho + dd - Rk * Rk;
    double den = 2.0 * f.rho * A;
    if (num >= den) return 0;
    if (num < -den) return 2;
    double T = num / den;
    double s = sqrt(fmax(0.0, 1.0 - T * T));
    double3 ep = make_double3((d1 * f.v1.x + d2 * f.v2.x) / A, (d1 * f.v1.y + d2 * f.v2.y) / A,
                              (d1 * f.v1.z + d2 * f.v2.z) / A);
    double3 en = make_double3(f.u.y * ep.z - f.u.z * ep.y, f.u.z * ep.x - f.u.x * ep.z, f.u.x * ep.y - f.u.y * ep.x);
    qa = make_double3(f.o.x + f.rho * (T * ep.x + s * en.x), f.o.y + f.rho * (T * ep.y + s * en.y),
                      f.o.z + f.rho * (T * ep.z + s * en.z));
    qb = make_double3(f.o.x + f.rho * (T * ep.x - s * en.x), f.o.y + f.rho * (T * ep.y - s * en.y),
                      f.o.z + f.rho * (T * ep.z - s * en.z));
    return 1;
}

__device__ __forceinline__ bool common_nb(const Model &M, int k, int i, int j, double4 cj, double Rj)
{
    if (k == i || k == j) return false;
    double4 ck = M.atom[k];
    double Rk = ck.w + M.rp;
    double dx = ck.x - cj.x, dy = ck.y - cj.y, dz = ck.z - cj.z;
    double S = Rk + Rj;
    return dx * dx + dy * dy + dz * dz < S * S;
}

// the end point q (on sphere k) is free iff no other common neighbour covers it
__device__ __forceinline__ bool endpoint_free(const Model &M, int i, int j, int k, double4 cj, double Rj, double3 q)
{
    for (int t = M.nb_start[i]; t < M.nb_start[i + 1]; ++t) {
        int m = M.nb_list[t];
        if (m == k || !common_nb(M, m, i, j, cj, Rj)) continue;
        double4 cm = M.atom[m];
        double Rm = cm.w + M.rp;
        double dx = q.x - cm.x, dy = q.y - cm.y, dz = q.z - cm.z;
        if (dx * dx + dy * dy + dz * dz < Rm * Rm) return false;
    }
    return true;
}

template <bool EMIT>
__device__ void arcs_of_pair(const Model &M, int p, uint8_t *pair_free, int *vert_count, const int *vert_start,
                             double4 *vert)
{
    int2 ij = M.pair_ij[p];
    const int i = ij.x, j = ij.y;
    CircleFrame f = frame_of(M.pair_o[p], M.pair_u[p]);
    double4 cj = M.atom[j];
    double Rj = cj.w + M.rp;
    bool full = false;
    int n_partial = 0, n_free_end = 0, n_emit = 0;
    int w = EMIT ? vert_start[p] : 0;
    for (int t = M.nb_start[i]; t < M.nb_start[i + 1] && !full; ++t) {
        int k = M.nb_list[t];
        if (!common_nb(M, k, i, j, cj, Rj)) continue;
        double4 ck = M.atom[k];
        double3 qa, qb;
        int c = cover_of(f, ck, ck.w + M.rp, qa, qb);
        if (c == 2) {
            full = true;
        } else if (c == 1) {
            ++n_partial;
            bool fa = endpoint_free(M, i, j, k, cj, Rj, qa);
            bool fb = endpoint_free(M, i, j, k, cj, Rj, qb);
            n_free_end += (int)fa + (int)fb;
            // each triple point is emitted once: from the circle of the triple's two
            // atoms with the smaller input indices (any cell order gives the same bits)
            if (M.atom_orig[k] > M.atom_orig[i] && M.atom_orig[k] > M.atom_orig[j]) {
                if (fa) {
                    if (EMIT) vert[w + n_emit] = make_double4(qa.x, qa.y, qa.z, (double)k);
                    ++n_emit;
                }
                if (fb) {
                    if (EMIT) vert[w + n_emit] = make_double4(qb.x, qb.y, qb.z, (double)k);
                    ++n_emit;
                }
            }
        }
    }
    if (!EMIT) {
        bool has_free = !full && (n_partial == 0 || n_free_end > 0);
        pair_free[p] = has_free ? 1 : 0;
        vert_count[p] = full ? 0 : n_emit;
    }
}

// FP32-filtered form of arcs_of_pair, one warp per circle: the common
// neighbours are cached in FP32 in the circle's frame (from the double-float
// copies: two roundings of the offset), and every decision -- common neighbour, no/partial/full cover,
// end point covered -- is taken in FP32 when it clears its error bound and in
// FP64 otherwise, so the decisions are those of the FP64 form.  FP32 end
// points carry a propagated error bound (the FP64 end point is used when that
// bound exceeds 2e-2 A, or past 2e-4 A when its first-order form may not hold);
// emitted triple points are always computed in FP64 (k_verts).
constexpr int ARC_MAXN = 256;
constexpr int ARC_CODES = 64;  // free end points of one circle listed for k_verts (more: the circle is emitted whole)

// 1: d2 < t^2 certain, 0: d2 >= t^2 certain, -1 undecided (delta: error of the vector)
__device__ __forceinline__ int arc_lt(float d2, float t, float delta)
{
    float t2 = t * t;
    float e = 2.0f * ((2.0f * t + delta) * delta + 1e-6f * t2);
    if (d2 < t2 - e) return 1;
    if (d2 >= t2 + e) return 0;
    return -1;
}

// The lanes gather the common neighbours (ballot compaction, list order;
// circles with more than ARC_MAXN take the FP64 form on one lane), then each
// lane takes candidates a = lane, lane + 32, ...: its cover of the circle, its
// end points and their freeness against every other candidate.  Emitted triple points keep the order (a, end point):
// the count pass lists them (2 k + end point) for k_verts, which computes them one thread each.
// Bound by issue and the latency of the neighbours' loads.  FP64 (one warp
// instruction per 16 cycles per SM) is left to end points that FP32 cannot
// decide (with FP64 end points past a bound of 2e-4 A about one lane in two
// circles took them: 2.0 ms on 5,000 atoms at 0.1 atoms/A^3, 1.4 ms on 32
// molecules at h 0.5).  Half the candidates of a circle cover nothing of it and
// are dropped as they are gathered (614 and 520 us); a circle covered whole by
// one ends there (two in three in the dense box), one covered all around by
// several before any end point is tested against the others, and blocks are
// one warp, so a long circle holds up no other warp's registers (410 and 537 us
// with four): 337 and 445 us.
constexpr int ARC_WARPS = 1;
constexpr int ARC_CTAS = 32;  // resident blocks asked for: 64 registers, the FP64 fallbacks' values spilled (106: 16)

struct ArcWarp {
    float4 nb[ARC_MAXN];
    int nbk[ARC_MAXN];
    int code[ARC_CODES];
};

// FP32 end points of a candidate's cover of the circle, in the circle's plane
// (c: its centre there, num, en + ed; see below): status 1 partial for certain
// with end points within dq (e = 0 counterclockwise of the centre, e = 1
// clockwise), 0 it covers nothing for certain, -1 FP64 decides.
struct ArcEnds {
    float q1[2], q2[2], dq;
    float gap;  // half the distance between the end points (0: unknown)
    int status;
};
__device__ __forceinline__ ArcEnds arc_ends(float4 c, float rho, float dlt)
{
    ArcEnds r;
    r.q1[0] = r.q1[1] = r.q2[0] = r.q2[1] = 0.0f;
    r.dq = 1.0f;
    r.gap = 0.0f;
    const float A = sqrtf(c.x * c.x + c.y * c.y);
    const float num = c.z, den = 2.0f * rho * A, err = 2.0f * c.w;
    if (num >= den + err) {
        r.status = 0;
    } else if (!(num < den - err && num > -den + err)) {
        r.status = -1;
    } else {
        const float T = num / den;
        const float sT = sqrtf(fmaxf(0.0f, 1.0f - T * T));
        const float iA = 1.0f / A, e1 = c.x * iA, e2 = c.y * iA;
        for (int e = 0; e < 2; ++e) {
            const float sg = e == 0 ? sT : -sT;
            r.q1[e] = rho * (T * e1 - sg * e2);
            r.q2[e] = rho * (T * e2 + sg * e1);
        }
        // (c.w bounds num's error and den's together, so also |T| of den's)
        const float dT = c.w / den;
        float dq = rho * (dT * (1.0f + fabsf(T) / fmaxf(sT, 1e-6f)) + 2.0f * (dlt / fmaxf(A, 1e-6f) + 3e-7f)) + 1e-6f;
        // past 2e-4 A the bound still holds to a tenth while dT << sT^2 (the second-order part of
        // the end point's shift is dT / (2 sT^2) of the first-order one)
        if (dq > 2e-4f) dq = dT < 0.05f * sT * sT && dq < 1.8e-2f ? 1.1f * dq : 1.0f;
        r.dq = dq;
        r.gap = rho * sT;
        r.status = dq > 2e-2f ? -1 : 1;
    }
    return r;
}

// place of a circle point on 64 bins of the circle, increasing counterclockwise
// (the diamond angle y / (|x| + |y|), unrolled over the half planes; at most
// one bin for 1/16 of the circle's radius along the circle)
__device__ __forceinline__ float circle_bin(float x, float y)
{
    const float p = __fdividef(y, fabsf(x) + fabsf(y));
    return 16.0f * (x >= 0.0f ? 1.0f + p : 3.0f - p);
}

template <bool EMIT>
__device__ int arcs_of_pair_warp(const Model &M, int p, ArcWarp &W, uint8_t *pair_free, int *vert_count,
                                  const int *vert_start, double4 *vert)
{
    const unsigned full_mask = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int2 ij = M.pair_ij[p];
    const int i = ij.x, j = ij.y;
    const float4 oh = M.pair_hi[p], ol = M.pair_lo[p], u4 = M.pair_u32[p];
    const float rho = oh.w;
    const float ux = u4.x, uy = u4.y, uz = u4.z;
    const float tx = fabsf(ux) > 0.6f ? 0.0f : 1.0f, ty = fabsf(ux) > 0.6f ? 1.0f : 0.0f;
    float v1x = -uz * ty, v1y = uz * tx, v1z = ux * ty - uy * tx;
    const float iv1 = 1.0f / sqrtf(v1x * v1x + v1y * v1y + v1z * v1z);
    v1x *= iv1; v1y *= iv1; v1z *= iv1;
    const float v2x = uy * v1z - uz * v1y, v2y = uz * v1x - ux * v1z, v2z = ux * v1y - uy * v1x;
    const float dlt = 3e-6f;
    const float4 jh = M.atom_hi[j], jl = M.atom_lo[j];
    const float djx = (jh.x - oh.x) + (jl.x - ol.x), djy = (jh.y - oh.y) + (jl.y - ol.y),
                djz = (jh.z - oh.z) + (jl.z - ol.z);
    const float rpf = (float)M.rp;
    const float Rj = jh.w + rpf;
    CircleFrame f;
    bool have64 = false;
    // 1. The common neighbours that could cover part of the circle, in list
    //    order.  One that covers the whole circle ends the work at once (at
    //    protein packing most circles are buried this way): FP64 when undecided.
    //    Each is left in the circle's plane: its centre (d1, d2), num
    //    = rho^2 + |d|^2 - R^2 (a circle point q is covered iff 2 q.d > num)
    //    and the error bound en + ed of either side.
    //    One that certainly covers nothing of the circle is dropped: it covers
    //    no end point either.
    bool full = false;
    float amax = 0.0f, emax = 0.0f;  // the lanes' largest |(d1, d2)| and error bound
    int n = 0;
    const int t_end = M.nb_start[i + 1];
    int t = M.nb_start[i] + lane;
    int k_next = t < t_end ? M.nb_list[t] : j;
    for (int t0 = t - lane; t0 < t_end && !full; t0 += 32) {
        const int k = k_next;
        t += 32;
        k_next = t < t_end ? M.nb_list[t] : j;
        bool whole = false, keep = false;
        float4 flat = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k != j) {
            const float4 kh = M.atom_hi[k], kl = M.atom_lo[k];
            const float dx = (kh.x - oh.x) + (kl.x - ol.x), dy = (kh.y - oh.y) + (kl.y - ol.y),
                        dz = (kh.z - oh.z) + (kl.z - ol.z);
            const float Rk = kh.w + rpf;
            const float ex = dx - djx, ey = dy - djy, ez = dz - djz;
            const int cm = arc_lt(ex * ex + ey * ey + ez * ez, Rk + Rj, 2.0f * dlt);
            if (cm != 0) {
                const float d1 = dx * v1x + dy * v1y + dz * v1z;
                const float d2 = dx * v2x + dy * v2y + dz * v2z;
                const float dd = dx * dx + dy * dy + dz * dz;
                const float A = sqrtf(d1 * d1 + d2 * d2);
                const float num = rho * rho + dd - Rk * Rk, den = 2.0f * rho * A;
                const float dk = sqrtf(dd);
                const float en = 2.0f * dk * dlt + 2e-6f * (rho * rho + dd + Rk * Rk);
                const float ed = 2.0f * rho * (dlt + 3e-7f * dk) + 2e-6f * den;
                const float err = 2.0f * (en + ed);
                keep = num < den + err;
                if (keep && cm < 0) {
                    const double4 cj = M.atom[j];
                    keep = common_nb(M, k, i, j, cj, cj.w + M.rp);
                }
                if (keep) {
                    flat = make_float4(d1, d2, num, en + ed);
                    amax = fmaxf(amax, A);
                    emax = fmaxf(emax, en + ed);
                    if (num < -den - err) {
                        whole = true;
                    } else if (num < -den + err) {  // undecided near a whole cover: FP64
                        if (!have64) {
                            f = frame_of(M.pair_o[p], M.pair_u[p]);
                            have64 = true;
                        }
                        const double4 ck = M.atom[k];
                        double3 qa, qb;
                        whole = cover_of(f, ck, ck.w + M.rp, qa, qb) == 2;
                    }
                }
            }
        }
        full = __any_sync(full_mask, whole);
        const unsigned m = __ballot_sync(full_mask, keep);
        const int pos = n + __popc(m & ((1u << lane) - 1));
        if (keep && pos < ARC_MAXN) {
            W.nb[pos] = flat;
            W.nbk[pos] = k;
        }
        n += __popc(m);
    }
    __syncwarp();
    if (!full && n > ARC_MAXN) {  // very crowded circle: the FP64 form, one lane
        int listed = 0;
        if (lane == 0) {
            arcs_of_pair<EMIT>(M, p, pair_free, vert_count, vert_start, vert);
            if (!EMIT && vert_count[p] > 0) listed = ARC_CODES + 1;  // emitted whole
        }
        return __shfl_sync(full_mask, listed, 0);
    }
    // 2. The bins of the circle that some candidate covers for certain: no end
    //    point in them is free, and a circle covered all around is buried
    //    without any end point tested against the others.
    unsigned cov_lo = 0u, cov_hi = 0u;
    for (int r = 0; r * 32 < n && !full; ++r) {
        unsigned long long bins = 0ull;
        if (r * 32 + lane < n) {
            const ArcEnds a = arc_ends(W.nb[r * 32 + lane], rho, dlt);
            const float eps = 16.5f * a.dq / rho + 1e-3f;
            // (end points further apart than their errors, so that their order on the circle is known)
            if (a.status == 1 && eps < 0.5f && a.gap > 4.0f * a.dq) {
                const float b0 = circle_bin(a.q1[0], a.q2[0]), b1 = circle_bin(a.q1[1], a.q2[1]);
                const int first = (int)ceilf(b1 + eps), last = (int)floorf((b0 < b1 ? b0 + 64.0f : b0) - eps);
                const int len = min(last - first, 63);
                if (len > 0) {
                    const unsigned long long ones = (1ull << len) - 1ull;
                    const int sh = first & 63;
                    bins = (ones << sh) | (sh ? ones >> (64 - sh) : 0ull);
                }
            }
        }
        cov_lo |= __reduce_or_sync(full_mask, (unsigned)bins);
        cov_hi |= __reduce_or_sync(full_mask, (unsigned)(bins >> 32));
    }
    if (full || (cov_lo & cov_hi) == 0xffffffffu) {
        if (!EMIT && lane == 0) {
            pair_free[p] = 0;
            vert_count[p] = 0;
        }
        return 0;
    }
    const unsigned long long covered = ((unsigned long long)cov_hi << 32) | cov_lo;
    for (int o = 16; o > 0; o >>= 1) {
        amax = fmaxf(amax, __shfl_xor_sync(full_mask, amax, o));
        emax = fmaxf(emax, __shfl_xor_sync(full_mask, emax, o));
    }
    __syncwarp();
    // 3. candidates a = lane + 32 r: covers, end points and their freeness.  An
    //    end point q (in the plane) outside the covered bins is tested against
    //    every other candidate with two multiply-adds and one bound for all of
    //    them: 2 q.d - num against 2 |dq| max |d| + 2 max(en + ed).  Only an end
    //    point that no candidate covers for certain and some could is taken to
    //    FP64.
    int n_partial = 0, n_free_end = 0, n_emit_total = 0;
    const int w0 = EMIT ? vert_start[p] : 0;
    for (int r = 0; r * 32 < n; ++r) {
        const int a = r * 32 + lane;
        int status = 0;  // 0 none, 1 partial, 2 full
        bool fr[2] = {false, false}, open[2] = {true, true};
        double3 qe[2];
        bool e64 = false;
        if (a < n) {
            const ArcEnds ar = arc_ends(W.nb[a], rho, dlt);
            float q1[2] = {ar.q1[0], ar.q1[1]}, q2[2] = {ar.q2[0], ar.q2[1]};
            float dq = ar.dq;
            status = ar.status;
            if (status < 0) {  // undecided cover or loose FP32 end points: FP64
                if (!have64) {
                    f = frame_of(M.pair_o[p], M.pair_u[p]);
                    have64 = true;
                }
                const double4 ck = M.atom[W.nbk[a]];
                const int cov = cover_of(f, ck, ck.w + M.rp, qe[0], qe[1]);
                status = cov;
                if (cov == 1) {
                    for (int e = 0; e < 2; ++e) {
                        const float qx = (float)(qe[e].x - f.o.x), qy = (float)(qe[e].y - f.o.y),
                                    qz = (float)(qe[e].z - f.o.z);
                        q1[e] = qx * v1x + qy * v1y + qz * v1z;
                        q2[e] = qx * v2x + qy * v2y + qz * v2z;
                    }
                    dq = 1e-6f + 1e-6f * rho;
                    e64 = true;
                }
            }
            if (status == 1) {
                const float eps = 16.5f * dq / rho + 1e-3f;
                for (int e = 0; e < 2 && eps < 0.5f; ++e) {
                    const float b = circle_bin(q1[e], q2[e]);
                    const int lo = (int)floorf(b - eps) & 63, hi = (int)floorf(b + eps) & 63;
                    open[e] = !((covered >> lo) & (covered >> hi) & 1ull);
                }
            }
            if (status == 1 && (open[0] || open[1])) {
                const float E = 2.0f * (dq * amax + emax);
                bool cov0 = !open[0], cov1 = !open[1], und0 = false, und1 = false;
                const float x0 = 2.0f * q1[0], y0 = 2.0f * q2[0], x1 = 2.0f * q1[1], y1 = 2.0f * q2[1];
                for (int b = 0; b < n && !(cov0 && cov1); ++b) {
                    const float4 cb = W.nb[b];
                    const float g0 = fmaf(x0, cb.x, fmaf(y0, cb.y, -cb.z)), g1 = fmaf(x1, cb.x, fmaf(y1, cb.y, -cb.z));
                    if (b == a) continue;
                    cov0 = cov0 || g0 > E;
                    cov1 = cov1 || g1 > E;
                    und0 = und0 || g0 >= -E;
                    und1 = und1 || g1 >= -E;
                }
                fr[0] = !cov0;
                fr[1] = !cov1;
                for (int e = 0; e < 2; ++e) {
                    if (!(fr[e] && (e == 0 ? und0 : und1))) continue;
                    if (!e64) {  // the exact end point against the exact balls that could cover it
                        if (!have64) {
                            f = frame_of(M.pair_o[p], M.pair_u[p]);
                            have64 = true;
                        }
                        const double4 ck = M.atom[W.nbk[a]];
                        cover_of(f, ck, ck.w + M.rp, qe[0], qe[1]);
                        e64 = true;
                    }
                    for (int b = 0; b < n && fr[e]; ++b) {
                        const float4 cb = W.nb[b];
                        if (b == a || 2.0f * (q1[e] * cb.x + q2[e] * cb.y) - cb.z < -1.5f * E) continue;
                        const double4 c64 = M.atom[W.nbk[b]];
                        const double Rb = c64.w + M.rp;
                        const double gx = qe[e].x - c64.x, gy = qe[e].y - c64.y, gz = qe[e].z - c64.z;
                        if (gx * gx + gy * gy + gz * gz < Rb * Rb) fr[e] = false;
                    }
                }
            }
        }
        full = full || __any_sync(full_mask, status == 2);
        if (full) break;  // uniform
        int np_ = status == 1 ? 1 : 0, nf_ = (int)fr[0] + (int)fr[1];
        // emitted once: from the circle of the two atoms with the smaller input indices
        const bool emits = status == 1 && a < n && M.atom_orig[W.nbk[a]] > M.atom_orig[i] &&
                           M.atom_orig[W.nbk[a]] > M.atom_orig[j];
        int ne_ = emits ? nf_ : 0;
        // inclusive scan of ne_ over the lanes (the serial order a = 0, 1, ...)
        int inc = ne_;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full_mask, inc, o);
            if (lane >= o) inc += u;
        }
        const int tot = __shfl_sync(full_mask, inc, 31);
        if (!EMIT && ne_ > 0) {
            int at = n_emit_total + inc - ne_;
            for (int e = 0; e < 2; ++e)
                if (fr[e]) {
                    if (at < ARC_CODES) W.code[at] = 2 * W.nbk[a] + e;
                    ++at;
                }
        }
        if (EMIT && ne_ > 0) {
            if (!e64) {
                if (!have64) {
                    f = frame_of(M.pair_o[p], M.pair_u[p]);
                    have64 = true;
                }
                const double4 ck = M.atom[W.nbk[a]];
                cover_of(f, ck, ck.w + M.rp, qe[0], qe[1]);
            }
            int wpos = w0 + n_emit_total + inc - ne_;
            const double kw = (double)W.nbk[a];  // the triple's third atom
            for (int e = 0; e < 2; ++e)
                if (fr[e]) vert[wpos++] = make_double4(qe[e].x, qe[e].y, qe[e].z, kw);
        }
        n_emit_total += tot;
        for (int o = 16; o > 0; o >>= 1) {
            np_ += __shfl_xor_sync(full_mask, np_, o);
            nf_ += __shfl_xor_sync(full_mask, nf_, o);
        }
        n_partial += np_;
        n_free_end += nf_;
    }
    if (!EMIT && lane == 0) {
        const bool has_free = !full && (n_partial == 0 || n_free_end > 0);
        pair_free[p] = has_free ? 1 : 0;
        vert_count[p] = full ? 0 : n_emit_total;
    }
    __syncwarp();
    return full ? 0 : n_emit_total;
}

// Free end points to emit, listed while their circle is at hand: entry (circle,
// third atom, end point, place among the circle's).  A circle with more than
// ARC_CODES, or whose run does not fit the list, goes to `whole`.
__global__ void __launch_bounds__(ARC_WARPS * 32, ARC_CTAS) k_arcs(Model M, uint8_t *__restrict__ pair_free,
                                                         int *__restrict__ vert_count, ArcList L)
{
    __shared__ ArcWarp W[ARC_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = blockIdx.x * ARC_WARPS + warp;
    if (p >= M.n_pairs) return;  // uniform per warp
    const int n = arcs_of_pair_warp<false>(M, p, W[warp], pair_free, vert_count, nullptr, nullptr);
    if (n == 0) return;
    int off = L.cap;
    if (lane == 0 && n <= ARC_CODES) off = atomicAdd(L.n, n);
    off = __shfl_sync(0xffffffffu, off, 0);
    const bool fits = n <= ARC_CODES && off >= 0 && off <= L.cap - n;
    if (!fits && lane == 0) L.whole[atomicAdd(L.n + 1, 1)] = p;
    for (int k = lane; k < n && off >= 0 && off + k < L.cap; k += 32)  // (a slot no run fills is dead)
        L.e[off + k] = fits ? make_int4(p, W[warp].code[k] >> 1, W[warp].code[k] & 1, k) : make_int4(-1, 0, 0, 0);
}

// one triple point's molecule, atoms and FP32 copies
__device__ __forceinline__ void vert_out(const Model &M, const VertOut &O, const double4 &v, int2 ij, int at)
{
    const int mol = M.atom_mol[ij.x];
    O.mol[at] = mol;
    O.atoms[at] = make_int4(ij.x, ij.y, (int)v.w, 0);
    const double *L = O.grids[mol].lo;
    float hx, hy, hz, ex, ey, ez;
    split_df(v.x - L[0], hx, ex);
    split_df(v.y - L[1], hy, ey);
    split_df(v.z - L[2], hz, ez);
    O.hi[at] = make_float4(hx, hy, hz, 0.0f);
    O.lo[at] = make_float4(ex, ey, ez, 0.0f);
}

// The listed triple points in FP64, one thread each (full warps of FP64 work;
// a warp per circle with a lane or two in FP64 took 0.77 ms for 64,000 points).
__global__ void __launch_bounds__(128) k_verts(Model M, const int *__restrict__ vert_start, ArcList L, VertOut O)
{
    const int n = min(*L.n, L.cap);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int4 e = L.e[q];
        if (e.x < 0) continue;
        const CircleFrame f = frame_of(M.pair_o[e.x], M.pair_u[e.x]);
        const double4 ck = M.atom[e.y];
        double3 qe[2];
        cover_of(f, ck, ck.w + M.rp, qe[0], qe[1]);
        const double3 x = e.z ? qe[1] : qe[0];
        const int at = vert_start[e.x] + e.w;
        const double4 v = make_double4(x.x, x.y, x.z, (double)e.y);
        O.vert[at] = v;
        vert_out(M, O, v, M.pair_ij[e.x], at);
    }
}

// the circles that were not listed: a warp each emits its triple points
__global__ void __launch_bounds__(ARC_WARPS * 32) k_arcs_emit(Model M, const int *__restrict__ vert_start, ArcList L,
                                                              VertOut O)
{
    __shared__ ArcWarp W[ARC_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = L.n[1];
    for (int q = blockIdx.x * ARC_WARPS + warp; q < n; q += gridDim.x * ARC_WARPS) {
        const int p = L.whole[q];
        arcs_of_pair_warp<true>(M, p, W[warp], nullptr, nullptr, vert_start, O.vert);
        __syncwarp();
        for (int k = vert_start[p] + lane; k < vert_start[p + 1]; k += 32) vert_out(M, O, O.vert[k], M.pair_ij[p], k);
        __syncwarp();
    }
}

int launch_arcs(const Model &M, uint8_t *pair_free, int *vert_count, const ArcList &L, cudaStream_t st)
{
    if (M.n_pairs <= 0) return 0;
    k_arcs<<<(M.n_pairs + ARC_WARPS - 1) / ARC_WARPS, ARC_WARPS * 32, 0, st>>>(M, pair_free, vert_count, L);
    return 1;
}

int launch_arcs_emit(const Model &M, const int *vert_start, const ArcList &L, const VertOut &O, cudaStream_t st)
{
    if (M.n_verts <= 0) return 0;
    k_verts<<<(M.n_verts + 127) / 128, 128, 0, st>>>(M, vert_start, L, O);
    k_arcs_emit<<<std::min(64, (M.n_pairs + ARC_WARPS - 1) / ARC_WARPS), ARC_WARPS * 32, 0, st>>>(M, vert_start, L, O);
    return 2;
}

__global__ void k_faces_init(int n, const int *__restrict__ circle_count, const uint8_t *__restrict__ contained,
                             uint8_t *__restrict__ face)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    face[i] = (circle_count[i] == 0 && !contained[i]) ? 1 : 0;
}

__global__ void k_faces_pairs(Model M, uint8_t *__restrict__ face)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M.n_pairs) return;
    if (M.pair_free[p]) {
        int2 ij = M.pair_ij[p];
        face[ij.x] = 1;
        face[ij.y] = 1;
    }
}

int launch_faces(const Model &M, const int *circle_count, const uint8_t *contained, uint8_t *face, cudaStream_t st)
{
    int nl = 0;
    if (M.n_atoms > 0) ++nl, k_faces_init<<<(M.n_atoms + 255) / 256, 256, 0, st>>>(M.n_atoms, circle_count, contained, face);
    if (M.n_pairs > 0) ++nl, k_faces_pairs<<<(M.n_pairs + 255) / 256, 256, 0, st>>>(M, face);
    return nl;
}

// which = 0: free-arc pairs by circle centre; which = 1: free triple points
// cull: bin only the circles that keep a free arc (buried saddle patches are
// culled before the classification); without it every circle is binned
__global__ void k_bin_count(Model M, int which, bool cull, int *__restrict__ count, int *__restrict__ item_cell)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    int n = which == 0 ? M.n_pairs : M.n_verts;
    if (p >= n) return;
    double x, y, z;
    int mol;
    if (which == 0) {
        if (cull && !M.pair_free[p]) {
            item_cell[p] = -1;
            return;
        }
        double4 o = M.pair_o[p];
        x = o.x; y = o.y; z = o.z;
        mol = M.atom_mol[M.pair_ij[p].x];
    } else {
        double4 v = M.vert[p];
        x = v.x; y = v.y; z = v.z;
        mol = M.vert_mol[p];
    }
    int id = cell_of(M.cg[mol], M.cell, x, y, z);
    item_cell[p] = id;
    atomicAdd(&count[id], 1);
}

__global__ void k_bin_scatter(int n, const int *__restrict__ item_cell, const int *__restrict__ start,
                              int *__restrict__ cursor, int *__restrict__ list)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    int id = item_cell[p];
    if (id < 0) return;
    list[start[id] + atomicAdd(&cursor[id], 1)] = p;
}

int launch_bin_count(const Model &M, int which, bool cull, int *count, int *item_cell, cudaStream_t st)
{
    int n = which == 0 ? M.n_pairs : M.n_verts;
    if (n <= 0) return 0;
    k_bin_count<<<(n + 255) / 256, 256, 0, st>>>(M, which, cull, count, item_cell);
    return 1;
}

int launch_bin_scatter(const Model &M, int which, const int *item_cell, const int *start, int *cursor, int *list,
                        cudaStream_t st)
{
    int n = which == 0 ? M.n_pairs : M.n_verts;
    if (n <= 0) return 0;
    k_bin_scatter<<<(n + 255) / 256, 256, 0, st>>>(n, item_cell, start, cursor, list);
    return 1;
}

}  // namespace eses
