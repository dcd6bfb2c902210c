// eses_classify.cu -- grid-point classification kernels (the second ESES
// stage, Eq. 2), one CTA per 8x8x8 tile.
//
// k_classify<T, FILT>:
//   1. stages the tile's atoms, free-arc pairs and free triple points in
//      shared memory (tile frame);
//   2. splits the tile into 16 bricks of 2x4x4 points, one warp per brick:
//      the lanes test the staged atoms against the brick's box and ballots
//      give the set of atoms whose expanded ball reaches the brick.  A warp
//      with an empty set labels its 32 points outside at once; otherwise every
//      lane tests its point against the set: inside a van der Waals ball -> 1,
//      in no expanded ball -> 0, else a shell point;
//   3. shell points go to a per-tile queue, brick by brick; when there are
//      any, the block builds the staged atoms' neighbour sets (expanded spheres
//      that meet) and works through the queue, a warp at a time on neighbouring
//      points (shell_points): free triple points within r_p, convex witnesses
//      of the containing balls, saddle witnesses of the circles near the warp's
//      points, each witness tested for freeness against the neighbours of its
//      atoms only.
//   Bound by instruction issue and the latency of a tile's slowest points.  One
//   thread per point walking its own balls' circles (12.9 active lanes, 65 % of
//   the kernel in this phase, 59,000 cycles a tile on the 5,000-atom globule at
//   h 0.25) became all lanes on one patch at a time: 2.19 -> 1.12 ms there,
//   8.2 -> 4.4 ms at 20,000 atoms, 3.6 -> 1.75 ms on 32 molecules at h 0.5,
//   1.30 -> 0.64 ms in FP64 on 200 atoms (single-tile queue pops, staging by
//   runs of cells and five CTAs an SM included).
//   T = double, FILT = false is the plain FP64 form; T = float, FILT = true
//   is the filtered form, whose undecided points get LABEL_BAND and whose
//   tiles with such points are listed.
// k_band: re-labels the undecided points of the tiles that have any, in FP64:
//   one warp per point runs the witness search over every staged item.
#include <algorithm>

#include "eses_kernels.h"
#include "eses_tile.cuh"

namespace eses {

constexpr int CLS_THREADS = 256;
constexpr int NBRICK = 16;     // 2x4x4-point bricks per tile
// lanes per shell point: doubled while points x lanes stays within this (one
// lane per point above it), so a tile of few points still uses its warps.
// Measured at 256 / 512 / 1,024: 1.61 / 1.39 / 1.54 ms on the 5,000-atom globule
// (216 points a tile), 2.74 / 2.30 / 2.36 ms at h 0.5
constexpr int CLS_SPLIT = 2 * CLS_THREADS;

template <class CP>
struct ClsSmem {
    static constexpr int HS = slot_hash_size<CP>(), AWC = atom_words<CP>();
    short2 pslot[CP::P];           // staged slots of each pair's atoms (-1: not staged)
    unsigned bmask[NBRICK][AWC];   // per-brick sets of the atoms whose expanded ball reaches the brick
    unsigned nbm[CP::A * AWC];     // neighbour set of every staged atom (build_neighbour_sets); before that
                                   // the staged-atom lookup of pair_slots (HS keys, HS slots)
    static_assert(CP::A * AWC * sizeof(unsigned) >= HS * (sizeof(int) + sizeof(short)), "lookup in nbm");
    short queue[TILE_PTS];         // shell points, brick by brick
    int nq, band, next;            // queue length, band points, next queue position to take
};

// a tile that overflowed the shared-memory staging goes to the list of the
// global-memory tier: ovf[0] counts such tiles over the run, ovf[1] is the
// stage's list length, ovf[2..] the global tiles
__device__ __forceinline__ void ovf_push(int *ovf, long long gt)
{
    atomicAdd(&ovf[0], 1);
    const int k = atomicAdd(&ovf[1], 1);
    ovf[2 + k] = (int)gt;
}

__device__ __forceinline__ void brick_point(int brick, int lane, int &li, int &lj, int &lk)
{
    int bi = brick >> 2, bj = (brick >> 1) & 1, bk = brick & 1;
    li = bi * 2 + (lane >> 4);
    lj = bj * 4 + ((lane >> 2) & 3);
    lk = bk * 4 + (lane & 3);
}

// tile-frame coordinate of local point k: FP32 table, or FP64 k * h
template <class T>
__device__ __forceinline__ T pt_coord(const Grid &G, int k)
{
    if constexpr (sizeof(T) == sizeof(float)) return G.hl[k];
    else return (double)k * G.h;
}

// Freeness of a witness against the staged atoms in m0 & m1 (m1 may be null),
// as free_set, inlined: the lanes of a warp test witnesses of one patch, so
// they walk the same atoms.
template <bool FILT, class T, class CP>
__device__ __forceinline__ int witness_free(const TileS<T, CP> &S, T qx, T qy, T qz, const unsigned *m0,
                                            const unsigned *m1, int nw, T rp, T Rmax, T delta, int &nt)
{
    int res = 1;
    const T e = FILT ? T(2) * ((T(2) * Rmax + delta) * delta + T(1e-6) * Rmax * Rmax) : T(0);  // lt_sq's bound at R_max
    for (int w = 0; w < nw; ++w) {
        unsigned bits = m1 ? (m0[w] & m1[w]) : m0[w];
        while (bits) {
            const int k = (w << 5) + __ffs(bits) - 1;
            bits &= bits - 1;
            ++nt;
            const P4<T> c = S.atom[k];
            const T dx = qx - c.x, dy = qy - c.y, dz = qz - c.z;
            const T R = c.w + rp, g = dx * dx + dy * dy + dz * dz - R * R;
            if (FILT ? g < -e : dx * dx + dy * dy + dz * dz < R * R) return 0;
            if (FILT && g < e) res = -1;
        }
    }
    return res;
}

// Shell points of one warp: 32 / G points, G lanes (a power of two) each;
// `code` is the lane's queue entry (-1: none), (x, y, z) its point, r its rank
// among the point's lanes.  Every patch that could hold a witness of some
// point of the warp is taken in turn, triple points, then convex, then
// saddle patches: lanes test their own point against the same patch, so its
// data and the atoms that could cover its witness are broadcast reads and the
// lanes stay together (rank r of G takes every G-th patch).  Circles are
// first culled against the box of the points still undecided, lanes over
// circles; a circle that meets no containing ball of a point is no nearer
// than r_p with a free witness unless the point is outside, so testing it
// changes no decision.  df: FP32 error bound of a staged difference (also in
// the FP64 form, whose cull is FP32).  Returns the point's label on each of its lanes:
// 0 a free witness within r_p (certain), 2 undecided, 1 none.
template <bool FILT, class T, class CP>
__device__ __forceinline__ int shell_points(const TileS<T, CP> &S, const ClsSmem<CP> &C, int code, T x, T y, T z, T rp,
                                            T Rmax, T d0, float hf, float df, int r, int G, int &nt)
{
    constexpr unsigned full = 0xffffffffu;
    constexpr int aw = ClsSmem<CP>::AWC;
    const int lane = threadIdx.x & 31;
    const SmemAcc<T, CP> A(S);
    // every G-th bit from r: this lane's share of a 32-patch word
    const unsigned share = (G == 32 ? 1u : full / ((1u << G) - 1u)) << r;
    const unsigned gmask = (G == 32 ? full : ((1u << G) - 1u)) << (lane & ~(G - 1));
    bool done = code < 0, hit = false, unsure = false;
    // a point is settled once any of its lanes has a witness
    auto settle = [&]() {
        const unsigned h = __ballot_sync(full, hit);  // every lane votes
        done = done || (h & gmask) != 0u;
        return __all_sync(full, done);
    };
    const T rp2 = rp * rp;
    for (int v = r; v < S.nv && !done; v += G) {
        const P4<T> q = S.vq[v];
        const T dx = x - q.x, dy = y - q.y, dz = z - q.z;
        const int t = lt_sq<FILT>(dx * dx + dy * dy + dz * dz, rp2, rp, d0);
        if (t == 1) hit = done = true;
        else if (t < 0) unsure = true;
    }
    const int nw = (S.na + 31) >> 5;
    if (!settle()) {
        // convex patches of the balls that reach the points' bricks
        const unsigned *bm = C.bmask[(code >> 9) & 15];
        for (int wd = 0; wd < nw; ++wd) {
            unsigned bits = __reduce_or_sync(full, done ? 0u : bm[wd]) & share;
            while (bits && !done) {
                const int a = (wd << 5) + __ffs(bits) - 1;
                bits &= bits - 1;
                T qx, qy, qz, dq;
                int e0, e1;
                const int tw = face_proposal<FILT>(A, a, x, y, z, rp, rp, d0, qx, qy, qz, dq, e0, e1);
                if (tw == 0) continue;
                if (tw == -2) {
                    unsure = true;
                    continue;
                }
                const int f = witness_free<FILT>(S, qx, qy, qz, C.nbm + a * aw, (const unsigned *)nullptr, nw, rp,
                                                 Rmax, dq + d0, nt);
                if (f == 1 && tw == 1) hit = done = true;
                else if (f != 0) unsure = true;
            }
        }
    }
    if (!settle()) {
        // box of the undecided points, then the circles that come within r_p of it
        const int li = (code >> 6) & 7, lj = (code >> 3) & 7, lk = code & 7;
        const int i0 = __reduce_min_sync(full, done ? 8 : li), i1 = __reduce_max_sync(full, done ? -1 : li);
        const int j0 = __reduce_min_sync(full, done ? 8 : lj), j1 = __reduce_max_sync(full, done ? -1 : lj);
        const int k0 = __reduce_min_sync(full, done ? 8 : lk), k1 = __reduce_max_sync(full, done ? -1 : lk);
        const float hh = 0.5f * hf;
        const float cx = hh * (float)(i0 + i1), cy = hh * (float)(j0 + j1), cz = hh * (float)(k0 + k1);
        const float ex = (float)(i1 - i0), ey = (float)(j1 - j0), ez = (float)(k1 - k0);
        // 4 df covers the FP32 rounding of the distance at the molecule's lengths (2e-3 A alone does not for
        // radii of 1e4 A)
        const float reach = (float)rp + hh * sqrtf(ex * ex + ey * ey + ez * ez) + 2e-3f + 4.0f * df;
        for (int p0 = 0; p0 < S.np; p0 += 32) {
            bool near = false;
            if (p0 + lane < S.np) {
                const P4<T> o = S.po[p0 + lane], u = S.pu[p0 + lane];
                const short2 sl = C.pslot[p0 + lane];
                const float yx = cx - (float)o.x, yy = cy - (float)o.y, yz = cz - (float)o.z;
                const float ux = (float)u.x, uy = (float)u.y, uz = (float)u.z;
                const float zc = yx * ux + yy * uy + yz * uz;
                const float wx = yx - zc * ux, wy = yy - zc * uy, wz = yz - zc * uz;
                const float e = sqrtf(wx * wx + wy * wy + wz * wz) - (float)o.w;
                // (an atom that is not staged is too far for the circle's points near the tile)
                near = e * e + zc * zc < reach * reach && sl.x >= 0 && sl.y >= 0;
            }
            unsigned bits = __ballot_sync(full, near) & share;
            while (bits && !done) {
                const int p = p0 + __ffs(bits) - 1;
                bits &= bits - 1;
                T qx, qy, qz, dq;
                int e0, e1;
                const int t = saddle_proposal<FILT>(A, p, x, y, z, rp, rp, d0, qx, qy, qz, dq, e0, e1);
                if (t == 0) continue;
                if (t == -2) {
                    unsure = true;
                    continue;
                }
                const short2 sl = C.pslot[p];
                const int f = witness_free<FILT>(S, qx, qy, qz, C.nbm + sl.x * aw, C.nbm + sl.y * aw, nw, rp, Rmax,
                                                 dq + d0, nt);
                if (f == 1 && t == 1) hit = done = true;
                else if (f != 0) unsure = true;
            }
            if (settle()) break;
        }
    }
    const unsigned h = __ballot_sync(full, hit), u = __ballot_sync(full, unsure);
    return (h & gmask) ? 0 : ((u & gmask) ? 2 : 1);
}

// bytes of a CTA's staging (TileS, then ClsSmem 16-byte aligned), rounded up to
// 256 so that consecutive slices of the global-memory tier stay aligned
template <class T, class CP>
__host__ __device__ constexpr size_t cls_bytes()
{
    return (((sizeof(TileS<T, CP>) + 15) & ~(size_t)15) + sizeof(ClsSmem<CP>) + 255) & ~(size_t)255;
}

// Five CTAs an SM in FP32 (48 registers, 42 KB: the lookup of pair_slots lies in
// the neighbour sets' place, else 48 KB and four): 1,808 -> 1,749 us on 32
// molecules, and in FP64, three CTAs either way, what is left to L1 takes
// 1.50 -> 1.37 ms off the run of 200 atoms.
// CP = CapMid: the staged lists in shared memory; a tile that overflows
// them goes to ovf.  CP = CapBig (BIG): the tiles listed in ovf, with the
// staged lists in this CTA's slice of the global scratch `big`; overflowing
// that too is a capacity error.
template <class T, bool FILT, class CP, bool BIG>
__global__ void __launch_bounds__(CLS_THREADS, sizeof(T) == sizeof(float) && !BIG ? 5 : 1) k_classify(Model M, Batch B, TileSched Q, int8_t *__restrict__ labels_all,
                                                          int *__restrict__ band, int *__restrict__ err,
                                                          int *__restrict__ ovf, unsigned char *__restrict__ big,
                                                          unsigned long long *__restrict__ n_tests)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *store = BIG ? big + (size_t)blockIdx.x * cls_bytes<T, CP>() : smem_raw;
    TileS<T, CP> &S = *reinterpret_cast<TileS<T, CP> *>(store);
    ClsSmem<CP> &C = *reinterpret_cast<ClsSmem<CP> *>(store + ((sizeof(TileS<T, CP>) + 15) & ~(size_t)15));
    __shared__ long long q_base;
    __shared__ Grid sG;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T rp = (T)M.rp, Rmax = (T)M.Rmax, rmax = (T)M.rmax;
    long long iter = 0;
    int ntests = 0;  // this thread's atom tests (witness freeness)
    const long long npos = sched_count(Q, B.n_tiles);
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
        int8_t *__restrict__ labels = labels_all + G.lab0;
        const T d0 = FILT ? (T)G.d0 : T(0);
        const T h = (T)G.h;
        if (threadIdx.x == 0) {  // before stage_tile's barriers, after the last tile's closing one
            C.nq = 0;
            C.band = 0;
            C.next = 0;
        }
        double x0[3];
        stage_tile<T>(M, G, mol, tile, S, x0);
        if (!BIG && (S.flags & ERR_CAP_ANY)) {  // uniform: set before stage_tile's last barrier
            if (threadIdx.x == 0) ovf_push(ovf, gt);
            __syncthreads();
            continue;
        }
        // (the global-memory tier classifies even a tile that overflows it,
        // with its lists cut at capacity, so every label is written; the
        // error bit makes the run report ESES_ECAPACITY)
        if (threadIdx.x == 0 && S.flags) atomicOr(err, S.flags);
        int t[3];
        tile_coords(G, tile, t);
        if (S.na == 0) {  // no atom within reach: every point is free (the labels start as outside)
            __syncthreads();
            continue;
        }
        // phase 1: bricks, two neighbours per warp
        static_assert(NBRICK == 2 * (CLS_THREADS / 32), "two bricks per warp");
        for (int brick = 2 * warp; brick < 2 * warp + 2; ++brick) {
            int li, lj, lk;
            brick_point(brick, 0, li, lj, lk);
            const T b0x = (T)li * h, b0y = (T)lj * h, b0z = (T)lk * h;
            const T b1x = b0x + h, b1y = b0y + T(3) * h, b1z = b0z + T(3) * h;
            int cnt = 0;
            for (int base = 0; base < S.na; base += 32) {
                int a = base + lane;
                bool hit = false;
                if (a < S.na) {
                    P4<T> c = S.atom[a];
                    T ex = c.x < b0x ? b0x - c.x : (c.x > b1x ? c.x - b1x : T(0));
                    T ey = c.y < b0y ? b0y - c.y : (c.y > b1y ? c.y - b1y : T(0));
                    T ez = c.z < b0z ? b0z - c.z : (c.z > b1z ? c.z - b1z : T(0));
                    T reach = c.w + rp + T(1e-3);
                    hit = ex * ex + ey * ey + ez * ez < reach * reach;
                }
                unsigned m = __ballot_sync(0xffffffffu, hit);
                if (lane == 0) C.bmask[brick][base >> 5] = m;
                cnt += __popc(m);
            }
            __syncwarp();
            brick_point(brick, lane, li, lj, lk);
            long long gi = (long long)TILE * t[0] + li, gj = (long long)TILE * t[1] + lj,
                      gk = (long long)TILE * t[2] + lk;
            bool valid = gi < G.dims[0] && gj < G.dims[1] && gk < G.dims[2];
            int lab = LABEL_OUT;
            if (cnt > 0) {
                T x = pt_coord<T>(G, li), y = pt_coord<T>(G, lj), z = pt_coord<T>(G, lk);
                bool vdw = false, sas = false, sas_u = false;
                const int nw = (S.na + 31) >> 5;
                // lt_sq's bounds at the largest radii
                const T er = FILT ? T(2) * ((T(2) * rmax + d0) * d0 + T(1e-6) * rmax * rmax) : T(0);
                const T eR = FILT ? T(2) * ((T(2) * Rmax + d0) * d0 + T(1e-6) * Rmax * Rmax) : T(0);
                for (int wd = 0; wd < nw && !vdw; ++wd) {
                    unsigned bits = C.bmask[brick][wd];
                    while (bits) {
                        const int a = (wd << 5) + __ffs(bits) - 1;
                        bits &= bits - 1;
                        P4<T> c = S.atom[a];
                        T dx = x - c.x, dy = y - c.y, dz = z - c.z;
                        T d2 = dx * dx + dy * dy + dz * dz;
                        T r = c.w, R = c.w + rp;
                        if (FILT ? d2 < r * r - er : d2 < r * r) {
                            vdw = true;
                            break;
                        }
                        if (FILT ? d2 < R * R - eR : d2 < R * R) sas = true;
                        else if (FILT && d2 < R * R + eR) sas_u = true;
                    }
                }
                if (vdw) lab = LABEL_IN;
                else if (!sas) lab = sas_u ? LABEL_BAND : LABEL_OUT;
                else lab = -1;  // shell point
            }
            // the brick's shell points, one after the other
            const unsigned shell = __ballot_sync(0xffffffffu, valid && lab == -1);
            int at = 0;
            if (lane == 0 && shell) at = atomicAdd(&C.nq, __popc(shell));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(shell & ((1u << lane) - 1u));
            if (valid) {
                if (lab == -1) {
                    C.queue[at] = (short)((li << 6) | (lj << 3) | lk | (brick << 9));
                } else {
                    labels[(gi * G.dims[1] + gj) * G.dims[2] + gk] = (int8_t)lab;
                    if (FILT && lab == LABEL_BAND) atomicAdd(&C.band, 1);
                }
            }
        }
        __syncthreads();
        const int nq = C.nq;
        if (nq > 0) {  // neighbour sets and pair slots for the witnesses' freeness tests
            int *hkey = reinterpret_cast<int *>(C.nbm);
            pair_slots<T>(S, hkey, reinterpret_cast<short *>(hkey + C.HS), C.pslot);
            build_neighbour_sets<T, CP>(S, C.nbm, rp);
            __syncthreads();
        }
        // phase 2: shell points, 32 / gs at a time per warp from a block counter
        int gs = 1;
        while (gs < 32 && nq * gs * 2 <= CLS_SPLIT) gs <<= 1;
        const int r = lane & (gs - 1), per = 32 / gs;
        while (nq > 0) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&C.next, per);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= nq) break;
            k += lane / gs;
            const int code = k < nq ? C.queue[k] : -1;
            const int li = (code >> 6) & 7, lj = (code >> 3) & 7, lk = code & 7;
            const T x = pt_coord<T>(G, li), y = pt_coord<T>(G, lj), z = pt_coord<T>(G, lk);
            const int lab = shell_points<FILT, T, CP>(S, C, code, x, y, z, rp, Rmax, d0, (float)G.h, G.d0, r, gs,
                                                      ntests);
            if (r == 0 && code >= 0) {
                const long long gi = (long long)TILE * t[0] + li, gj = (long long)TILE * t[1] + lj,
                                gk = (long long)TILE * t[2] + lk;
                labels[(gi * G.dims[1] + gj) * G.dims[2] + gk] = (int8_t)lab;
                if (FILT && lab == LABEL_BAND) atomicAdd(&C.band, 1);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && band && C.band > 0) band[1 + atomicAdd(&band[0], 1)] = (int)gt;
        __syncthreads();
      }
    }
    unsigned long long nw = (unsigned long long)ntests;
    for (int o = 16; o > 0; o >>= 1) nw += __shfl_down_sync(0xffffffffu, nw, o);
    if (lane == 0 && nw && n_tests) atomicAdd(n_tests, nw);
}

// The undecided points of global tile gt re-labelled in FP64 (whole block):
// one warp per point runs the witness search over every staged item.  A tile
// that overflows the staging goes to ovf (or, in the global-memory tier, is a
// capacity error).
template <class CP>
__device__ void band_tile(const Model &M, const Batch &B, long long gt, int8_t *__restrict__ labels_all,
                          TileS<double, CP> &S, Grid &sG, short *s_pts, int &s_np, int *err, int *ovf, bool big)
{
    const int mol = mol_of_tile(B, gt);
    load_grid(B, mol, sG);
    const Grid &G = sG;
    const long long tile = gt - G.tile0;
    int8_t *__restrict__ labels = labels_all + G.lab0;
    double x0[3];
    stage_tile<double>(M, G, mol, tile, S, x0);
    if (!big && (S.flags & ERR_CAP_ANY)) {  // the global-memory tier relabels even an overflowing tile
        if (threadIdx.x == 0) ovf_push(ovf, gt);
        __syncthreads();
        return;
    }
    if (threadIdx.x == 0 && S.flags) atomicOr(err, S.flags);
    int t[3];
    tile_coords(G, tile, t);
    SmemAcc<double, CP> A(S);
    // the tile's undecided points, then one warp per point: the FP64
    // witness search (a free probe centre closer than r_p: outside)
    if (threadIdx.x == 0) s_np = 0;
    __syncthreads();
    for (int p = threadIdx.x; p < TILE_PTS; p += CLS_THREADS) {
        int li = p >> 6, lj = (p >> 3) & 7, lk = p & 7;
        long long gi = (long long)TILE * t[0] + li, gj = (long long)TILE * t[1] + lj, gk = (long long)TILE * t[2] + lk;
        if (gi >= G.dims[0] || gj >= G.dims[1] || gk >= G.dims[2]) continue;
        if (labels[(gi * G.dims[1] + gj) * G.dims[2] + gk] == LABEL_BAND) s_pts[atomicAdd(&s_np, 1)] = (short)p;
    }
    __syncthreads();
    const int npts = s_np;
    for (int k = threadIdx.x >> 5; k < npts; k += CLS_THREADS / 32) {
        const int p = s_pts[k];
        const int li = p >> 6, lj = (p >> 3) & 7, lk = p & 7;
        unsigned um_p, um_v;
        const int r = warp_witness<false>(A, (double)li * G.h, (double)lj * G.h, (double)lk * G.h, M.rp, M.rp, 0.0, -1,
                                          -1, um_p, um_v);
        if ((threadIdx.x & 31) == 0) {
            const long long gi = (long long)TILE * t[0] + li, gj = (long long)TILE * t[1] + lj,
                            gk = (long long)TILE * t[2] + lk;
            labels[(gi * G.dims[1] + gj) * G.dims[2] + gk] = r == 1 ? LABEL_OUT : LABEL_IN;
        }
    }
    __syncthreads();
}

template <class CP>
__host__ __device__ constexpr size_t band_bytes()
{
    return (sizeof(TileS<double, CP>) + 255) & ~(size_t)255;
}

// CapSmall: the tiles that the classification listed (band[0] of them, any
// order), a block each.  CapBig (BIG): the tiles listed in ovf, staged in
// global memory.  Bound by the latency of a tile's FP64 staging and witness
// search; blocks that picked the tiles out of 256-tile chunks took a chunk's
// listed tiles one after the other (95-130 us at any size; 40-50 us now, 73 us on the
// packed box, 108 us at 20,000 atoms).
template <class CP, bool BIG>
__global__ void __launch_bounds__(CLS_THREADS) k_band(Model M, Batch B, int8_t *__restrict__ labels_all,
                                                      const int *__restrict__ band, int *__restrict__ err,
                                                      int *__restrict__ ovf, unsigned char *__restrict__ big)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *store = BIG ? big + (size_t)blockIdx.x * band_bytes<CP>() : smem_raw;
    TileS<double, CP> &S = *reinterpret_cast<TileS<double, CP> *>(store);
    __shared__ Grid sG;
    __shared__ short s_pts[TILE_PTS];
    __shared__ int s_np;
    const int *list = BIG ? ovf + 1 : band;
    const int n = list[0];
    for (int k = blockIdx.x; k < n; k += gridDim.x)
        band_tile<CP>(M, B, list[1 + k], labels_all, S, sG, s_pts, s_np, err, ovf, BIG);
}

// The tiles whose staging range of cells holds an atom, one thread per tile
// (the range of stage_tile): the others are outside everywhere, and a CTA that
// staged them spent 13,000 cycles to find out (half the tiles of a molecule's
// box at h 0.5).
__global__ void __launch_bounds__(256) k_tile_list(Model M, Batch B, int *__restrict__ list)
{
    const int lane = threadIdx.x & 31;
    for (long long g0 = (long long)blockIdx.x * 256 + (threadIdx.x & ~31); g0 < B.n_tiles;
         g0 += (long long)gridDim.x * 256) {
        const long long gt = g0 + lane;
        bool any = false;
        if (gt < B.n_tiles) {
            const int mol = mol_of_tile(B, gt);
            const Grid &G = B.grid[mol];
            const CellGrid &CG = M.cg[mol];
            int t[3], c0[3], c1[3];
            tile_coords(G, gt - G.tile0, t);
            const float icell = 1.0f / (float)M.cell, halo = (float)G.halo + 1e-2f;
            for (int a = 0; a < 3; ++a) {
                const double fx0 = G.lo[a] + G.h * (double)(TILE * (t[a] + G.toff[a]));
                const double fx1 = fx0 + G.h * (double)TILE;
                c0[a] = max((int)floorf(((float)(fx0 - CG.clo[a]) - halo) * icell), 0);
                c1[a] = min((int)floorf(((float)(fx1 - CG.clo[a]) + halo) * icell), CG.cn[a] - 1);
            }
            if (c0[2] <= c1[2])
                for (int x = c0[0]; x <= c1[0] && !any; ++x)
                    for (int y = c0[1]; y <= c1[1] && !any; ++y) {
                        const int id = CG.coff + (x * CG.cn[1] + y) * CG.cn[2];
                        any = M.cell_start[id + c1[2] + 1] > M.cell_start[id + c0[2]];
                    }
        }
        const unsigned m = __ballot_sync(0xffffffffu, any);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(&list[0], __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (any) list[1 + base + __popc(m & ((1u << lane) - 1u))] = (int)gt;
    }
}

int launch_tile_list(const Model &M, const Batch &B, int *list, cudaStream_t st)
{
    cudaMemsetAsync(list, 0, sizeof(int), st);
    const long long nb = ceil_div_ll(std::max(B.n_tiles, 1LL), 256);
    k_tile_list<<<(unsigned)std::min(nb, 65536LL), 256, 0, st>>>(M, B, list);
    return 1;
}

static long long g_band_grid = 1;  // resident k_band CTAs on the device
static int g_n_sm = 1;              // SMs: the grid of the global-memory tier

// dynamic shared memory limits and the band kernel's grid (once per device,
// before any launch or capture)
void classify_init()
{
    cudaFuncSetAttribute(k_classify<double, false, CapMid, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)cls_bytes<double, CapMid>());
    cudaFuncSetAttribute(k_classify<float, true, CapMid, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)cls_bytes<float, CapMid>());
    cudaFuncSetAttribute(k_band<CapSmall, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)band_bytes<CapSmall>());
    int dev = 0, n_sm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_band<CapSmall, false>, CLS_THREADS,
                                                  band_bytes<CapSmall>());
    g_n_sm = n_sm > 0 ? n_sm : 1;
    g_band_grid = (long long)g_n_sm * (per_sm > 0 ? per_sm : 1);
}

// bytes of global scratch the global-memory tier of the classification and
// the band re-labelling need (one slice per CTA, one CTA per SM)
size_t classify_big_bytes()
{
    size_t per = cls_bytes<double, CapBig>();
    if (cls_bytes<float, CapBig>() > per) per = cls_bytes<float, CapBig>();
    if (band_bytes<CapBig>() > per) per = band_bytes<CapBig>();
    return per * (size_t)g_n_sm;
}

int classify_ctas_per_sm(int precision)
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    if (precision == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_classify<double, false, CapMid, false>, CLS_THREADS,
                                                      cls_bytes<double, CapMid>());
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_classify<float, true, CapMid, false>, CLS_THREADS,
                                                      cls_bytes<float, CapMid>());
    return n > 0 ? n : 1;
}

// the shared-memory tier over the scheduled tiles, then the global-memory
// tier over the tiles that overflowed it (ovf: count, then tiles)
int launch_classify(const Model &M, const Batch &B, int precision, const TileSched &Q, int grid, int8_t *labels,
                    int *band, int *err, int *ovf, unsigned char *big, unsigned long long *n_tests,
                    cudaStream_t st)
{
    if (grid < 1) grid = 1;
    if (band) cudaMemsetAsync(band, 0, sizeof(int), st);
    cudaMemsetAsync(ovf + 1, 0, sizeof(int), st);
    TileSched QB{nullptr, 1, ovf + 2, ovf + 1};
    if (precision == 0) {
        k_classify<double, false, CapMid, false><<<grid, CLS_THREADS, cls_bytes<double, CapMid>(), st>>>(
            M, B, Q, labels, band, err, ovf, nullptr, n_tests);
        if (big)
            k_classify<double, false, CapBig, true><<<g_n_sm, CLS_THREADS, 0, st>>>(M, B, QB, labels, band, err, ovf,
                                                                               big, n_tests);
    } else {
        k_classify<float, true, CapMid, false><<<grid, CLS_THREADS, cls_bytes<float, CapMid>(), st>>>(
            M, B, Q, labels, band, err, ovf, nullptr, n_tests);
        if (big)
            k_classify<float, true, CapBig, true><<<g_n_sm, CLS_THREADS, 0, st>>>(M, B, QB, labels, band, err, ovf,
                                                                             big, n_tests);
    }
    return big ? 2 : 1;
}

int launch_band(const Model &M, const Batch &B, int8_t *labels, const int *band, int *err, int *ovf,
                unsigned char *big, cudaStream_t st)
{
    const long long grid = std::max(1LL, std::min(B.n_tiles, g_band_grid));
    cudaMemsetAsync(ovf + 1, 0, sizeof(int), st);
    k_band<CapSmall, false><<<(int)grid, CLS_THREADS, band_bytes<CapSmall>(), st>>>(M, B, labels, band, err, ovf,
                                                                                 nullptr);
    if (big) k_band<CapBig, true><<<g_n_sm, CLS_THREADS, 0, st>>>(M, B, labels, band, err, ovf, big);
    return big ? 2 : 1;
}

}  // namespace eses
