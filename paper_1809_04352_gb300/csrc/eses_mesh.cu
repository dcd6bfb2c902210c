// eses_mesh.cu -- triangle mesh of the surface from the labels and the edge
// intersections of a run, cube by cube (the next item after the hot path;
// the paper stops at the labels and intersections, Eq. 2-4).
//
// The cube rule (reading M1).  Corner i of a grid cube sits at offset
// ((i >> 2) & 1, (i >> 1) & 1, i & 1) from the cube's lower corner.  Cube edge
// 4 a + j runs along axis a from the j-th corner, in increasing corner number,
// whose axis-a offset is 0; it is cut when its corner labels differ, and its
// surface point is that edge's intersection.  On each face the cut edges pair
// into segments: two cut edges make one; four (inside corners on a diagonal)
// make two, each joining the two edges at one inside corner.  The rule sees
// only the face's labels, so cubes sharing a face agree and the mesh closes.
// The segments form loops (each cut edge is on two faces); a loop starts at
// its smallest edge, walks first towards the smaller of its two neighbours,
// is reversed after its first vertex if its Newell normal (from the edge
// midpoints) points on the whole from outside corners to inside ones, and is
// cut into the fan (v0, v_k, v_k+1).  The 256-case table is built on the host
// once, at the first mesh.
//
// Kernels (one warp per 8x8x8 tile, cubes by their lower corner; the tile's
// labels and the next layer's as rows of bits, tile_rows):
//   k_mesh_count  per tile and axis, a 512-bit mask of the crossing edges
//                 leaving its points and the counts of the bits before each of
//                 its words (an edge's rank in the tile's run of the axis'
//                 output is then one look-up and a popcount), triangles per
//                 tile and their 64-bit total;
//   k_mesh_emit   after an exclusive scan, the triangles: per vertex the key
//                 3 * (lower point of its edge) + axis and the intersection
//                 point (FP64), read from the run's outputs; the triangles of
//                 32 cubes are listed first and the lanes take their vertices in
//                 order, so keys and points are written in runs.  Bound by the
//                 writes (96 bytes a triangle) and the dependent reads of an
//                 edge's intersection.  Cubes a lane each, their vertices one
//                 after the other: 382 us for the three kernels on 3,000 atoms at
//                 h 0.4 (5.6 M points, 0.5 M triangles).
#include <cstring>
#include <memory>
#include <vector>

#include "eses_kernels.h"
#include "eses_tile.cuh"

namespace eses {

constexpr int MESH_WARPS = 8;
constexpr int MC_MAXT = 12;  // triangles per cube at most (the rule gives at most 5)

// The case table as the kernels read it, from a buffer of the context that its
// first mesh fills on its own stream: no other context or thread writes it,
// and the copy is ordered before the kernels.
struct MeshTable {
    int8_t tri[256][3 * MC_MAXT];
    uint8_t n[256];
    int8_t edge[12][4];  // axis, offsets of the lower corner
};

// ---------------------------------------------------------------------------
// the case table (host)
// ---------------------------------------------------------------------------
static int corner_off(int i, int a) { return (i >> (2 - a)) & 1; }

struct CubeEdge {
    int axis, lo, hi;
};

static std::vector<CubeEdge> cube_edges()
{
    std::vector<CubeEdge> out;
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < 8; ++i)
            if (corner_off(i, a) == 0) out.push_back({a, i, i | (1 << (2 - a))});
    return out;
}

// one case: triangles as cube-edge triples; false if the rule fails (never expected)
static bool mc_case(int cs, const std::vector<CubeEdge> &E, std::vector<int> &tris)
{
    tris.clear();
    int in[8];
    for (int i = 0; i < 8; ++i) in[i] = (cs >> i) & 1;
    bool cut[12];
    for (int e = 0; e < 12; ++e) cut[e] = in[E[e].lo] != in[E[e].hi];
    int nb[12][2], nn[12] = {0};
    auto link = [&](int x, int y) {
        if (nn[x] < 2) nb[x][nn[x]] = y;
        if (nn[y] < 2) nb[y][nn[y]] = x;
        ++nn[x];
        ++nn[y];
    };
    for (int a = 0; a < 3; ++a)
        for (int side = 0; side < 2; ++side) {
            int fe[4], nf = 0;
            for (int e = 0; e < 12; ++e)
                if (E[e].axis != a && corner_off(E[e].lo, a) == side && corner_off(E[e].hi, a) == side) fe[nf++] = e;
            if (nf != 4) return false;
            int ce[4], nc = 0;
            for (int k = 0; k < 4; ++k)
                if (cut[fe[k]]) ce[nc++] = fe[k];
            if (nc == 2) {
                link(ce[0], ce[1]);
            } else if (nc == 4) {
                for (int c = 0; c < 8; ++c) {  // each inside corner of the face: its two face edges
                    if (corner_off(c, a) != side || !in[c]) continue;
                    int at[2], na = 0;
                    for (int k = 0; k < 4; ++k)
                        if ((E[fe[k]].lo == c || E[fe[k]].hi == c) && na < 2) at[na++] = fe[k];
                    if (na != 2) return false;
                    link(at[0], at[1]);
                }
            } else if (nc != 0) {
                return false;
            }
        }
    for (int e = 0; e < 12; ++e)
        if (cut[e] != (nn[e] == 2) || nn[e] > 2) return false;
    bool seen[12] = {false};
    for (int s = 0; s < 12; ++s) {
        if (!cut[s] || seen[s]) continue;
        int loop[12], nl = 0;
        loop[nl++] = s;
        seen[s] = true;
        int cur = s, nxt = nb[s][0] < nb[s][1] ? nb[s][0] : nb[s][1];
        while (nxt != s) {
            if (nl >= 12) return false;
            loop[nl++] = nxt;
            seen[nxt] = true;
            const int after = nb[nxt][0] == cur ? nb[nxt][1] : nb[nxt][0];
            cur = nxt;
            nxt = after;
        }
        // Newell normal of the edge midpoints against inside -> outside
        double mid[12][3], n[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < nl; ++k)
            for (int a = 0; a < 3; ++a)
                mid[k][a] = 0.5 * (corner_off(E[loop[k]].lo, a) + corner_off(E[loop[k]].hi, a));
        for (int k = 0; k < nl; ++k) {
            const double *p = mid[k], *q = mid[(k + 1) % nl];
            n[0] += (p[1] - q[1]) * (p[2] + q[2]);
            n[1] += (p[2] - q[2]) * (p[0] + q[0]);
            n[2] += (p[0] - q[0]) * (p[1] + q[1]);
        }
        double score = 0.0;
        for (int k = 0; k < nl; ++k) {
            const CubeEdge &ed = E[loop[k]];
            const int ci = in[ed.lo] ? ed.lo : ed.hi, co = in[ed.lo] ? ed.hi : ed.lo;
            for (int a = 0; a < 3; ++a) score += (corner_off(co, a) - corner_off(ci, a)) * n[a];
        }
        if (score == 0.0) return false;
        if (score < 0.0)
            for (int x = 1, y = nl - 1; x < y; ++x, --y) std::swap(loop[x], loop[y]);
        for (int k = 1; k + 1 < nl; ++k) {
            tris.push_back(loop[0]);
            tris.push_back(loop[k]);
            tris.push_back(loop[k + 1]);
        }
    }
    return (int)tris.size() <= 3 * MC_MAXT;
}

// the table: tri[case][3 k + v] cube edges, n[case] triangles; false on a rule failure
static bool mc_table(int8_t (*tri)[3 * MC_MAXT], uint8_t *n)
{
    const std::vector<CubeEdge> E = cube_edges();
    std::vector<int> t;
    for (int cs = 0; cs < 256; ++cs) {
        if (!mc_case(cs, E, t)) return false;
        n[cs] = (uint8_t)(t.size() / 3);
        for (int k = 0; k < 3 * MC_MAXT; ++k) tri[cs][k] = k < (int)t.size() ? (int8_t)t[k] : (int8_t)-1;
    }
    return true;
}

// built once, by whichever thread asks first (null if the rule fails)
static const MeshTable *mesh_table_build()
{
    static const std::unique_ptr<const MeshTable> table = [] {
        auto t = std::make_unique<MeshTable>();
        if (!mc_table(t->tri, t->n)) return std::unique_ptr<const MeshTable>();
        const std::vector<CubeEdge> E = cube_edges();
        for (int e = 0; e < 12; ++e) {
            t->edge[e][0] = (int8_t)E[e].axis;
            for (int a = 0; a < 3; ++a) t->edge[e][1 + a] = (int8_t)corner_off(E[e].lo, a);
        }
        return std::unique_ptr<const MeshTable>(std::move(t));
    }();
    return table.get();
}

int mesh_table_host(int8_t *tri, uint8_t *n, int max_tri)
{
    const MeshTable *T = mesh_table_build();
    if (!T) return -1;
    for (int cs = 0; cs < 256; ++cs) {
        if (T->n[cs] > max_tri) return -1;
        n[cs] = T->n[cs];
        for (int k = 0; k < 3 * max_tri; ++k) tri[cs * 3 * max_tri + k] = k < 3 * MC_MAXT ? T->tri[cs][k] : (int8_t)-1;
    }
    return 0;
}

size_t mesh_table_bytes() { return sizeof(MeshTable); }

int mesh_table_copy(void *table, cudaStream_t st)
{
    const MeshTable *T = mesh_table_build();
    if (!T) return -1;
    return cudaMemcpyAsync(table, T, sizeof(*T), cudaMemcpyHostToDevice, st) == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// kernels (one molecule: B.grid[0], tiles 0 .. n_tiles - 1)
// ---------------------------------------------------------------------------
constexpr int MASK_WORDS = TILE_PTS / 32;
// per tile and axis: the mask, then 16-bit prefix counts (two to a word)
constexpr int MASK_STRIDE = MASK_WORDS + MASK_WORDS / 2;

// case of the cube whose lower corner is local point p (-1 when the cube leaves the grid); k_on: the points of a
// row on the grid, at most 9
__device__ __forceinline__ int cube_case(const uint16_t *row, int p, int k_on)
{
    const int r = 9 * (p >> 6) + ((p >> 3) & 7), k = p & 7;
    const unsigned a = row[r], b = row[r + 1], c = row[r + 9], d = row[r + 10];
    if (!(a & b & c & d & 0x8000u) || k + 1 >= k_on) return -1;
    return (int)(((a >> k) & 3u) | (((b >> k) & 3u) << 2) | (((c >> k) & 3u) << 4) | (((d >> k) & 3u) << 6));
}

__global__ void __launch_bounds__(MESH_WARPS * 32) k_mesh_count(Batch B, const MeshTable *__restrict__ Tb,
                                                                const int8_t *__restrict__ labels,
                                                               uint32_t *__restrict__ mask,
                                                               int *__restrict__ tile_tri,
                                                               unsigned long long *__restrict__ total)
{
    __shared__ uint16_t rows[MESH_WARPS][81];
    const int lane = threadIdx.x & 31;
    uint16_t *row = rows[threadIdx.x >> 5];
    const Grid &G = B.grid[0];
    const long long nw = (long long)gridDim.x * MESH_WARPS;
    unsigned long long sum = 0;
    for (long long gt = (long long)blockIdx.x * MESH_WARPS + (threadIdx.x >> 5); gt < B.n_tiles; gt += nw) {
        int t[3];
        tile_coords(G, gt, t);
        tile_rows(G, labels, t, row);
        const int n_on = (int)min(9LL, G.dims[2] - (long long)TILE * t[2]);
        const unsigned on = (1u << min(n_on, 8)) - 1u, onz = (1u << (n_on - 1)) - 1u & 0xffu;
        for (int a = 0; a < 3; ++a) {
            unsigned m = 0u;  // 16 edges: rows 2 lane and 2 lane + 1
            for (int q = 0; q < 2; ++q) {
                const int l = 2 * lane + q, r = 9 * (l >> 3) + (l & 7);
                const unsigned x = row[r], y = a == 0 ? row[r + 9] : (a == 1 ? row[r + 1] : x >> 1);
                const bool both = (x & 0x8000u) && (a == 2 || (y & 0x8000u));
                m |= (both ? (x ^ y) & (a == 2 ? onz : on) : 0u) << (8 * q);
            }
            const unsigned w = m | (__shfl_down_sync(0xffffffffu, m, 1) << 16);  // even lanes: word lane / 2
            const int c = (lane & 1) ? 0 : __popc(w);
            int inc = c;
            for (int o = 2; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            uint32_t *out = mask + (size_t)(gt * 3 + a) * MASK_STRIDE;
            if (!(lane & 1)) {
                out[lane >> 1] = w;
                reinterpret_cast<uint16_t *>(out + MASK_WORDS)[lane >> 1] = (uint16_t)(inc - c);
            }
        }
        int n = 0;
        for (int p = lane; p < TILE_PTS; p += 32) {
            const int cs = cube_case(row, p, n_on);
            if (cs > 0) n += Tb->n[cs];
        }
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) tile_tri[gt] = n;
        sum += (unsigned long long)n;
        __syncwarp();
    }
    if (lane == 0 && sum) atomicAdd(total, sum);
}

__global__ void __launch_bounds__(MESH_WARPS * 32) k_mesh_emit(Batch B, const MeshTable *__restrict__ Tb,
                                                               const int8_t *__restrict__ labels,
                                                              const uint32_t *__restrict__ mask,
                                                              const int *__restrict__ edge_start, EdgeOut out,
                                                              const int *__restrict__ tile_off,
                                                              long long *__restrict__ keys, double *__restrict__ xyz,
                                                              int *__restrict__ err)
{
    __shared__ uint16_t rows[MESH_WARPS][81];
    __shared__ uint16_t tris[MESH_WARPS][32 * MC_MAXT];  // a round's triangles: cube's lane | place in its case << 5
    const int lane = threadIdx.x & 31;
    uint16_t *row = rows[threadIdx.x >> 5], *tri = tris[threadIdx.x >> 5];
    const Grid &G = B.grid[0];
    const long long d[3] = {G.dims[0], G.dims[1], G.dims[2]};
    const long long nt = B.n_tiles;
    const long long nw = (long long)gridDim.x * MESH_WARPS;
    const double h = G.h;
    for (long long gt = (long long)blockIdx.x * MESH_WARPS + (threadIdx.x >> 5); gt < nt; gt += nw) {
        long long run = tile_off[gt];
        if (tile_off[gt + 1] == run) continue;  // uniform
        int t[3];
        tile_coords(G, gt, t);
        tile_rows(G, labels, t, row);
        const int n_on = (int)min(9LL, d[2] - (long long)TILE * t[2]);
        for (int r = 0; r < TILE_PTS / 32; ++r) {
            const int cs = cube_case(row, 32 * r + lane, n_on);
            const int cnt = cs > 0 ? Tb->n[cs] : 0;
            int inc = cnt;  // cubes in local order: inclusive warp scan
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            const int tot = __shfl_sync(0xffffffffu, inc, 31);
            for (int k = 0; k < cnt; ++k) tri[inc - cnt + k] = (uint16_t)(lane | (k << 5));
            __syncwarp();
            for (int q0 = 0; q0 < 3 * tot; q0 += 32) {
                const int q = q0 + lane;
                const unsigned e5 = q < 3 * tot ? tri[q / 3] : 0u;
                const int src = e5 & 31, k = e5 >> 5, v = q - 3 * (q / 3);
                const int c = __shfl_sync(0xffffffffu, cs, src);
                if (q >= 3 * tot) continue;
                const int p = 32 * r + src;
                const int e = Tb->tri[c][3 * k + v];
                const int a = Tb->edge[e][0];
                const int l[3] = {(p >> 6) + Tb->edge[e][1], ((p >> 3) & 7) + Tb->edge[e][2],
                                  (p & 7) + Tb->edge[e][3]};
                // the edge's rank in its tile's run of axis a's output
                const long long tl = ((long long)(t[0] + (l[0] >> 3)) * G.tiles[1] + (t[1] + (l[1] >> 3))) * G.tiles[2] +
                                     (t[2] + (l[2] >> 3));
                const int lp = ((l[0] & 7) * TILE + (l[1] & 7)) * TILE + (l[2] & 7);
                const uint32_t *mw = mask + (size_t)(tl * 3 + a) * MASK_STRIDE;
                const uint32_t w = mw[lp >> 5];
                const int rank = reinterpret_cast<const uint16_t *>(mw + MASK_WORDS)[lp >> 5] +
                                 __popc(w & ((1u << (lp & 31)) - 1u));
                const long long id = (long long)edge_start[a * nt + tl] - edge_start[a * nt] + rank;
                const long long na = (long long)edge_start[(a + 1) * nt] - edge_start[a * nt];
                double tau = 0.0;
                if (((w >> (lp & 31)) & 1u) && id >= 0 && id < na) tau = out.tau[a][id];
                else atomicOr(err, 1);  // the cube's cut edge is not in the run's output
                const long long gl[3] = {(long long)TILE * t[0] + l[0], (long long)TILE * t[1] + l[1],
                                         (long long)TILE * t[2] + l[2]};
                const long long o = 3 * run + q;
                keys[o] = 3 * ((gl[0] * d[1] + gl[1]) * d[2] + gl[2]) + a;
                for (int b = 0; b < 3; ++b)
                    xyz[3 * o + b] = G.lo[b] + h * (double)gl[b] + (b == a ? tau * h : 0.0);
            }
            run += tot;
            __syncwarp();
        }
    }
}

static int warp_grid(long long n_tiles)
{
    const long long g = (n_tiles + MESH_WARPS - 1) / MESH_WARPS;
    return (int)(g < 1 ? 1 : (g > 1048576 ? 1048576 : g));
}

size_t mesh_mask_words(long long n_tiles) { return (size_t)n_tiles * 3 * MASK_STRIDE; }

int launch_mesh_count(const Batch &B, const void *table, const int8_t *labels, uint32_t *mask, int *tile_tri,
                      unsigned long long *total, cudaStream_t st)
{
    cudaMemsetAsync(total, 0, sizeof(*total), st);
    k_mesh_count<<<warp_grid(B.n_tiles), MESH_WARPS * 32, 0, st>>>(B, (const MeshTable *)table, labels, mask,
                                                                   tile_tri, total);
    return 1;
}

int launch_mesh_emit(const Batch &B, const void *table, const int8_t *labels, const uint32_t *mask,
                     const int *edge_start, const EdgeOut &out, const int *tile_off, long long *keys, double *xyz,
                     int *err, cudaStream_t st)
{
    k_mesh_emit<<<warp_grid(B.n_tiles), MESH_WARPS * 32, 0, st>>>(B, (const MeshTable *)table, labels, mask,
                                                                  edge_start, out, tile_off, keys, xyz, err);
    return 1;
}

}  // namespace eses
