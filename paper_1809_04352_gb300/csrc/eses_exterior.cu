// eses_exterior.cu -- exterior-only surface (cavities filled).
//
// §1 counts every free probe position as solvent; the exterior-only variant
// keeps only the solvent a probe can reach from outside the molecule.  On the
// grid (reading X1): an outside point is exterior iff a path of outside
// points, each step between 6-neighbours, joins it to the domain boundary
// (whose points are all outside, reading C2); every other outside point is in
// a cavity and becomes inside.  The crossing edges, roots and area/volume are
// then computed from the relabelled grid by the usual stages.
//
// State per tile, in bits (one 16-bit word per lane of a warp, rows 2 lane and
// 2 lane + 1 of 8 points): the outside points, and the reached ones among them.
//   k_ext_init:  outside points from the labels, those on the domain boundary
//                reached; a tile is open while it holds others;
//   k_ext_sweep: one warp per open tile: the reached neighbours' facing points
//                seed the tile (a word per lane from each of the six tiles
//                around), then the reached set grows inside it until it stops
//                (bounded: a path inside the tile has fewer than 512 steps) with
//                shifts within a row and lane exchanges between rows; new points
//                are written back and a flag set; a tile all reached closes and
//                is not read again.  Sweeps repeat until one changes nothing
//                (the reached set only grows, so neighbours read mid-sweep are
//                either state and the fixed point is the same): k_ext_fill
//                runs them all in one cooperative launch with a grid-wide
//                barrier after each sweep (k_ext_sweep, one sweep per launch
//                driven from the host, where cooperative launch is missing);
//   k_ext_apply: outside points not reached are cavity points: label 1, counted.
// Bound by the latency of a sweep (the barrier, the tile's few reads and the
// steps of its growth).  A byte per point and a block per tile, one barrier per
// step of growth, took 439 us for 11 sweeps on 2,003 atoms at h 0.4.
#include <cooperative_groups.h>

#include "eses_kernels.h"
#include "eses_tile.cuh"

namespace eses {

constexpr int EXT_WARPS = 8;
constexpr int EXT_THREADS = EXT_WARPS * 32;

// points of rows 2 lane and 2 lane + 1 of the tile (16 bits) from a row function
template <class F>
__device__ __forceinline__ unsigned two_rows(F f)
{
    const int r0 = 2 * (threadIdx.x & 31);
    return f(r0 >> 3, r0 & 7) | (f((r0 + 1) >> 3, (r0 + 1) & 7) << 8);
}

__global__ void __launch_bounds__(EXT_THREADS) k_ext_init(Batch B, const int8_t *__restrict__ labels_all,
                                                         uint16_t *__restrict__ ext, uint8_t *__restrict__ tile_open)
{
    __shared__ uint16_t rows[EXT_WARPS][81];
    const int lane = threadIdx.x & 31;
    uint16_t *row = rows[threadIdx.x >> 5];
    const long long nw = (long long)gridDim.x * EXT_WARPS;
    for (long long gt = (long long)blockIdx.x * EXT_WARPS + (threadIdx.x >> 5); gt < B.n_tiles; gt += nw) {
        const Grid &G = B.grid[mol_of_tile(B, gt)];
        int t[3];
        tile_coords(G, gt - G.tile0, t);
        tile_rows(G, labels_all, t, row);
        const long long gk = (long long)TILE * t[2], n = G.dims[2] - gk;
        const unsigned on = n >= 8 ? 0xffu : (1u << n) - 1u;
        const unsigned face = (t[2] == 0 ? 1u : 0u) | (n <= 8 ? 1u << (n - 1) : 0u);  // first and last k of the grid
        const unsigned out = two_rows([&](int i, int j) {
            const unsigned m = row[9 * i + j];
            return (m & 0x8000u) ? ~m & on : 0u;
        });
        const unsigned edge = two_rows([&](int i, int j) {
            const long long gi = (long long)TILE * t[0] + i, gj = (long long)TILE * t[1] + j;
            return gi == 0 || gj == 0 || gi == G.dims[0] - 1 || gj == G.dims[1] - 1 ? 0xffu : face;
        });
        ext[64 * gt + lane] = (uint16_t)out;
        ext[64 * gt + 32 + lane] = (uint16_t)(out & edge);
        const bool open = __any_sync(0xffffffffu, (out & ~edge) != 0u);
        if (lane == 0) tile_open[gt] = open ? 1 : 0;
        __syncwarp();
    }
}

// word `at` of the reached points of tile (a, b, c) of the grid, 0 off it
__device__ __forceinline__ unsigned reached_word(const Grid &G, const uint16_t *ext, int a, int b, int c, int at)
{
    if (a < 0 || b < 0 || c < 0 || a >= G.tiles[0] || b >= G.tiles[1] || c >= G.tiles[2]) return 0u;
    const long long gt = G.tile0 + ((long long)a * G.tiles[1] + b) * G.tiles[2] + c;
    return __ldcg(&ext[64 * gt + 32 + at]);  // (other blocks write it during the sweep)
}

// one sweep over the warp's tiles w, w + n_warps, ...
__device__ __forceinline__ void sweep_tiles(const Batch &B, uint16_t *__restrict__ ext,
                                            uint8_t *__restrict__ tile_open, int *__restrict__ changed)
{
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, jj = lane & 3;
    const long long nw = (long long)gridDim.x * EXT_WARPS;
    for (long long gt = (long long)blockIdx.x * EXT_WARPS + (threadIdx.x >> 5); gt < B.n_tiles; gt += nw) {
        if (!tile_open[gt]) continue;  // uniform: every lane reads the same byte
        const Grid &G = B.grid[mol_of_tile(B, gt)];
        int t[3];
        tile_coords(G, gt - G.tile0, t);
        const unsigned open = ext[64 * gt + lane], was = __ldcg(&ext[64 * gt + 32 + lane]);
        // seeds: the facing points of the six tiles around
        unsigned seed = (reached_word(G, ext, t[0], t[1], t[2] - 1, lane) >> 7) & 0x0101u;
        seed |= (reached_word(G, ext, t[0], t[1], t[2] + 1, lane) & 0x0101u) << 7;
        if (jj == 0) seed |= reached_word(G, ext, t[0], t[1] - 1, t[2], lane + 3) >> 8;             // its row j = 7
        if (jj == 3) seed |= (reached_word(G, ext, t[0], t[1] + 1, t[2], lane - 3) & 0xffu) << 8;  // its row j = 0
        if (lane < 4) seed |= reached_word(G, ext, t[0] - 1, t[1], t[2], lane + 28);
        if (lane >= 28) seed |= reached_word(G, ext, t[0] + 1, t[1], t[2], lane - 28);
        unsigned r = was | (seed & open);
        for (int it = 0; it < TILE_PTS; ++it) {  // grow inside the tile until it stops
            const unsigned up = __shfl_up_sync(full, r, 1), down = __shfl_down_sync(full, r, 1);
            const unsigned before = __shfl_up_sync(full, r, 4), after = __shfl_down_sync(full, r, 4);
            unsigned g = ((r << 1) & 0xfefeu) | ((r >> 1) & 0x7f7fu);    // along k
            g |= (r << 8) | (r >> 8);                                      // along j, within the word
            if (jj > 0) g |= up >> 8;
            if (jj < 3) g |= down << 8;
            if (lane >= 4) g |= before;                                   // along i
            if (lane < 28) g |= after;
            g = (r | g) & open;
            const bool grew = g != r;
            r = g;
            if (!__any_sync(full, grew)) break;
        }
        const bool any = __any_sync(full, r != was), left = __any_sync(full, r != open);
        if (r != was) __stcg(&ext[64 * gt + 32 + lane], (uint16_t)r);
        if (lane == 0 && any) atomicExch(changed, 1);
        if (lane == 0 && !left) tile_open[gt] = 0;
    }
}

__global__ void __launch_bounds__(EXT_THREADS) k_ext_sweep(Batch B, uint16_t *__restrict__ ext,
                                                          uint8_t *__restrict__ tile_open, int *__restrict__ changed)
{
    sweep_tiles(B, ext, tile_open, changed);
}

// Every sweep in one cooperative launch (all blocks resident): after each
// sweep a grid-wide barrier, then every block reads that sweep's changed flag
// and all stop together when it is clear.  Three flags rotate: block 0 clears
// the next sweep's flag, which every block last read before the previous
// barrier.  At most max_sweeps sweeps (the host loop's bound); flags[3]
// receives the number of sweeps run.
__global__ void __launch_bounds__(EXT_THREADS) k_ext_fill(Batch B, uint16_t *__restrict__ ext,
                                                         uint8_t *__restrict__ tile_open, int *__restrict__ flags,
                                                         long long max_sweeps)
{
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    long long it = 0;
    for (; it < max_sweeps; ++it) {
        if (blockIdx.x == 0 && threadIdx.x == 0) flags[(it + 1) % 3] = 0;
        sweep_tiles(B, ext, tile_open, &flags[it % 3]);
        grid.sync();
        if (*(volatile int *)&flags[it % 3] == 0) break;  // the same value in every block
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) flags[3] = (int)(it < max_sweeps ? it + 1 : it);
}

__global__ void __launch_bounds__(EXT_THREADS) k_ext_apply(Batch B, int8_t *__restrict__ labels_all,
                                                          const uint16_t *__restrict__ ext,
                                                          unsigned long long *__restrict__ filled)
{
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * EXT_WARPS;
    unsigned n = 0;
    for (long long gt = (long long)blockIdx.x * EXT_WARPS + (threadIdx.x >> 5); gt < B.n_tiles; gt += nw) {
        unsigned m = (unsigned)ext[64 * gt + lane] & ~(unsigned)ext[64 * gt + 32 + lane];
        if (!m) continue;
        const Grid &G = B.grid[mol_of_tile(B, gt)];
        int t[3];
        tile_coords(G, gt - G.tile0, t);
        n += (unsigned)__popc(m);
        for (; m; m &= m - 1) {
            const int b = __ffs(m) - 1, row = 2 * lane + (b >> 3);
            const long long gi = (long long)TILE * t[0] + (row >> 3), gj = (long long)TILE * t[1] + (row & 7),
                            gk = (long long)TILE * t[2] + (b & 7);
            labels_all[G.lab0 + (gi * G.dims[1] + gj) * G.dims[2] + gk] = LABEL_IN;
        }
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0 && n) atomicAdd(filled, (unsigned long long)n);
}

static int warp_grid(long long n_tiles)
{
    const long long g = (n_tiles + EXT_WARPS - 1) / EXT_WARPS;
    return (int)(g < 1 ? 1 : (g > 1048576 ? 1048576 : g));
}

int launch_ext_init(const Batch &B, const int8_t *labels, uint16_t *ext, uint8_t *tile_open, cudaStream_t st)
{
    k_ext_init<<<warp_grid(B.n_tiles), EXT_WARPS * 32, 0, st>>>(B, labels, ext, tile_open);
    return 1;
}

int launch_ext_sweep(const Batch &B, uint16_t *ext, uint8_t *tile_open, int *changed, int grid, cudaStream_t st)
{
    k_ext_sweep<<<grid < 1 ? 1 : grid, EXT_THREADS, 0, st>>>(B, ext, tile_open, changed);
    return 1;
}

// all sweeps in one cooperative launch; returns 0 when the device cannot
// launch cooperatively (the caller then drives k_ext_sweep from the host)
int launch_ext_fill(const Batch &B, uint16_t *ext, uint8_t *tile_open, int *flags, long long max_sweeps,
                    cudaStream_t st)
{
    int dev = 0, coop = 0, n_sm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop) return 0;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ext_fill, EXT_THREADS, 0);
    if (per_sm < 1) return 0;
    long long grid = (long long)per_sm * n_sm;
    const long long need = (B.n_tiles + EXT_WARPS - 1) / EXT_WARPS;
    if (grid > need) grid = need < 1 ? 1 : need;
    Batch b = B;
    void *args[] = {&b, &ext, &tile_open, &flags, &max_sweeps};
    if (cudaLaunchCooperativeKernel((void *)k_ext_fill, dim3((unsigned)grid), dim3(EXT_THREADS), args, 0, st) !=
        cudaSuccess)
        return -1;
    return 1;
}

int launch_ext_apply(const Batch &B, int8_t *labels, const uint16_t *ext, unsigned long long *filled, cudaStream_t st)
{
    k_ext_apply<<<warp_grid(B.n_tiles), EXT_WARPS * 32, 0, st>>>(B, labels, ext, filled);
    return 1;
}

}  // namespace eses
