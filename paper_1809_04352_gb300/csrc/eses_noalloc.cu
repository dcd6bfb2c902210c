// eses_noalloc.cu -- crossing-edge extraction that allocates no memory.
//
// eses_crossing_edges_noalloc() lists, for each axis, the lower point of every
// grid edge whose two end labels differ, in the same order as
// eses_intersections() (8x8x8 tiles in C order, then lower index).  It is for
// callers that cannot call cudaMalloc: code whose device memory is owned by a
// framework allocator or a fixed budget, or work issued where an allocation
// call is not allowed.  The caller passes the labels and the output arrays;
// the per-tile counts and offsets it needs live in one file-scope __device__
// array of NAL_MAX_TILES tiles, which every GPU that loads the library holds
// until the process exits.
//
// The first call on a device looks up that array's device address with
// cudaGetSymbolAddress (with the device current) and caches it; make that
// first call before any stream capture.  The cached address belongs to the
// device's current context: after cudaDeviceReset the process must not call
// this entry point again on that device.  Every call reuses the same array and
// leaves its contents behind; each call rewrites every entry it reads, so no
// state carries over, but two calls that overlap on the GPU (different
// streams, or one launched before the previous has finished on another
// stream) race on the array.
//
// Two launches, bound by the label reads (each label once from HBM, its word
// up to five times from L1/L2) and the host round trip for the counts.  On
// 16.3 M labels the call took 487 us with byte loads per point and axis and a
// one-block scan between the passes (164 + 144 + 114 us), 102 us now.
#include <mutex>

#include "../../include/eses.h"
#include "eses_internal.cuh"

namespace eses {

constexpr long long NAL_MAX_TILES = 1LL << 17;  // 131,072 tiles = 67,108,864 points
constexpr int NAL_WARPS = 8;                    // one warp per tile at a time
constexpr int NAL_THREADS = 32 * NAL_WARPS;
constexpr int NAL_RUN_MAX = 8;                  // tiles per warp at most
constexpr int NAL_MAX_BLOCKS = (int)(NAL_MAX_TILES / (NAL_WARPS * NAL_RUN_MAX));
// layout: counts [3][NAL_MAX_TILES], block sums [3][NAL_MAX_BLOCKS], totals [4]
constexpr long long NAL_SUMS = 3 * NAL_MAX_TILES;
constexpr long long NAL_TOTALS = NAL_SUMS + 3 * NAL_MAX_BLOCKS;
constexpr long long NAL_SCRATCH_INTS = NAL_TOTALS + 4;
static_assert(TILE == 8, "noalloc kernels read rows of 8 + 1 labels");
// nal_run gives at most NAL_MAX_BLOCKS blocks up to NAL_MAX_TILES tiles
static_assert(NAL_MAX_TILES % (NAL_WARPS * NAL_RUN_MAX) == 0, "block sums hold every block");

static __device__ __align__(256) int g_nal_scratch[NAL_SCRATCH_INTS];

struct NalGrid {
    long long dims[3];
    int tiles[3];
    long long nt, np;  // tiles, grid points
    int run;           // tiles per warp: block b takes tiles [b, b + 1) * NAL_WARPS * run
};

// The labels of a tile and of the next layer along each axis: row 9 i + j
// (i, j = 0..8) holds its 8 points' bytes, the byte after them and how many of
// the 9 lie on the grid (0: none).
struct NalTile {
    uint2 b[81];
    uint8_t next[81], n[81];
};

// Rows are read as aligned words (three hold 9 bytes at any alignment) and
// shifted into place: a byte load per point and axis, as this kernel once had
// (three loads a point, 54 GB/s of labels), is 12 times the instructions.  Rows
// that end within a word of the array's ends are read byte by byte, so
// nothing outside the array is touched.
__device__ __forceinline__ void nal_load(const NalGrid &G, const int8_t *__restrict__ labels, const int t[3],
                                         NalTile &T)
{
    const int lane = threadIdx.x & 31;
    for (int r = lane; r < 81; r += 32) {
        const int i = r / 9, j = r - 9 * i;
        const long long gi = (long long)TILE * t[0] + i, gj = (long long)TILE * t[1] + j, gk = (long long)TILE * t[2];
        unsigned w0 = 0u, w1 = 0u, w2 = 0u;
        int n = 0;
        if (gi < G.dims[0] && gj < G.dims[1]) {
            n = (int)(G.dims[2] - gk < 9 ? G.dims[2] - gk : 9);
            const long long at = (gi * G.dims[1] + gj) * G.dims[2] + gk;
            const uint8_t *p = reinterpret_cast<const uint8_t *>(labels) + at;
            const int off = (int)(reinterpret_cast<uintptr_t>(p) & 3);
            if (at >= 4 && at + 12 <= G.np) {
                const unsigned *q = reinterpret_cast<const unsigned *>(p - off);
                const unsigned a0 = __ldg(q), a1 = __ldg(q + 1), a2 = __ldg(q + 2);
                w0 = __funnelshift_r(a0, a1, 8 * off);
                w1 = __funnelshift_r(a1, a2, 8 * off);
                w2 = a2 >> (8 * off);
            } else {
                for (int k = 0; k < n; ++k) {
                    const unsigned v = p[k];
                    if (k < 4) w0 |= v << (8 * k);
                    else if (k < 8) w1 |= v << (8 * (k - 4));
                    else w2 = v;
                }
            }
        }
        T.b[r] = make_uint2(w0, w1);
        T.next[r] = (uint8_t)w2;
        T.n[r] = (uint8_t)n;
    }
    __syncwarp();
}

// bit k: bytes k of (x, y) are nonzero
__device__ __forceinline__ unsigned nal_bytes(unsigned x, unsigned y)
{
    const unsigned lo = (__vcmpne4(x, 0u) & 0x01010101u) * 0x01020408u >> 24;
    const unsigned hi = (__vcmpne4(y, 0u) & 0x01010101u) * 0x01020408u >> 24;
    return lo | (hi << 4);
}

// crossing edges along axis a from the points of row (i, j), i, j < 8: bit k
__device__ __forceinline__ unsigned nal_cross(const NalTile &T, int i, int j, int a)
{
    const int r = 9 * i + j, n = T.n[r];
    const uint2 b = T.b[r];
    if (a == 2) {
        const unsigned y = T.next[r];
        return nal_bytes(b.x ^ __funnelshift_r(b.x, b.y, 8), b.y ^ __funnelshift_r(b.y, y, 8)) &
               (n > 1 ? (1u << (n - 1)) - 1u : 0u);
    }
    const int q = a == 0 ? r + 9 : r + 1;
    const uint2 c = T.b[q];
    return T.n[q] ? nal_bytes(b.x ^ c.x, b.y ^ c.y) & ((1u << min(n, 8)) - 1u) : 0u;
}

__device__ __forceinline__ void nal_tile(const NalGrid &G, long long tile, int t[3])
{
    const unsigned u = (unsigned)tile, q = u / (unsigned)G.tiles[2];
    t[2] = (int)(u - q * (unsigned)G.tiles[2]);
    t[1] = (int)(q % (unsigned)G.tiles[1]);
    t[0] = (int)(q / (unsigned)G.tiles[1]);
}

// per tile and axis: number of crossing edges; per block and axis their sum
__global__ void __launch_bounds__(NAL_THREADS) k_nal_count(NalGrid G, const int8_t *__restrict__ labels,
                                                           int *__restrict__ scratch)
{
    __shared__ NalTile tiles[NAL_WARPS];
    __shared__ int sum[3][NAL_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    NalTile &T = tiles[warp];
    int mine = 0;  // lanes 0..2: the warp's edges along that axis
    const long long t0 = (long long)blockIdx.x * NAL_WARPS * G.run + warp;
    for (int k = 0; k < G.run; ++k) {
        const long long tile = t0 + (long long)k * NAL_WARPS;
        if (tile >= G.nt) break;
        int t[3];
        nal_tile(G, tile, t);
        nal_load(G, labels, t, T);
        int c[3];
        for (int a = 0; a < 3; ++a) {
            const int r0 = 2 * lane;
            c[a] = __popc(nal_cross(T, r0 >> 3, r0 & 7, a)) + __popc(nal_cross(T, (r0 + 1) >> 3, (r0 + 1) & 7, a));
            c[a] = __reduce_add_sync(0xffffffffu, c[a]);
        }
        if (lane < 3) {
            const int v = lane == 0 ? c[0] : (lane == 1 ? c[1] : c[2]);
            scratch[lane * NAL_MAX_TILES + tile] = v;
            mine += v;
        }
        __syncwarp();
    }
    if (lane < 3) sum[lane][warp] = mine;
    __syncthreads();
    if (threadIdx.x < 3) {
        int s = 0;
        for (int w = 0; w < NAL_WARPS; ++w) s += sum[threadIdx.x][w];
        scratch[NAL_SUMS + threadIdx.x * NAL_MAX_BLOCKS + blockIdx.x] = s;
    }
}

// Per tile: the lower indices at the tile's offset, in point order.  A block
// takes the tiles it counted; its first offset is the sum of the earlier
// blocks' sums (at most 2,048 a axis, read by the whole block), so no scan
// stands between the two passes (one block's scan over 3 counts a tile was a
// quarter of the call).  Tiles without crossing edges are not read again.
__global__ void __launch_bounds__(NAL_THREADS) k_nal_write(NalGrid G, const int8_t *__restrict__ labels,
                                                           int *__restrict__ scratch, long long *out0,
                                                           long long *out1, long long *out2, long long cap0,
                                                           long long cap1, long long cap2)
{
    __shared__ NalTile tiles[NAL_WARPS];
    __shared__ int part[6][NAL_WARPS];
    __shared__ int cnt[3][NAL_WARPS * NAL_RUN_MAX];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long b0 = (long long)blockIdx.x * NAL_WARPS * G.run;
    const int ntl = (int)(G.nt - b0 < NAL_WARPS * G.run ? G.nt - b0 : NAL_WARPS * G.run);
    for (int a = 0; a < 3; ++a) {
        int before = 0, all = 0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += NAL_THREADS) {
            const int v = scratch[NAL_SUMS + a * NAL_MAX_BLOCKS + b];
            if (b < (int)blockIdx.x) before += v;
            all += v;
        }
        before = __reduce_add_sync(0xffffffffu, before);
        all = __reduce_add_sync(0xffffffffu, all);
        if (lane == 0) {
            part[a][warp] = before;
            part[3 + a][warp] = all;
        }
        if (threadIdx.x < ntl) cnt[a][threadIdx.x] = scratch[a * NAL_MAX_TILES + b0 + threadIdx.x];
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x < 3) {
        int s = 0;
        for (int w = 0; w < NAL_WARPS; ++w) s += part[3 + threadIdx.x][w];
        scratch[NAL_TOTALS + threadIdx.x] = s;
    }
    NalTile &T = tiles[warp];
    long long *const outs[3] = {out0, out1, out2};
    const long long caps[3] = {cap0, cap1, cap2};
    for (int k = 0; k < G.run; ++k) {
        const int q = k * NAL_WARPS + warp;
        if (q >= ntl) break;
        if (cnt[0][q] + cnt[1][q] + cnt[2][q] == 0) continue;
        int t[3];
        nal_tile(G, b0 + q, t);
        nal_load(G, labels, t, T);
        const int r0 = 2 * lane, i = r0 >> 3, j = r0 & 7;
        const long long base = (((long long)TILE * t[0] + i) * G.dims[1] + ((long long)TILE * t[1] + j)) * G.dims[2] +
                               (long long)TILE * t[2];
        for (int a = 0; a < 3; ++a) {
            if (cnt[a][q] == 0) continue;
            int off = 0;  // the block's earlier edges: earlier blocks, then its tiles before q
            for (int z = lane; z < NAL_WARPS; z += 32) off += part[a][z];
            for (int z = lane; z < q; z += 32) off += cnt[a][z];
            off = __reduce_add_sync(0xffffffffu, off);
            const unsigned m0 = nal_cross(T, i, j, a), m1 = nal_cross(T, i, j + 1, a);
            const int c = __popc(m0) + __popc(m1);
            int inc = c;
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            long long r = (long long)off + inc - c;
            long long *out = outs[a];
            const long long cap = caps[a];
            for (unsigned m = m0; m; m &= m - 1, ++r)
                if (r < cap) out[r] = base + __ffs(m) - 1;
            for (unsigned m = m1; m; m &= m - 1, ++r)
                if (r < cap) out[r] = base + G.dims[2] + __ffs(m) - 1;
        }
        __syncwarp();
    }
}

static std::mutex g_nal_mutex;
static int *g_nal_ptr[64] = {nullptr};

}  // namespace eses

using namespace eses;

extern "C" int eses_crossing_edges_noalloc(const int8_t *labels, const int64_t dims[3], int64_t *idx0, int64_t *idx1,
                                           int64_t *idx2, const int64_t capacity[3], int64_t counts[3], void *stream)
{
    if (!labels || !dims || !capacity || !counts || !idx0 || !idx1 || !idx2) return ESES_EINVAL;
    NalGrid G;
    G.nt = 1;
    for (int a = 0; a < 3; ++a) {
        if (dims[a] < 1 || capacity[a] < 0) return ESES_EINVAL;
        G.dims[a] = dims[a];
        // tile count in 64 bits, compared before it is narrowed (a wrapped int would pass the check)
        const long long ta = (dims[a] - 1) / TILE + 1;
        if (ta > NAL_MAX_TILES) return ESES_EINVAL;
        G.tiles[a] = (int)ta;
        G.nt *= ta;
        if (G.nt > NAL_MAX_TILES) return ESES_EINVAL;  // grid larger than the scratch array covers
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ESES_ECUDA;
    int *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_nal_mutex);
        if (!g_nal_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_nal_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return ESES_ECUDA;
            }
            g_nal_ptr[dev] = (int *)p;
        }
        scratch = g_nal_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    // up to 512 blocks with one tile per warp; larger grids take up to NAL_RUN_MAX tiles per warp
    const long long run = ceil_div_ll(G.nt, 512LL * NAL_WARPS);
    G.run = (int)(run < NAL_RUN_MAX ? run : NAL_RUN_MAX);
    const int grid = (int)ceil_div_ll(G.nt, (long long)NAL_WARPS * G.run);
    G.np = dims[0] * dims[1] * dims[2];
    k_nal_count<<<grid, NAL_THREADS, 0, st>>>(G, labels, scratch);
    k_nal_write<<<grid, NAL_THREADS, 0, st>>>(G, labels, scratch, (long long *)idx0, (long long *)idx1,
                                              (long long *)idx2, capacity[0], capacity[1], capacity[2]);
    int tot[3] = {0, 0, 0};
    bool ok = cudaGetLastError() == cudaSuccess;
    if (ok)
        ok = cudaMemcpyAsync(tot, scratch + NAL_TOTALS, sizeof(tot), cudaMemcpyDeviceToHost, st) == cudaSuccess;
    if (ok) ok = cudaStreamSynchronize(st) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return ESES_ECUDA;
    }
    int over = 0;
    for (int a = 0; a < 3; ++a) {
        counts[a] = tot[a];
        if (counts[a] > capacity[a]) over = 1;
    }
    return over ? ESES_ECAPACITY : ESES_OK;
}
