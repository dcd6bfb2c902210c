// eses_mlp.cu -- the learned tile proposer: per-tile features, the MLP
// 32 -> 64 -> 64 -> 1 (ReLU), its training kernels (forward, backward, Adam)
// and the exact far-tile certificate.
//
// A tile whose labels are all equal (no surface crossing inside it) is "far".
// The proposer scores every tile from cheap atom-density features; a tile it
// scores far is checked by an exact certificate built from nearest-atom
// distance bounds around the tile's centre t (the tile's points lie within
// delta = 3.5 h sqrt(3) of t):
//   all points free (label 0) if  min_i (|t - c_i| - R_i) >= delta
//     (then |x - c_i| >= R_i for every point x and atom i: x is a free probe
//      position, at distance 0 < r_p from the free set);
//   all points inside (label 1) if  max_i (r_i - |t - c_i|) > delta
//     (then every point lies inside van der Waals ball i).
// A certified tile is filled with its label; every other tile (a miss, or a
// tile scored near) goes to the exact classification, so the labels do not
// depend on the network.  Features of a tile (molecule cell grid, cells of
// edge `cell` around the cell holding t):
//   f[0..26]  log(1 + atoms) in the 27 cells around t's cell
//   f[27..29] position of t in its cell, in cell units, minus 1/2
//   f[30]     log(1 + atoms in the 27 cells)
//   f[31]     tile edge (8 h) over the cell edge
#include <math.h>

#include <algorithm>

#include "eses_kernels.h"
#include "eses_mlp_tc.cuh"
#include "eses_tile.cuh"

namespace eses {

constexpr int GRAD_S = 32;        // samples per block of the gradient kernel
constexpr int GRAD_THREADS = 256;
constexpr int PROP_THREADS = 128;  // tiles per block of the proposer kernel

// ---------------------------------------------------------------------------
// MLP forward (FP32), one thread per sample
// ---------------------------------------------------------------------------
__device__ __forceinline__ float mlp_eval(const float *P, const float *x)
{
    float h2[MLP_H];
#pragma unroll
    for (int k = 0; k < MLP_H; ++k) h2[k] = P[P_B2 + k];
    for (int j = 0; j < MLP_H; ++j) {
        float a = P[P_B1 + j];
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) a = fmaf(x[i], P[P_W1 + i * MLP_H + j], a);
        a = fmaxf(a, 0.0f);
#pragma unroll
        for (int k = 0; k < MLP_H; ++k) h2[k] = fmaf(a, P[P_W2 + j * MLP_H + k], h2[k]);
    }
    float z = P[P_B3];
#pragma unroll
    for (int k = 0; k < MLP_H; ++k) z = fmaf(fmaxf(h2[k], 0.0f), P[P_W3 + k], z);
    return z;
}

__global__ void __launch_bounds__(256) k_mlp_forward(const float *__restrict__ X, int n, const float *__restrict__ Pg,
                                                     float *__restrict__ z)
{
    __shared__ float P[MLP_NPARAM];
    for (int k = threadIdx.x; k < MLP_NPARAM; k += blockDim.x) P[k] = Pg[k];
    __syncthreads();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[MLP_IN];
#pragma unroll
    for (int i = 0; i < MLP_IN; ++i) x[i] = X[(size_t)s * MLP_IN + i];
    z[s] = mlp_eval(P, x);
}

// ---------------------------------------------------------------------------
// gradient of L = sum_s w_s * BCE(z_s, y_s) (BCE with logits) with respect to
// every parameter; per-block partial sums in fixed order, then a fixed-order
// reduction over blocks (deterministic)
// ---------------------------------------------------------------------------
// 32 samples per block (4,096 samples: 128 blocks, one wave on 152 SMs) and every
// layer as a register tile: a thread takes 2 samples x 4 units of an
// activation, 4 x 4 (2 x 4) weights of a gradient, so each 16-byte word from
// shared memory feeds 4 to 8 multiply-adds (one output per thread, two 4-byte
// words per multiply-add, took 45 us on 64 blocks).  Bound by shared-memory
// bandwidth and the block's five barriers.
struct GradSmem {
    float P[MLP_NPARAM + 3];               // rounded to 16 bytes
    float W2T[MLP_H][MLP_H + 4];           // W2 transposed
    float X[GRAD_S][MLP_IN];
    float H1[GRAD_S][MLP_H], H2[GRAD_S][MLP_H];
    float D1[GRAD_S][MLP_H], D2[GRAD_S][MLP_H];
    float dz[GRAD_S], loss[GRAD_S];
};
static_assert(MLP_NPARAM % 4 == 1 && P_B1 % 4 == 0 && P_W2 % 4 == 0 && P_B2 % 4 == 0 && P_W3 % 4 == 0,
              "16-byte parameter rows");
static_assert(GRAD_THREADS == (GRAD_S / 2) * (MLP_H / 4), "two samples x four units a thread");

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
// (the caller's scratch is aligned to a float only)
__device__ __forceinline__ void st4(float *p, const float4 &v)
{
    p[0] = v.x;
    p[1] = v.y;
    p[2] = v.z;
    p[3] = v.w;
}
__device__ __forceinline__ void fma4(float4 &a, float x, const float4 &w)
{
    a.x = fmaf(x, w.x, a.x);
    a.y = fmaf(x, w.y, a.y);
    a.z = fmaf(x, w.z, a.z);
    a.w = fmaf(x, w.w, a.w);
}

// a[q] += sum_k A[s + q][k] * W[k][j .. j + 3] for the thread's two samples
template <int K, int LD>
__device__ __forceinline__ void rows_times(const float (*A)[K], const float *W, int s, int j, float4 a[2])
{
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 x0 = ld4(&A[s][k]), x1 = ld4(&A[s + 1][k]);
        const float4 w0 = ld4(W + (k + 0) * LD + j), w1 = ld4(W + (k + 1) * LD + j), w2 = ld4(W + (k + 2) * LD + j),
                     w3 = ld4(W + (k + 3) * LD + j);
        fma4(a[0], x0.x, w0);
        fma4(a[1], x1.x, w0);
        fma4(a[0], x0.y, w1);
        fma4(a[1], x1.y, w1);
        fma4(a[0], x0.z, w2);
        fma4(a[1], x1.z, w2);
        fma4(a[0], x0.w, w3);
        fma4(a[1], x1.w, w3);
    }
}

__device__ __forceinline__ float4 relu4(const float4 &a)
{
    return make_float4(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f), fmaxf(a.z, 0.0f), fmaxf(a.w, 0.0f));
}

__global__ void __launch_bounds__(GRAD_THREADS) k_mlp_grad_part(const float *__restrict__ X,
                                                                const float *__restrict__ y,
                                                                const float *__restrict__ w, int n,
                                                                const float *__restrict__ Pg,
                                                                float *__restrict__ part)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem &G = *reinterpret_cast<GradSmem *>(smem_raw);
    const int tid = threadIdx.x;
    const int s0 = blockIdx.x * GRAD_S;
    const int ns = min(GRAD_S, n - s0);
    for (int k = tid; k < MLP_NPARAM; k += GRAD_THREADS) {
        const float p = Pg[k];
        G.P[k] = p;
        if (k >= P_W2 && k < P_B2) G.W2T[(k - P_W2) % MLP_H][(k - P_W2) / MLP_H] = p;
    }
    for (int k = tid; k < GRAD_S * MLP_IN; k += GRAD_THREADS) {
        const int s = k / MLP_IN, i = k % MLP_IN;
        G.X[s][i] = s < ns ? X[(size_t)(s0 + s) * MLP_IN + i] : 0.0f;
    }
    __syncthreads();
    // the thread's samples and units
    const int s = 2 * (tid / (MLP_H / 4)), j = 4 * (tid % (MLP_H / 4));
    float4 h[2];
    h[0] = h[1] = ld4(G.P + P_B1 + j);
    rows_times<MLP_IN, MLP_H>(G.X, G.P + P_W1, s, j, h);
    for (int q = 0; q < 2; ++q) *reinterpret_cast<float4 *>(&G.H1[s + q][j]) = relu4(h[q]);
    __syncthreads();
    h[0] = h[1] = ld4(G.P + P_B2 + j);
    rows_times<MLP_H, MLP_H>(G.H1, G.P + P_W2, s, j, h);
    // z: the 16 threads of a sample pair are neighbouring lanes
    const float4 w3 = ld4(G.P + P_W3 + j);
    float z[2];
    for (int q = 0; q < 2; ++q) {
        h[q] = relu4(h[q]);
        *reinterpret_cast<float4 *>(&G.H2[s + q][j]) = h[q];
        z[q] = fmaf(h[q].x, w3.x, fmaf(h[q].y, w3.y, fmaf(h[q].z, w3.z, h[q].w * w3.w)));
        for (int o = 1; o < MLP_H / 4; o <<= 1) z[q] += __shfl_xor_sync(0xffffffffu, z[q], o);
        z[q] += G.P[P_B3];
    }
    for (int q = 0; q < 2; ++q) {
        float dz = 0.0f, l = 0.0f;
        if (s + q < ns) {
            const float yy = y[s0 + s + q], ww = w[s0 + s + q];
            const float sg = 1.0f / (1.0f + expf(-z[q]));
            dz = ww * (sg - yy);
            l = ww * (fmaxf(z[q], 0.0f) - z[q] * yy + log1pf(expf(-fabsf(z[q]))));
        }
        if (j == 0) {
            G.dz[s + q] = dz;
            G.loss[s + q] = l;
        }
        *reinterpret_cast<float4 *>(&G.D2[s + q][j]) =
            make_float4(h[q].x > 0.0f ? dz * w3.x : 0.0f, h[q].y > 0.0f ? dz * w3.y : 0.0f,
                        h[q].z > 0.0f ? dz * w3.z : 0.0f, h[q].w > 0.0f ? dz * w3.w : 0.0f);
    }
    __syncthreads();
    h[0] = h[1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    rows_times<MLP_H, MLP_H + 4>(G.D2, &G.W2T[0][0], s, j, h);
    for (int q = 0; q < 2; ++q) {
        const float4 a = ld4(&G.H1[s + q][j]);
        *reinterpret_cast<float4 *>(&G.D1[s + q][j]) =
            make_float4(a.x > 0.0f ? h[q].x : 0.0f, a.y > 0.0f ? h[q].y : 0.0f, a.z > 0.0f ? h[q].z : 0.0f,
                        a.w > 0.0f ? h[q].w : 0.0f);
    }
    __syncthreads();
    // weight gradients: rows r .. of W2 (4) and of W1 (2), columns c .. c + 3
    float *out = part + (size_t)blockIdx.x * (MLP_NPARAM + 1);
    const int c = 4 * (tid % 16), r = tid / 16;
    float4 g2[4], g1[2];
    for (int q = 0; q < 4; ++q) g2[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    g1[0] = g1[1] = g2[0];
#pragma unroll 4
    for (int k = 0; k < GRAD_S; ++k) {
        const float4 d2 = ld4(&G.D2[k][c]), d1 = ld4(&G.D1[k][c]), a = ld4(&G.H1[k][4 * r]);
        const float2 x = *reinterpret_cast<const float2 *>(&G.X[k][2 * r]);
        fma4(g2[0], a.x, d2);
        fma4(g2[1], a.y, d2);
        fma4(g2[2], a.z, d2);
        fma4(g2[3], a.w, d2);
        fma4(g1[0], x.x, d1);
        fma4(g1[1], x.y, d1);
    }
    for (int q = 0; q < 4; ++q) st4(out + P_W2 + (4 * r + q) * MLP_H + c, g2[q]);
    for (int q = 0; q < 2; ++q) st4(out + P_W1 + (2 * r + q) * MLP_H + c, g1[q]);
    // biases, w3 and the loss: one sum per thread
    if (tid < 3 * MLP_H + 2) {
        const int u = tid % MLP_H, kind = tid / MLP_H;
        float g = 0.0f;
        for (int k = 0; k < GRAD_S; ++k) {
            if (kind == 0) g += G.D1[k][u];
            else if (kind == 1) g += G.D2[k][u];
            else if (kind == 2) g = fmaf(G.dz[k], G.H2[k][u], g);
            else g += u == 0 ? G.dz[k] : G.loss[k];
        }
        out[kind == 0 ? P_B1 + u : (kind == 1 ? P_B2 + u : (kind == 2 ? P_W3 + u : P_B3 + u))] = g;
    }
}

// sums of the blocks' parts in a fixed order: warps take every eighth block, lanes neighbouring parameters
constexpr int RED_WARPS = 8;

__global__ void __launch_bounds__(32 * RED_WARPS) k_mlp_grad_reduce(const float *__restrict__ part, int nblocks,
                                                                   float *__restrict__ grad, float *__restrict__ loss)
{
    __shared__ float sum[RED_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = blockIdx.x * 32 + lane;
    float g = 0.0f;
    if (q <= MLP_NPARAM)
        for (int b = warp; b < nblocks; b += RED_WARPS) g += part[(size_t)b * (MLP_NPARAM + 1) + q];
    sum[warp][lane] = g;
    __syncthreads();
    if (warp == 0 && q <= MLP_NPARAM) {
        for (int k = 1; k < RED_WARPS; ++k) g += sum[k][lane];
        if (q < MLP_NPARAM) grad[q] = g;
        else if (loss) *loss = g;
    }
}

__global__ void k_adam(float *__restrict__ P, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= MLP_NPARAM) return;
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.0f - b1) * gq;
    const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    P[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

// ---------------------------------------------------------------------------
// tile features, targets, certificate
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tile_centre(const Grid &G, long long tile, double t[3])
{
    int tc[3];
    tile_coords(G, tile, tc);
    for (int a = 0; a < 3; ++a) t[a] = G.lo[a] + G.h * ((double)(TILE * (tc[a] + G.toff[a])) + 0.5 * (TILE - 1));
}

__device__ __forceinline__ long long floor_ll(double v) { return (long long)floor(v); }

__device__ void tile_features(const Model &M, const Grid &G, int mol, long long tile, float *f)
{
    const CellGrid cg = M.cg[mol];
    double t[3];
    tile_centre(G, tile, t);
    long long ci[3];
    for (int a = 0; a < 3; ++a) {
        const double u = (t[a] - cg.clo[a]) / M.cell;
        ci[a] = floor_ll(u);
        f[27 + a] = fminf(fmaxf((float)(u - (double)ci[a]) - 0.5f, -1.5f), 1.5f);
    }
    int tot = 0, k = 0;
    for (int dx = -1; dx <= 1; ++dx)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dz = -1; dz <= 1; ++dz, ++k) {
                const long long a = ci[0] + dx, b = ci[1] + dy, c = ci[2] + dz;
                int n = 0;
                if (a >= 0 && b >= 0 && c >= 0 && a < cg.cn[0] && b < cg.cn[1] && c < cg.cn[2]) {
                    const int id = cg.coff + (int)((a * cg.cn[1] + b) * cg.cn[2] + c);
                    n = M.cell_start[id + 1] - M.cell_start[id];
                }
                tot += n;
                f[k] = log1pf((float)n);
            }
    f[30] = log1pf((float)tot);
    f[31] = (float)(TILE * G.h / M.cell);
}

__global__ void k_tile_features(Model M, Batch B, float *__restrict__ feat)
{
    for (long long base = (long long)blockIdx.x * blockDim.x; base < B.n_tiles; base += (long long)gridDim.x * blockDim.x) {
        const long long gt = base + threadIdx.x;
        if (gt < B.n_tiles) {
            const int mol = mol_of_tile(B, gt);
            const Grid &G = B.grid[mol];
            float f[MLP_IN];
            tile_features(M, G, mol, gt - G.tile0, f);
            for (int i = 0; i < MLP_IN; ++i) feat[(size_t)gt * MLP_IN + i] = f[i];
        }
    }
}

// 1 when the tile's labels are not all equal (the tile holds surface)
__global__ void k_tile_targets(Batch B, const int8_t *__restrict__ labels_all, uint8_t *__restrict__ target)
{
    const int lane = threadIdx.x & 31;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long gt = w; gt < B.n_tiles; gt += nw) {
        const int mol = mol_of_tile(B, gt);
        const Grid &G = B.grid[mol];
        const int8_t *labels = labels_all + G.lab0;
        int tc[3];
        tile_coords(G, gt - G.tile0, tc);
        int mn = 127, mx = -128;
        for (int p = lane; p < TILE_PTS; p += 32) {
            const long long g0 = (long long)TILE * tc[0] + (p >> 6), g1 = (long long)TILE * tc[1] + ((p >> 3) & 7),
                            g2 = (long long)TILE * tc[2] + (p & 7);
            if (g0 >= G.dims[0] || g1 >= G.dims[1] || g2 >= G.dims[2]) continue;
            const int v = labels[(g0 * G.dims[1] + g1) * G.dims[2] + g2];
            mn = min(mn, v);
            mx = max(mx, v);
        }
        for (int o = 16; o > 0; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane == 0) target[gt] = mn != mx ? 1 : 0;
    }
}

// Certificate of one tile (whole warp): 0 all points outside, 1 all inside,
// -1 neither proven.  FP32 on the double-float atom copies (relative to the
// grid origin) and squared distances, with the rounding covered: a squared
// distance carries a relative error below 1e-6, the thresholds get 1e-4 A of
// slack, so a certified answer is exact.
__device__ int certify_tile(const Model &M, const Grid &G, int mol, long long tile)
{
    const int lane = threadIdx.x & 31;
    const CellGrid &cg = M.cg[mol];
    int tc[3];
    tile_coords(G, tile, tc);
    float th[3], tl[3];
    int c0[3], c1[3];
    const float delta = (float)(0.5 * (TILE - 1) * G.h * 1.7320508075688772);
    const float slack = 1e-4f, rel_lo = 1.0f - 2e-6f, rel_hi = 1.0f + 2e-6f;
    const float rp = (float)M.rp;
    // every atom that can matter lies within delta + R_max of t: the cells that
    // ball meets, indices in FP32 with 1e-2 A of room for their rounding (no
    // FP64 division: a handful per tile would bound the whole kernel)
    const float icell = 1.0f / (float)M.cell;
    const float reach = (delta + (float)M.Rmax + 1e-2f) * icell;
    for (int a = 0; a < 3; ++a) {
        const double rel = G.h * ((double)(TILE * (tc[a] + G.toff[a])) + 0.5 * (TILE - 1));
        th[a] = (float)rel;
        tl[a] = (float)(rel - (double)th[a]);
        const float u = ((float)(G.lo[a] - cg.clo[a]) + th[a]) * icell;  // centre in cell units
        c0[a] = max((int)floorf(u - reach), 0);
        c1[a] = min((int)floorf(u + reach), cg.cn[a] - 1);
    }
    bool not_out = false, in = false;
    auto test = [&](int k) {
        const float4 hi = M.atom_hi[k], lo = M.atom_lo[k];
        const float dx = (hi.x - th[0]) + (lo.x - tl[0]);
        const float dy = (hi.y - th[1]) + (lo.y - tl[1]);
        const float dz = (hi.z - th[2]) + (lo.z - tl[2]);
        const float d2 = dx * dx + dy * dy + dz * dz;
        const float to = hi.w + rp + delta + slack;  // outside needs d >= R + delta
        if (d2 * rel_lo < to * to) not_out = true;
        const float ti = hi.w - delta - slack;  // inside needs d < r - delta
        if (ti > 0.0f && d2 * rel_hi < ti * ti) in = true;
    };
    // per (x, y) cell column, the atoms of its z cells are contiguous: one lane
    // per column reads its range and the lanes walk the ranges laid end to end
    // (column by column, two dependent loads each, cost a far tile nine round
    // trips to find no atom)
    const int n0 = c1[0] - c0[0] + 1, n1 = c1[1] - c0[1] + 1;
    if (n0 <= 0 || n1 <= 0 || c0[2] > c1[2]) return 0;
    if ((long long)n0 * n1 <= 32) {
        int start = 0, len = 0;
        if (lane < n0 * n1) {
            const int id0 = cg.coff + ((c0[0] + lane / n1) * cg.cn[1] + c0[1] + lane % n1) * cg.cn[2];
            start = M.cell_start[id0 + c0[2]];
            len = M.cell_start[id0 + c1[2] + 1] - start;
        }
        int end = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        start -= end - len;  // atom of position t in column r: start[r] + t
        const int total = __shfl_sync(0xffffffffu, end, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int r = 0;  // columns that end at or before t
            for (int q = 0; q < n0 * n1 - 1; ++q) r += t >= __shfl_sync(0xffffffffu, end, q) ? 1 : 0;
            const int k = __shfl_sync(0xffffffffu, start, r) + t;
            if (t < total) test(k);
        }
    } else {
        for (int a = c0[0]; a <= c1[0]; ++a)
            for (int b = c0[1]; b <= c1[1]; ++b) {
                const int id0 = cg.coff + (a * cg.cn[1] + b) * cg.cn[2];
                const int e = M.cell_start[id0 + c1[2] + 1];
                for (int k = M.cell_start[id0 + c0[2]] + lane; k < e; k += 32) test(k);
            }
    }
    if (!__any_sync(0xffffffffu, not_out)) return 0;
    if (__any_sync(0xffffffffu, in)) return 1;
    return -1;
}

// Proposer: features and tensor-core score per tile (thread per tile, 128
// tiles per CTA step), then the certificate for the tiles scored far (warp
// per tile); tiles certified inside are filled (the labels start as outside
// everywhere), the others flagged for the exact classification.  mode 1: MLP +
// certificate; mode 2: certificate on every tile.  Bound by the latency of the
// cell look-ups; filling the outside tiles here, 8-byte rows at any alignment,
// cost more than clearing all labels at HBM speed does.
__global__ void __launch_bounds__(PROP_THREADS) k_propose(Model M, Batch B, int mode, const float *__restrict__ Pg,
                                                          float z_far, int8_t *__restrict__ labels_all,
                                                          int *__restrict__ need,
                                                          int *__restrict__ counts, int *__restrict__ err,
                                                          long long wait_limit)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    TcSmem &T = *reinterpret_cast<TcSmem *>(smem_raw);
    __shared__ int far_list[PROP_THREADS];
    __shared__ int n_far;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t phase = 0;
    int proposed = 0, certified = 0;  // the warp's tiles
    if (mode == 1) tc_setup(T, Pg, wait_limit);
    for (long long base = (long long)blockIdx.x * PROP_THREADS; base < B.n_tiles;
         base += (long long)gridDim.x * PROP_THREADS) {
        if (threadIdx.x == 0) n_far = 0;
        __syncthreads();
        const long long gt = base + threadIdx.x;
        const bool valid = gt < B.n_tiles;
        bool far = valid;
        if (mode == 1) {
            float f[MLP_IN];
            if (valid) {
                const int mol = mol_of_tile(B, gt);
                const Grid &G = B.grid[mol];
                tile_features(M, G, mol, gt - G.tile0, f);
            }
            const float zt = tc_score(T, f, valid, phase, err);  // every thread: block-wide barriers inside
            far = valid && zt < z_far;
        }
        if (valid) need[gt] = 1;
        if (far) far_list[atomicAdd(&n_far, 1)] = (int)threadIdx.x;
        __syncthreads();
        const int nf = n_far;
        for (int k = warp; k < nf; k += PROP_THREADS / 32) {
            const long long g2 = base + far_list[k];
            const int mol = mol_of_tile(B, g2);
            const Grid &G = B.grid[mol];
            const long long tile = g2 - G.tile0;
            const int r = certify_tile(M, G, mol, tile);
            if (r == 1) {
                int8_t *labels = labels_all + G.lab0;
                int tc[3];
                tile_coords(G, tile, tc);
                for (int p = lane; p < TILE_PTS; p += 32) {
                    const long long g0 = (long long)TILE * tc[0] + (p >> 6),
                                    g1 = (long long)TILE * tc[1] + ((p >> 3) & 7), gz = (long long)TILE * tc[2] + (p & 7);
                    if (g0 < G.dims[0] && g1 < G.dims[1] && gz < G.dims[2])
                        labels[(g0 * G.dims[1] + g1) * G.dims[2] + gz] = (int8_t)r;
                }
            }
            if (r >= 0 && lane == 0) need[g2] = 0;
            proposed += 1;
            certified += r >= 0 ? 1 : 0;
        }
        __syncthreads();
    }
    if (lane == 0 && proposed) {
        atomicAdd(&counts[0], proposed);
        atomicAdd(&counts[1], certified);
    }
    if (mode == 1) tc_teardown(T, phase);
}

// The tensor-core MLP on arbitrary rows (n x 32 features): z = MLP(X), BF16
// weights and activations, FP32 accumulation (the proposer's scoring path).
__global__ void __launch_bounds__(PROP_THREADS) k_mlp_forward_tc(const float *__restrict__ X, int n,
                                                                 const float *__restrict__ Pg, float *__restrict__ z,
                                                                 int *__restrict__ err)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    TcSmem &T = *reinterpret_cast<TcSmem *>(smem_raw);
    uint32_t phase = 0;
    tc_setup(T, Pg);
    for (long long base = (long long)blockIdx.x * PROP_THREADS; base < n; base += (long long)gridDim.x * PROP_THREADS) {
        const long long s = base + threadIdx.x;
        const bool valid = s < n;
        float x[MLP_IN];
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) x[i] = valid ? X[s * MLP_IN + i] : 0.0f;
        const float v = tc_score(T, x, valid, phase, err);
        if (valid) z[s] = v;
    }
    tc_teardown(T, phase);
}

// list of the tiles flagged in `need`, from their exclusive scan
__global__ void k_compact(long long n, const int *__restrict__ need, const int *__restrict__ pos,
                          int *__restrict__ list)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && need[i]) list[pos[i]] = (int)i;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static size_t grad_smem() { return sizeof(GradSmem); }

void mlp_init()
{
    cudaFuncSetAttribute(k_mlp_grad_part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)grad_smem());
    cudaFuncSetAttribute(k_propose, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TcSmem));
    cudaFuncSetAttribute(k_mlp_forward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TcSmem));
}

int launch_mlp_forward(const float *X, int n, const float *P, float *z, cudaStream_t st)
{
    if (n <= 0) return 0;
    k_mlp_forward<<<(n + 255) / 256, 256, 0, st>>>(X, n, P, z);
    return 1;
}

long long mlp_grad_scratch(int n) { return (long long)((n + GRAD_S - 1) / GRAD_S) * (MLP_NPARAM + 1); }

int launch_mlp_grad(const float *X, const float *y, const float *w, int n, const float *P, float *part, float *grad,
                    float *loss, cudaStream_t st)
{
    if (n <= 0) return 0;
    const int nb = (n + GRAD_S - 1) / GRAD_S;
    k_mlp_grad_part<<<nb, GRAD_THREADS, grad_smem(), st>>>(X, y, w, n, P, part);
    k_mlp_grad_reduce<<<(MLP_NPARAM + 1 + 31) / 32, 32 * RED_WARPS, 0, st>>>(part, nb, grad, loss);
    return 2;
}

int launch_adam(float *P, const float *g, float *m, float *v, int step, float lr, cudaStream_t st)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    k_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, st>>>(P, g, m, v, lr, b1, b2, eps, c1, c2);
    return 1;
}

int launch_tile_features(const Model &M, const Batch &B, float *feat, cudaStream_t st)
{
    const long long g = std::min<long long>((B.n_tiles + 127) / 128, 1 << 20);
    k_tile_features<<<(unsigned)std::max(g, 1LL), 128, 0, st>>>(M, B, feat);
    return 1;
}

int launch_tile_targets(const Batch &B, const int8_t *labels, uint8_t *target, cudaStream_t st)
{
    const long long g = std::min<long long>((B.n_tiles + 7) / 8, 1 << 20);
    k_tile_targets<<<(unsigned)std::max(g, 1LL), 256, 0, st>>>(B, labels, target);
    return 1;
}

// persistent grids: at most 4 CTAs per SM, so every CTA's 128 TMEM columns fit (512 per SM)
static int tc_grid(long long rows)
{
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long need = (rows + PROP_THREADS - 1) / PROP_THREADS;
    return (int)std::max(1LL, std::min(need, 4LL * nsm));
}

int launch_propose(const Model &M, const Batch &B, int mode, const float *P, float z_far, int8_t *labels,
                   int *need, int *counts, int *err, long long wait_limit, cudaStream_t st)
{
    k_propose<<<tc_grid(B.n_tiles), PROP_THREADS, sizeof(TcSmem), st>>>(M, B, mode, P, z_far, labels, need,
                                                                       counts, err, wait_limit);
    return 1;
}

int launch_mlp_forward_tc(const float *X, int n, const float *P, float *z, int *err, cudaStream_t st)
{
    if (n <= 0) return 0;
    k_mlp_forward_tc<<<tc_grid(n), PROP_THREADS, sizeof(TcSmem), st>>>(X, n, P, z, err);
    return 1;
}

int launch_compact(long long n, const int *need, const int *pos, int *list, cudaStream_t st)
{
    if (n <= 0) return 0;
    k_compact<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, need, pos, list);
    return 1;
}

}  // namespace eses
