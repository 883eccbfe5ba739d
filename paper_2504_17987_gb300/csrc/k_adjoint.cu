// Adjoint of the zero-shift correlation score with respect to the
// displacement grid (differentiation of the deformation step of paper Sec. 2).
//
//   S = sum_w C_w(0),  C_w = sum a~ b~ / sqrt(E_A E_B),  B'(x) = B(x + d(x)),
//   d(x) = sum_k phi_k(x) d_k  (bilinear weights, border value outside the hull)
//   dC_w/dB'(x) = a~(x)/sqrt(E_A E_B) - C_w b~(x)/E_B
//   dS/dd_k = sum_x phi_k(x) grad B(x + d(x)) sum_{w containing x} dC_w/dB'(x)
//
// Deterministic kernels, no floating-point atomics.  G = gcd(w, s): every
// window is a union of G x G blocks, and all pixels of a block lie in the same
// windows.
//   1. adj_blocks: d(x), B'(x) and the in-cell gradient of B, once per pixel, and
//      per block the means of A and B' and their centred second moments
//                                                          -> px4, blk, blk_ab
//   2. adj_windows: the moments of a window from its blocks, C_w, and the score
//      (sums of CTAs, added in a fixed order by the last one)  -> win4, score
//   3. adj_nodes: per tile of nodes, the window sums of dC_w/dB' of every block it
//      touches, dS/dB' grad B of every pixel, and the node sums, separable in the
//      bilinear weights, along x and then y                         -> grad
// One 1 MP pair moves a few megabytes through L2: the chain is bound by the
// latency of its launches, so there are three (two for the score alone).  As
// seven launches it took 73 us (125 x 125 nodes, score and gradient); now 30, of which
// the host's side of the call is 25.
// Blocks above 32 px, steps below 3 px and steps whose node tiles do not fit shared memory run
// steps 1 and 3 as separate launches over pixels, rows and nodes.
#include <algorithm>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "grid_interp.cuh"
#include "rpiv_internal.h"

namespace rpiv {

namespace {

constexpr float kTauPerPixel = 1e-6f;

__device__ __forceinline__ float wsum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void axis_wt(int pos, int n, float c0, int s, int &i0, int &i1, float &t)
{
    if (n <= 1) {
        i0 = i1 = 0;
        t = 0.f;
        return;
    }
    float f = over_step((float)pos - c0, s);
    f = fminf(fmaxf(f, 0.f), (float)(n - 1));
    int ia = (int)floorf(f);
    if (ia > n - 2) ia = n - 2;
    i0 = ia;
    i1 = ia + 1;
    t = f - (float)ia;
}

// bilinear weight of node i at a pixel position along one axis
__device__ __forceinline__ float node_wt(int pos, int i, int n, float c0, int s)
{
    int i0, i1;
    float t;
    axis_wt(pos, n, c0, s, i0, i1, t);
    return (i0 == i ? 1.f - t : 0.f) + (i1 == i && i1 != i0 ? t : 0.f);
}

__device__ __forceinline__ void field(const AdjArgs &a, int x, int y, float &du, float &dv)
{
    const float c0 = 0.5f * (float)(a.w - 1);
    int i0, i1, j0, j1;
    float tx, ty;
    axis_wt(x, a.nx, c0, a.s, i0, i1, tx);
    axis_wt(y, a.ny, c0, a.s, j0, j1, ty);
    const float *u = a.u, *v = a.v;
    float t0 = u[j0 * a.nx + i0] + tx * (u[j0 * a.nx + i1] - u[j0 * a.nx + i0]);
    float t1 = u[j1 * a.nx + i0] + tx * (u[j1 * a.nx + i1] - u[j1 * a.nx + i0]);
    du = t0 + ty * (t1 - t0);
    t0 = v[j0 * a.nx + i0] + tx * (v[j0 * a.nx + i1] - v[j0 * a.nx + i0]);
    t1 = v[j1 * a.nx + i0] + tx * (v[j1 * a.nx + i1] - v[j1 * a.nx + i0]);
    dv = t0 + ty * (t1 - t0);
}

// integer pixels placed under the exponent of 2^23 instead of converted (exact)
__device__ __forceinline__ float as_float(uint8_t v) { return __uint_as_float(0x4B000000u | (uint32_t)v) - 8388608.f; }
__device__ __forceinline__ float as_float(uint16_t v) { return __uint_as_float(0x4B000000u | (uint32_t)v) - 8388608.f; }
__device__ __forceinline__ float as_float(float v) { return v; }

template <typename T>
__device__ __forceinline__ float px(const unsigned char *img, long long pitch, int x, int y)
{
    return as_float(__ldg(reinterpret_cast<const T *>(img + (long long)y * pitch) + x));
}

// B' = bilinear(B) at (x + du, y + dv), clamp-to-edge, and its in-cell gradient.
template <typename T>
__device__ __forceinline__ float deformed(const AdjArgs &a, const unsigned char *B, int x, int y, float du, float dv,
                                          float *gx, float *gy)
{
    if (!(fabsf(du) <= 1048576.f && fabsf(dv) <= 1048576.f)) {
        du = isfinite(du) ? fminf(fmaxf(du, -1048576.f), 1048576.f) : 0.f;
        dv = isfinite(dv) ? fminf(fmaxf(dv, -1048576.f), 1048576.f) : 0.f;
    }
    // floors: the add rounds down at a unit in the last place of one
    const float fx = __fadd_rd(du, 12582912.f), fy = __fadd_rd(dv, 12582912.f);
    const int ix = x + (__float_as_int(fx) - 0x4B400000), iy = y + (__float_as_int(fy) - 0x4B400000);
    const float tx = du - (fx - 12582912.f), ty = dv - (fy - 12582912.f);
    const T *p00, *p10, *p01, *p11;
    if ((unsigned)ix < (unsigned)(a.W - 1) && (unsigned)iy < (unsigned)(a.H - 1)) {
        p00 = reinterpret_cast<const T *>(B + (long long)iy * a.pitch) + ix;
        p10 = p00 + 1;
        p01 = reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(p00) + a.pitch);
        p11 = p01 + 1;
    } else {
        const int x0 = min(max(ix, 0), a.W - 1), x1 = min(max(ix + 1, 0), a.W - 1);
        const int y0 = min(max(iy, 0), a.H - 1), y1 = min(max(iy + 1, 0), a.H - 1);
        const T *r0 = reinterpret_cast<const T *>(B + (long long)y0 * a.pitch);
        const T *r1 = reinterpret_cast<const T *>(B + (long long)y1 * a.pitch);
        p00 = r0 + x0;
        p10 = r0 + x1;
        p01 = r1 + x0;
        p11 = r1 + x1;
    }
    const float b00 = as_float(__ldg(p00)), b10 = as_float(__ldg(p10));
    const float b01 = as_float(__ldg(p01)), b11 = as_float(__ldg(p11));
    *gx = (1.f - ty) * (b10 - b00) + ty * (b11 - b01);
    *gy = (1.f - tx) * (b01 - b00) + tx * (b11 - b10);
    const float top = b00 + tx * (b10 - b00), bot = b01 + tx * (b11 - b01);
    return top + ty * (bot - top);
}

// Workspace carve-up (floats, each part 256-byte aligned).
struct AdjWs {
    unsigned *ticket;  // CTAs of adj_windows that have finished; zero between calls
    float *part;       // their sums of C
    float4 *win4;      // per window: mean A, mean B', 1/sqrt(E_A E_B), C/E_B
    float4 *blk;       // per block: mean A, mean B', centred A.A, B'.B'
    float *blk_ab;     // per block: centred A.B'
    float4 *px4;       // per pixel: B', grad B at the deformed position, A
    float2 *pix_g;     // dS/dB' times grad B per pixel (separate launches)
    float2 *rows;      // per (image row, node column): the node's support summed along x (separate launches)
};

__host__ __device__ inline size_t up64(size_t n) { return (n + 63) & ~(size_t)63; }

__host__ __device__ inline int gcd_i(int a, int b)
{
    while (b) {
        const int t = a % b;
        a = b;
        b = t;
    }
    return a;
}

struct BlockGrid {
    int G, nbx, nby;  // block size; blocks across the windows' union
};

__host__ __device__ inline BlockGrid block_grid(int w, int s, int nx, int ny)
{
    BlockGrid b;
    b.G = gcd_i(w, s);
    b.nbx = ((nx - 1) * s + w) / b.G;
    b.nby = ((ny - 1) * s + w) / b.G;
    return b;
}

constexpr int WIN_CTA = 64;      // windows per CTA of adj_windows, WIN_LANES threads each
constexpr int WIN_LANES = 4;
constexpr int MAX_G = 32;        // blocks of adj_blocks
constexpr int NODE_SMEM = 192 * 1024;  // most shared memory of adj_nodes
constexpr int TILE_W = 64, TILE_H = 32;  // its tile is about TILE_W x TILE_H pixels, whole blocks

inline int win_ctas(int nx, int ny) { return (nx * ny + WIN_CTA - 1) / WIN_CTA; }

__host__ __device__ inline int max_i(int a, int b) { return a > b ? a : b; }
__host__ __device__ inline int min_i(int a, int b) { return a < b ? a : b; }

// support of node i along an axis of n nodes: the pixels strictly between its
// neighbours, extended to the image border for the first and last node
__host__ __device__ inline void support(int i, int n, float c0, int s, int len, int &lo, int &hi)
{
    lo = (i == 0) ? 0 : max_i(0, (int)floorf(c0 + (float)((i - 1) * s)) + 1);
    hi = (i == n - 1) ? len - 1 : min_i(len - 1, (int)ceilf(c0 + (float)((i + 1) * s)) - 1);
}

// Node tile of adj_nodes: about 64 x 32 pixels of node steps, and the largest
// region (union of its nodes' supports) and block range of such a tile.
struct NodeTile {
    int tx, ty, rw, rh, bw, bh, smem;
    bool ok;
};

int region(int n, int tile, float c0, int s, int len)
{
    int most = 0;
    for (int i = 0; i < n; i += tile) {
        int lo, hi, q;
        support(i, n, c0, s, len, lo, q);
        support(std::min(n, i + tile) - 1, n, c0, s, len, q, hi);
        most = std::max(most, hi - lo + 1);
    }
    return most;
}

NodeTile node_tile(int W, int H, int w, int s, int nx, int ny)
{
    NodeTile t;
    t.tx = std::min(nx, std::max(1, 64 / s));
    t.ty = std::min(ny, std::max(1, 32 / s));
    const float c0 = 0.5f * (float)(w - 1);
    t.rw = region(nx, t.tx, c0, s, W);
    t.rh = region(ny, t.ty, c0, s, H);
    const int G = gcd_i(w, s);
    t.bw = t.rw / G + 2;
    t.bh = t.rh / G + 2;
    // coefficients, the region's products (odd pitch), row sums, the axes' cells, weights and blocks
    const long long nblk = (long long)t.bw * t.bh;
    const long long bytes = 4ll * (6ll * nblk + 2ll * t.rh * (t.rw | 1) + 2ll * t.rh * t.tx + 3ll * t.rw + 3ll * t.rh);
    t.ok = bytes - 4ll * nblk <= 160 * 1024;  // so bytes <= NODE_SMEM: nblk takes at least 20 of the bytes on the left
    t.smem = t.ok ? (int)bytes : 0;
    return t;
}

size_t ws_floats(int W, int H, int w, int s, int nx, int ny, AdjWs *out, float *base)
{
    const BlockGrid bg = block_grid(w, s, nx, ny);
    size_t off = 0;
    auto take = [&](size_t n) {
        const size_t o = off;
        off += up64(n);
        return o;
    };
    const size_t o_ticket = take(1), o_part = take(win_ctas(nx, ny)), o_win = take(4ull * nx * ny);
    const size_t o_blk = take(4ull * bg.nbx * bg.nby), o_ab = take((size_t)bg.nbx * bg.nby), o_px = take(4ull * W * H);
    const bool tiles = node_tile(W, H, w, s, nx, ny).ok;
    const size_t o_pix = take(tiles ? 0 : 2ull * W * H), o_rows = take(tiles ? 0 : 2ull * H * nx);
    if (out) {
        out->ticket = reinterpret_cast<unsigned *>(base + o_ticket);
        out->part = base + o_part;
        out->win4 = reinterpret_cast<float4 *>(base + o_win);
        out->blk = reinterpret_cast<float4 *>(base + o_blk);
        out->blk_ab = base + o_ab;
        out->px4 = reinterpret_cast<float4 *>(base + o_px);
        out->pix_g = reinterpret_cast<float2 *>(base + o_pix);
        out->rows = reinterpret_cast<float2 *>(base + o_rows);
    }
    return off;
}

// Row-major walk over a width-W region by a fixed stride, without a division per step.
struct Walk {
    int x, y, sx, sy, W;
    __device__ __forceinline__ Walk(int start, int stride, int W_) : W(W_)
    {
        y = start / W_;
        x = start - y * W_;
        sy = stride / W_;
        sx = stride - sy * W_;
    }
    __device__ __forceinline__ void next()
    {
        x += sx;
        y += sy;
        if (x >= W) {
            x -= W;
            ++y;
        }
    }
};

// 1: a tile of whole blocks per CTA, one of its up to 64 columns and every
// fourth row per thread.  The node rows the tile touches are interpolated once
// per column (cuv), so that a pixel needs one interpolation along y.  B' and A
// wait in shared memory for the block sums (two passes: means, then centred
// moments), where a power of two of lanes shares a block so that the tile's
// blocks fill the CTA.  GRAD: also the pixels' values for step 3.  Bound by
// instruction issue.  Steps of 3 px and more.
constexpr int NODES_X = TILE_W / 3 + 3, NODES_Y = MAX_G / 3 + 3;

template <typename T, bool GRAD>
__global__ void __launch_bounds__(256) adj_blocks(const AdjArgs a, const AdjWs ws, const BlockGrid bg, int tbx, int tby,
                                                  int lanes)
{
    __shared__ float sa[MAX_G * (TILE_W + 1)], sb[MAX_G * (TILE_W + 1)];
    __shared__ float2 nodes[NODES_Y * NODES_X], cuv[NODES_Y * TILE_W];
    __shared__ int2 rinfo[MAX_G];  // node row's offset in cuv and weight
    const int tid = threadIdx.x, G = bg.G;
    const int bx0 = blockIdx.x * tbx, by0 = blockIdx.y * tby;
    const int nbx = min(tbx, bg.nbx - bx0), nby = min(tby, bg.nby - by0);
    const int x0 = bx0 * G, y0 = by0 * G, pw = nbx * G, ph = nby * G, pitch = TILE_W + 1;
    const float c0 = 0.5f * (float)(a.w - 1);
    const int lx = tid & (TILE_W - 1), ly = tid / TILE_W;
    int ilo, jlo, ihi, jhi, i0, q;
    float tx, t;
    axis_wt(x0, a.nx, c0, a.s, ilo, q, t);
    axis_wt(x0 + pw - 1, a.nx, c0, a.s, q, ihi, t);
    axis_wt(y0, a.ny, c0, a.s, jlo, q, t);
    axis_wt(y0 + ph - 1, a.ny, c0, a.s, q, jhi, t);
    const int nwn = ihi - ilo + 1, nhn = jhi - jlo + 1;
    for (int e = tid; e < nwn * nhn; e += 256) {
        const int jj = e / nwn, k = (jlo + jj) * a.nx + ilo + (e - jj * nwn);
        nodes[e] = make_float2(a.u[k], a.v[k]);
    }
    if (tid < ph) {
        int j0;
        axis_wt(y0 + tid, a.ny, c0, a.s, j0, q, t);
        rinfo[tid] = make_int2((j0 - jlo) * TILE_W, __float_as_int(t));
    }
    axis_wt(x0 + min(lx, pw - 1), a.nx, c0, a.s, i0, q, tx);
    __syncthreads();
    {
        const int ci = i0 - ilo, di = a.nx > 1 ? 1 : 0;
        for (int jj = ly; jj < nhn; jj += 256 / TILE_W) {
            const float2 p = nodes[jj * nwn + ci], r = nodes[jj * nwn + ci + di];
            cuv[jj * TILE_W + lx] = make_float2(p.x + tx * (r.x - p.x), p.y + tx * (r.y - p.y));
        }
    }
    __syncthreads();
    const unsigned char *A = (const unsigned char *)resolve(a.img_a, 0), *B = (const unsigned char *)resolve(a.img_b, 0);
    const int dj = a.ny > 1 ? TILE_W : 0;
    if (lx < pw) {
#pragma unroll 4
        for (int r = ly; r < ph; r += 256 / TILE_W) {
            const int x = x0 + lx, y = y0 + r;
            const int2 ri = rinfo[r];
            const float wy = __int_as_float(ri.y);
            const float2 n0 = cuv[ri.x + lx], n1 = cuv[ri.x + dj + lx];
            float gx, gy;
            const float b = deformed<T>(a, B, x, y, n0.x + wy * (n1.x - n0.x), n0.y + wy * (n1.y - n0.y), &gx, &gy);
            const float av = px<T>(A, a.pitch, x, y);
            sa[r * pitch + lx] = av;
            sb[r * pitch + lx] = b;
            if (GRAD) ws.px4[(long long)y * a.W + x] = make_float4(b, gx, gy, av);
        }
    }
    __syncthreads();
    const int l = tid & (lanes - 1), nb = nbx * nby;
    const float inv_n = 1.f / (float)(G * G);
    // means are summed relative to the least of the tile's corners, so that a background's
    // offset does not take the sums' digits (sparse particles on 100 counts, 32 px at 75 %:
    // gradient error 0.9e-6 instead of 1.35e-6)
    auto base = [&](const float *v) {
        const float *w = v + (ph - 1) * pitch;
        const float m = fminf(fminf(v[0], v[pw - 1]), fminf(w[0], w[pw - 1]));
        return isfinite(m) ? m : 0.f;
    };
    const float ra = base(sa), rb = base(sb);
    // warp-uniform trip count for the shuffles; threads past the last block repeat it
    for (int k0 = 0; k0 < nb; k0 += blockDim.x / lanes) {
        const int k = k0 + tid / lanes, kc = min(k, nb - 1);
        const int by = kc / nbx, bx = kc - by * nbx;
        const float *pa = sa + by * G * pitch + bx * G, *pb = sb + by * G * pitch + bx * G;
        float m0 = 0.f, m1 = 0.f;
        for (int x = l, y = 0;; x += lanes) {
            for (; x >= G; x -= G) ++y;
            if (y >= G) break;
            m0 += pa[y * pitch + x] - ra;
            m1 += pb[y * pitch + x] - rb;
        }
        for (int o = lanes >> 1; o > 0; o >>= 1) {
            m0 += __shfl_xor_sync(0xffffffffu, m0, o);
            m1 += __shfl_xor_sync(0xffffffffu, m1, o);
        }
        m0 = fmaf(m0, inv_n, ra);
        m1 = fmaf(m1, inv_n, rb);
        float caa = 0.f, cbb = 0.f, cab = 0.f;
        for (int x = l, y = 0;; x += lanes) {
            for (; x >= G; x -= G) ++y;
            if (y >= G) break;
            const float at = pa[y * pitch + x] - m0, bt = pb[y * pitch + x] - m1;
            caa = fmaf(at, at, caa);
            cbb = fmaf(bt, bt, cbb);
            cab = fmaf(at, bt, cab);
        }
        for (int o = lanes >> 1; o > 0; o >>= 1) {
            caa += __shfl_xor_sync(0xffffffffu, caa, o);
            cbb += __shfl_xor_sync(0xffffffffu, cbb, o);
            cab += __shfl_xor_sync(0xffffffffu, cab, o);
        }
        if (l == 0 && k < nb) {
            const int out = (by0 + by) * bg.nbx + bx0 + bx;
            ws.blk[out] = make_float4(m0, m1, caa, cbb);
            ws.blk_ab[out] = cab;
        }
    }
}

// 1, blocks above MAX_G and steps below 3 px: the pixels, then the blocks
template <typename T>
__global__ void adj_deform_kernel(const AdjArgs a, const AdjWs ws)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= a.W) return;
    const unsigned char *A = (const unsigned char *)resolve(a.img_a, 0), *B = (const unsigned char *)resolve(a.img_b, 0);
    float du, dv, gx, gy;
    field(a, x, y, du, dv);
    const float b = deformed<T>(a, B, x, y, du, dv, &gx, &gy);
    ws.px4[(long long)y * a.W + x] = make_float4(b, gx, gy, px<T>(A, a.pitch, x, y));
}

// WARPS warps per block: one, or eight for blocks above MAX_G, which are few and have
// thousands of pixels each (score of a 1 MP pair: 128 px windows without overlap, 64
// blocks, 229 -> 50 us; 64 px, 256 blocks, 73 -> 26 us).
template <int WARPS>
__global__ void __launch_bounds__(256) adj_block_kernel(const AdjArgs a, const AdjWs ws, const BlockGrid bg)
{
    __shared__ float part[5][WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, own = WARPS > 1 ? warp : 0;
    const int b = WARPS > 1 ? (int)blockIdx.x : (int)blockIdx.x * 8 + warp;
    if (b >= bg.nbx * bg.nby) return;  // (one warp per block only)
    // sum k of the warp, and, after a barrier, of the block's warps
    auto put = [&](float v, int k) {
        v = wsum(v);
        if (WARPS > 1 && lane == 0) part[k][own] = v;
        return v;
    };
    auto get = [&](float v, int k) {
        if (WARPS == 1) return v;
        float s = 0.f;
        for (int i = 0; i < WARPS; ++i) s += part[k][i];
        return s;
    };
    const int by = b / bg.nbx, bx = b - by * bg.nbx;
    const int G = bg.G, n = G * G;
    const float4 *p = ws.px4 + (long long)(by * G) * a.W + bx * G;
    const int start = own * 32 + lane;
    const float4 f = *p;  // the means are summed relative to the first pixel (offsets)
    float sa = 0.f, sb = 0.f;
    for (Walk e(start, 32 * WARPS, G); e.y < G; e.next()) {
        const float4 v = p[(long long)e.y * a.W + e.x];
        sa += v.w - f.w;
        sb += v.x - f.x;
    }
    sa = put(sa, 0);
    sb = put(sb, 1);
    if (WARPS > 1) __syncthreads();
    const float ma = f.w + get(sa, 0) / (float)n, mb = f.x + get(sb, 1) / (float)n;
    float caa = 0.f, cbb = 0.f, cab = 0.f;
    for (Walk e(start, 32 * WARPS, G); e.y < G; e.next()) {
        const float4 v = p[(long long)e.y * a.W + e.x];
        const float at = v.w - ma, bt = v.x - mb;
        caa = fmaf(at, at, caa);
        cbb = fmaf(bt, bt, cbb);
        cab = fmaf(at, bt, cab);
    }
    caa = put(caa, 2);
    cbb = put(cbb, 3);
    cab = put(cab, 4);
    if (WARPS > 1) __syncthreads();
    if (lane == 0 && own == 0) {
        ws.blk[b] = make_float4(ma, mb, get(caa, 2), get(cbb, 3));
        ws.blk_ab[b] = get(cab, 4);
    }
}

// The score from the sums of adj_windows' CTAs, by one warp in a fixed order.
// These few sums are as large as the result: in 64 bits, which adds no time.
__device__ __forceinline__ void score_sum(const AdjArgs &a, const AdjWs &ws, int n)
{
    const int lane = threadIdx.x & 31;
    double t = 0.;
    for (int k = lane; k < n; k += 32) t += (double)__ldcg(ws.part + k);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) *a.score_out = (float)t;
}

// 2: per window, its (w/G)^2 blocks combined: equal-size parts, so the mean
// is the mean of the block means, and each centred moment gains
// G^2 sum (mean_k - mean)(mean'_k - mean').  Two passes: a reference near the mean
// (the mean up to 4 x 4 blocks, that of four whole block rows above), then
// sum (d - mean d)^2 = sum d^2 - (sum d)^2 / k with d relative to it, whose second term
// is small.  (With d relative to the window's first block the two terms cancelled:
// score error against 64 bits 3.0e-7 instead of 2e-8 with 64 px windows at 6 px steps,
// gradient error 3.0e-6 instead of 2.2e-6 with 16 px windows at 5 px steps on sparse
// particles; relative to a mean of sixteen blocks 5.0e-7, whose few bits make the dark
// pixels' equal terms round all to one side.)
// The block rows of a window are dealt to WIN_LANES lanes and added by shuffles,
// so that its loads are in flight together.
// FEW: windows of up to 4 x 4 blocks (50 and 75 % overlap among them): a lane's row stays
// in registers, one latency for both passes.  A kernel of its own: the loops of larger
// windows want the CTAs that its registers cost (score of a 1 MP pair, 64 px at 4 px
// steps: 90 us in one, 71 apart, and 60 with the reference from four rows).
template <bool FEW>
__global__ void __launch_bounds__(WIN_CTA *WIN_LANES) adj_windows(const AdjArgs a, const AdjWs ws, const BlockGrid bg,
                                                                    bool sum_here)
{
    constexpr int NW = WIN_CTA * WIN_LANES / 32;
    __shared__ float sums[NW];
    __shared__ bool last;
    const int l = threadIdx.x & (WIN_LANES - 1), win = blockIdx.x * WIN_CTA + threadIdx.x / WIN_LANES;
    const int winc = min(win, a.nx * a.ny - 1);
    float C = 0.f;
    {
        const int j = winc / a.nx, i = winc - j * a.nx;
        const int G = bg.G, kb = a.w / G;
        const int b0 = (j * a.s / G) * bg.nbx + i * a.s / G;
        auto all = [](float v) {
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            return v + __shfl_xor_sync(0xffffffffu, v, 2);
        };
        static_assert(WIN_LANES == 4, "two shuffles, a row each up to 4 x 4 blocks");
        const float inv_k = 1.f / (float)(kb * kb), nb = (float)(G * G);
        // the reference, then the moments relative to it
        float2 f = make_float2(0.f, 0.f);
        float da = 0.f, db = 0.f, daa = 0.f, dbb = 0.f, dab = 0.f, ea = 0.f, eb = 0.f, num = 0.f;
        auto moments = [&](const float4 &o, float ab) {
            const float x = o.x - f.x, y = o.y - f.y;
            da += x;
            db += y;
            daa = fmaf(x, x, daa);
            dbb = fmaf(y, y, dbb);
            dab = fmaf(x, y, dab);
            ea += o.z;
            eb += o.w;
            num += ab;
        };
        if (FEW) {
            float4 o[4];
            float ab[4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (l < kb && p < kb) {
                    const int k = b0 + l * bg.nbx + p;
                    o[p] = ws.blk[k];
                    ab[p] = ws.blk_ab[k];
                    f.x += o[p].x;
                    f.y += o[p].y;
                }
            f.x = all(f.x) * inv_k;
            f.y = all(f.y) * inv_k;
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (l < kb && p < kb) moments(o[p], ab[p]);
        } else {
            const int q0 = (l * kb) >> 2;
#pragma unroll 4
            for (int p = 0; p < kb; ++p) {
                const float2 o = *reinterpret_cast<const float2 *>(ws.blk + b0 + q0 * bg.nbx + p);
                f.x += o.x;
                f.y += o.y;
            }
            f.x = all(f.x) * (1.f / (float)(4 * kb));
            f.y = all(f.y) * (1.f / (float)(4 * kb));
            for (int q = l; q < kb; q += WIN_LANES)
#pragma unroll 4
                for (int p = 0; p < kb; ++p) {
                    const int k = b0 + q * bg.nbx + p;
                    moments(ws.blk[k], ws.blk_ab[k]);
                }
        }
        da = all(da);
        db = all(db);
        const float ma = da * inv_k, mb = db * inv_k;
        ea = fmaf(nb, fmaf(-da, ma, all(daa)), all(ea));
        eb = fmaf(nb, fmaf(-db, mb, all(dbb)), all(eb));
        num = fmaf(nb, fmaf(-da, mb, all(dab)), all(num));
        const float tau = kTauPerPixel * (float)(a.w * a.w);
        const bool ok = ea > tau && eb > tau;
        const float rs = ok ? 1.f / sqrtf(ea * eb) : 0.f;
        const float c = ok ? num * rs : 0.f;
        if (win == winc && l == 0) {
            C = c;
            ws.win4[win] = make_float4(f.x + ma, f.y + mb, rs, ok ? c / eb : 0.f);
        }
    }
    if (!a.score_out) return;
    // the CTA's sum; without a gradient the sums of all CTAs are added by the
    // last one to finish, which leaves the ticket at zero for the next call
    // (otherwise by adj_nodes, beside its own work)
    const float v = wsum(C);
    if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int k = 0; k < NW; ++k) t += sums[k];
        ws.part[blockIdx.x] = t;
        last = false;
        if (sum_here) {
            __threadfence();
            last = atomicAdd(ws.ticket, 1u) == gridDim.x - 1;
        }
    }
    if (!sum_here) return;
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    score_sum(a, ws, gridDim.x);
    if (threadIdx.x == 0) *ws.ticket = 0u;
}

// sum over a block's windows of dC_w/dB' = (A - mean A_w) rs_w - (B' - mean B'_w) q_w
// (rs_w = 1/sqrt(E_A E_B), q_w = C_w/E_B).  Where the frames correlate the two products
// nearly cancel, and a rounding of the sums P = sum rs_w or Q = sum q_w is common to all
// of a block's pixels, which the sums over nodes do not average out.  So the difference
// is formed first: e P + y D - K with e = (A - rA) - rho B', y = B' - mB (the block's
// mean), D = sum (rho rs_w - q_w) and K the same with the windows' means.
//   rho  the gain q / rs of the middle window (its regression of A on B'; 0: it has none),
//   rA   the frames' offset mA - rho mB, cut to 12 bits so that A - rA is exact for integers;
// every term is then about as small as the result, whatever the contrasts and offsets of
// the frames are (256^2, 32 px at 75 %, error against 64 bits with B k times as bright:
// 2.2e-7 at every k, 2.2e-7 with A raised by 1000; with the plain difference A - B' it was
// 2.2e-7, 4.4e-7 at k = 4, 3.3e-5 at k = 255, and 6.7e-7 for the raised A).  P is the
// middle window's rs as often as there are windows, plus the sum of the small
// differences, which rounds once.
// LANES threads (a power of two, neighbours) share a block, every LANES-th window row
// each, and all of them must call.
struct BlockCoefs {
    float rA, mB, rho, P, D, K;
};

template <int LANES>
__device__ __forceinline__ BlockCoefs block_coefs(const AdjArgs &a, const AdjWs &ws, const BlockGrid &bg, int bx, int by)
{
    const int w = a.w, s = a.s, l = LANES > 1 ? threadIdx.x & (LANES - 1) : 0;
    // G divides w and s, so that indices are those of blocks (usually s = G)
    const int kb = w / bg.G, ks = s / bg.G;
    const int ilo = max(0, ks == 1 ? bx - kb + 1 : (bx - kb + ks) / ks), ihi = min(a.nx - 1, ks == 1 ? bx : bx / ks);
    const int jlo = max(0, ks == 1 ? by - kb + 1 : (by - kb + ks) / ks), jhi = min(a.ny - 1, ks == 1 ? by : by / ks);
    const float4 b = ws.blk[by * bg.nbx + bx];
    // every block of the windows' union lies in a window (s <= w): ilo <= ihi, jlo <= jhi
    const float4 m = ws.win4[((jlo + jhi) >> 1) * a.nx + ((ilo + ihi) >> 1)];
    BlockCoefs r{0.f, b.y, m.z > 0.f ? __fdividef(m.w, m.z) : 0.f, 0.f, 0.f, 0.f};  // rho need not be exact
    r.rA = __uint_as_float(__float_as_uint(fmaf(-r.rho, b.y, b.x)) & 0xfffff000u);
    for (int j = jlo + l; j <= jhi; j += LANES)
#pragma unroll 4
        for (int i = ilo; i <= ihi; ++i) {
            const float4 t = ws.win4[j * a.nx + i];
            const float d = fmaf(r.rho, t.z, -t.w);
            r.P += t.z - m.z;
            r.D += d;
            r.K = fmaf(fmaf(-r.rho, t.y, t.x - r.rA), t.z, fmaf(t.y - b.y, d, r.K));
        }
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
        r.P += __shfl_xor_sync(0xffffffffu, r.P, o);
        r.D += __shfl_xor_sync(0xffffffffu, r.D, o);
        r.K += __shfl_xor_sync(0xffffffffu, r.K, o);
    }
    r.P = fmaf((float)((ihi - ilo + 1) * (jhi - jlo + 1)), m.z, r.P);
    return r;
}

// a pixel (B', grad B, A) of the block
__device__ __forceinline__ float pixel_g(float4 v, const BlockCoefs &c)
{
    return fmaf(fmaf(-c.rho, v.x, v.w - c.rA), c.P, fmaf(v.x - c.mB, c.D, -c.K));
}

// 3: one tile of nodes per CTA.  Its region (the union of the nodes' supports)
// overlaps its neighbours' by one step; recomputing that is cheaper than a
// launch that hands the pixels over.  Bound by instruction issue.
__global__ void __launch_bounds__(256) adj_nodes(const AdjArgs a, const AdjWs ws, const BlockGrid bg, const NodeTile t,
                                                 int score_parts)
{
    extern __shared__ float4 smem4[];
    const int pitch = t.rw | 1;
    float4 *coef = smem4;                                              // bw x bh: rA, mB, rho, P
    float2 *coef2 = reinterpret_cast<float2 *>(coef + t.bw * t.bh);    // bw x bh: D, K
    float2 *gxy = coef2 + t.bw * t.bh;                                 // region, odd pitch
    float2 *rows = gxy + t.rh * pitch;                                 // rh x tx
    int2 *cw = reinterpret_cast<int2 *>(rows + t.rh * t.tx);           // per column: node cell and weight
    int2 *rw_ = cw + t.rw;                                             // per row
    int *cb = reinterpret_cast<int *>(rw_ + t.rh);                     // blocks of the columns and rows
    int *rb = cb + t.rw;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = bg.G;
    const float c0 = 0.5f * (float)(a.w - 1);
    const int n0 = blockIdx.x * t.tx, m0 = blockIdx.y * t.ty;
    const int nn = min(t.tx, a.nx - n0), mm = min(t.ty, a.ny - m0);
    int xl, xh, yl, yh, q;
    support(n0, a.nx, c0, a.s, a.W, xl, q);
    support(n0 + nn - 1, a.nx, c0, a.s, a.W, q, xh);
    support(m0, a.ny, c0, a.s, a.H, yl, q);
    support(m0 + mm - 1, a.ny, c0, a.s, a.H, q, yh);
    const int rw = xh - xl + 1, rh = yh - yl + 1;
    const int bx0 = xl / G, by0 = yl / G;
    for (int e = tid; e < rw + rh; e += 256) {
        int i0, i1;
        float wgt;
        if (e < rw) {
            axis_wt(xl + e, a.nx, c0, a.s, i0, i1, wgt);
            cw[e] = make_int2(i0, __float_as_int(wgt));
            cb[e] = (xl + e) / G - bx0;
        } else {
            axis_wt(yl + e - rw, a.ny, c0, a.s, i0, i1, wgt);
            rw_[e - rw] = make_int2(i0, __float_as_int(wgt));
            rb[e - rw] = ((yl + e - rw) / G - by0) * t.bw;
        }
    }
    // the blocks' coefficients: a warp per block row, four lanes per block (the
    // same trip count for all of a warp's lanes: they meet in the shuffles)
    const int bw = min(xh / G, bg.nbx - 1) - bx0 + 1, bh = min(yh / G, bg.nby - 1) - by0 + 1;
    if (score_parts > 0 && blockIdx.x + blockIdx.y == 0 && warp == 7) score_sum(a, ws, score_parts);
    for (int by = warp; by < bh; by += 8)
        for (int b8 = 0; b8 < bw; b8 += 8) {
            const int bx = b8 + (lane >> 2);
            const BlockCoefs c = block_coefs<4>(a, ws, bg, bx0 + min(bx, bw - 1), by0 + by);
            if ((lane & 3) == 0 && bx < bw) {
                coef[by * t.bw + bx] = make_float4(c.rA, c.mB, c.rho, c.P);
                coef2[by * t.bw + bx] = make_float2(c.D, c.K);
            }
        }
    __syncthreads();
    // pixels: a warp takes 32 columns of four rows at a time; those past the
    // windows' union do not enter S
    const int xe = min(rw, bg.nbx * G - xl), ye = min(rh, bg.nby * G - yl);
    constexpr int NR = 4;
    for (int x = lane; x < rw; x += 32)
        for (int y0 = warp; y0 < rh; y0 += 8 * NR) {
            float4 v[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int y = y0 + 8 * r;
                v[r] = x < xe && y < ye ? ws.px4[(long long)(yl + y) * a.W + xl + x] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            const int col = x < xe ? cb[x] : 0;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int y = y0 + 8 * r;
                if (y >= rh) break;
                const int k = rb[y] + col;
                const float4 c = coef[k];
                const float2 d = coef2[k];
                const float g = x < xe && y < ye ? pixel_g(v[r], BlockCoefs{c.x, c.y, c.z, c.w, d.x, d.y}) : 0.f;
                gxy[y * pitch + x] = make_float2(g * v[r].y, g * v[r].z);
            }
        }
    __syncthreads();
    // along x: lanes down the rows (odd pitch: no bank conflicts).  Inside a
    // node's support the cell of a column is the node's own or the one before.
    const int rc = (rh + 31) / 32;
    for (int task = warp; task < nn * rc; task += 8) {
        const int i = task / rc, y = (task - i * rc) * 32 + lane;
        int lo, hi;
        support(n0 + i, a.nx, c0, a.s, a.W, lo, hi);
        if (y >= rh) continue;
        float su = 0.f, sv = 0.f;
        for (int x = lo - xl; x <= hi - xl; ++x) {
            const int2 c = cw[x];
            const float2 g = gxy[y * pitch + x];
            const float f = __int_as_float(c.y), wgt = c.x == n0 + i ? 1.f - f : f;
            su = fmaf(wgt, g.x, su);
            sv = fmaf(wgt, g.y, sv);
        }
        rows[y * t.tx + i] = make_float2(su, sv);
    }
    __syncthreads();
    // along y
    for (int e = tid; e < nn * mm; e += 256) {
        const int m = e / nn, i = e - m * nn, node = m0 + m;
        int lo, hi;
        support(node, a.ny, c0, a.s, a.H, lo, hi);
        float su = 0.f, sv = 0.f;
        for (int y = lo - yl; y <= hi - yl; ++y) {
            const int2 c = rw_[y];
            const float f = __int_as_float(c.y), wgt = c.x == node ? 1.f - f : f;
            const float2 r = rows[y * t.tx + i];
            su = fmaf(wgt, r.x, su);
            sv = fmaf(wgt, r.y, sv);
        }
        const int k = node * a.nx + n0 + i;
        if (a.grad_u) a.grad_u[k] = a.grad_scale * su;
        if (a.grad_v) a.grad_v[k] = a.grad_scale * sv;
    }
}

// 3, node tiles too large for shared memory: the pixels, then the rows, then the nodes
__global__ void adj_pix_kernel(const AdjArgs a, const AdjWs ws, const BlockGrid bg)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= a.W) return;
    const long long p = (long long)y * a.W + x;
    float2 g = make_float2(0.f, 0.f);
    if (x < bg.nbx * bg.G && y < bg.nby * bg.G) {
        const float4 v = ws.px4[p];
        const float d = pixel_g(v, block_coefs<1>(a, ws, bg, x / bg.G, y / bg.G));
        g = make_float2(d * v.y, d * v.z);
    }
    ws.pix_g[p] = g;
}

// per (image row y, node column i): sum over x of the x weight times pix_g
__global__ void adj_rows_kernel(const AdjArgs a, const AdjWs ws)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (i >= a.nx) return;
    const float c0 = 0.5f * (float)(a.w - 1);
    int xl, xh;
    support(i, a.nx, c0, a.s, a.W, xl, xh);
    const float2 *row = ws.pix_g + (long long)y * a.W;
    float gu = 0.f, gv = 0.f;
    for (int x = xl; x <= xh; ++x) {
        const float wx = node_wt(x, i, a.nx, c0, a.s);
        if (wx == 0.f) continue;
        gu = fmaf(wx, row[x].x, gu);
        gv = fmaf(wx, row[x].y, gv);
    }
    ws.rows[(long long)y * a.nx + i] = make_float2(gu, gv);
}

// per node: sum over y of the y weight times the row sums
__global__ void adj_node_kernel(const AdjArgs a, const AdjWs ws)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.nx * a.ny) return;
    const int j = k / a.nx, i = k - j * a.nx;
    const float c0 = 0.5f * (float)(a.w - 1);
    int yl, yh;
    support(j, a.ny, c0, a.s, a.H, yl, yh);
    float gu = 0.f, gv = 0.f;
    for (int y = yl; y <= yh; ++y) {
        const float wy = node_wt(y, j, a.ny, c0, a.s);
        if (wy == 0.f) continue;
        const float2 r = ws.rows[(long long)y * a.nx + i];
        gu = fmaf(wy, r.x, gu);
        gv = fmaf(wy, r.y, gv);
    }
    if (a.grad_u) a.grad_u[k] = a.grad_scale * gu;
    if (a.grad_v) a.grad_v[k] = a.grad_scale * gv;
}

template <typename T>
cudaError_t run(const AdjArgs &a, cudaStream_t st)
{
    AdjWs ws;
    ws_floats(a.W, a.H, a.w, a.s, a.nx, a.ny, &ws, reinterpret_cast<float *>(a.ws));
    const BlockGrid bg = block_grid(a.w, a.s, a.nx, a.ny);
    const int nwin = a.nx * a.ny, nblk = bg.nbx * bg.nby;
    const bool grad = a.grad_u || a.grad_v;
    if (bg.G <= MAX_G && a.s >= 3) {  // the tile's node rows are sized for steps of 3
        const int tbx = std::max(1, TILE_W / bg.G), tby = std::max(1, TILE_H / bg.G);
        int lanes = 32;
        while (lanes > 1 && tbx * tby * lanes > 256) lanes >>= 1;
        const dim3 grid((bg.nbx + tbx - 1) / tbx, (bg.nby + tby - 1) / tby);
        if (grad) adj_blocks<T, true><<<grid, 256, 0, st>>>(a, ws, bg, tbx, tby, lanes);
        else adj_blocks<T, false><<<grid, 256, 0, st>>>(a, ws, bg, tbx, tby, lanes);
    } else {
        adj_deform_kernel<T><<<dim3((a.W + 255) / 256, a.H), 256, 0, st>>>(a, ws);
        if (bg.G > MAX_G) adj_block_kernel<8><<<nblk, 256, 0, st>>>(a, ws, bg);
        else adj_block_kernel<1><<<(nblk + 7) / 8, 256, 0, st>>>(a, ws, bg);
    }
    const NodeTile t = node_tile(a.W, a.H, a.w, a.s, a.nx, a.ny);
    const int wc = win_ctas(a.nx, a.ny);
    const bool sum_in_nodes = grad && t.ok;
    if (a.w / bg.G <= 4) adj_windows<true><<<wc, WIN_CTA * WIN_LANES, 0, st>>>(a, ws, bg, !sum_in_nodes);
    else adj_windows<false><<<wc, WIN_CTA * WIN_LANES, 0, st>>>(a, ws, bg, !sum_in_nodes);
    if (grad) {
        if (t.ok) {
            adj_nodes<<<dim3((a.nx + t.tx - 1) / t.tx, (a.ny + t.ty - 1) / t.ty), 256, t.smem, st>>>(a, ws, bg, t, a.score_out ? wc : 0);
        } else {
            adj_pix_kernel<<<dim3((a.W + 255) / 256, a.H), 256, 0, st>>>(a, ws, bg);
            adj_rows_kernel<<<dim3((a.nx + 127) / 128, a.H), 128, 0, st>>>(a, ws);
            adj_node_kernel<<<(nwin + 127) / 128, 128, 0, st>>>(a, ws);
        }
    }
    return cudaGetLastError();
}

}  // namespace

// ------------------------------------------------ refinement step helpers --

namespace {

// cu = u + eta gu, cv = v + eta gv (FP32, one element per thread)
__global__ void refine_axpy_kernel(const float *u, const float *v, const float *gu, const float *gv, float eta,
                                   float *cu, float *cv, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    cu[i] = fmaf(eta, gu[i], u[i]);
    cv[i] = fmaf(eta, gv[i], v[i]);
}

// out = max(|a|, |b|) over n elements: one CTA, fixed order (max is exact)
__global__ void refine_absmax_kernel(const float *a, const float *b, int n, float *out)
{
    __shared__ float part[32];
    float m = 0.f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmaxf(m, fmaxf(fabsf(a[i]), fabsf(b[i])));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (threadIdx.x == 0) *out = m;
    }
}

}  // namespace

cudaError_t launch_refine_axpy(const float *u, const float *v, const float *gu, const float *gv, float eta, float *cu,
                               float *cv, int n, cudaStream_t st)
{
    refine_axpy_kernel<<<(n + 255) / 256, 256, 0, st>>>(u, v, gu, gv, eta, cu, cv, n);
    return cudaGetLastError();
}

cudaError_t launch_refine_absmax(const float *a, const float *b, int n, float *out, cudaStream_t st)
{
    refine_absmax_kernel<<<1, 1024, 0, st>>>(a, b, n, out);
    return cudaGetLastError();
}

size_t adjoint_workspace_bytes(int W, int H, int w, int s, int nx, int ny)
{
    return sizeof(float) * ws_floats(W, H, w, s, nx, ny, nullptr, nullptr) + 256;
}

// Once per allocation of the workspace, on the stream of its first use: the
// ticket of adj_windows starts at zero.
cudaError_t init_adjoint_workspace(void *ws, cudaStream_t st) { return cudaMemsetAsync(ws, 0, 256, st); }

void prepare_adjoint()
{
    cudaFuncSetAttribute(adj_nodes, cudaFuncAttributeMaxDynamicSharedMemorySize, NODE_SMEM);
    cudaGetLastError();
}

cudaError_t launch_adjoint(const AdjArgs &a, cudaStream_t st)
{
    if (a.fmt == PIX_U8) return run<uint8_t>(a, st);
    if (a.fmt == PIX_U16) return run<uint16_t>(a, st);
    return run<float>(a, st);
}

}  // namespace rpiv
