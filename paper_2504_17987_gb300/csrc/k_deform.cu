// Image deformation by the predictor (paper Sec. 2: the pre-processed pair is
// warped by the current displacement estimate before the correlation).
//
//   out(x, y) = I(x + c du(x, y), y + c dv(x, y))     bilinear, clamp-to-edge
//
// where (du, dv) is the bilinear interpolation of the predictor grid at the
// pixel (border values continued outside the node hull), c = 1 for the
// frame-B-only warp and +-1/2 for the central warp of either frame.  The output
// covers the image grown by a margin M on every side, because correlation
// shifts reach M pixels outside the windows; it is written once per pixel
// and read by the correlation pass of the same grid.
#include <algorithm>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "grid_interp.cuh"
#include "rpiv_internal.h"

namespace rpiv {

namespace {

// A tile is DTX x DTY output pixels: 64 x 128 when the batch fills the GPU
// (the per-tile set-up is spread over more pixels), 64 x 64 or 64 x 32 otherwise.
constexpr int DTX = 64, DTY_MAX = 128;
constexpr int DROWS = 4;            // consecutive rows per thread and slice (256 threads = 64 columns x 4 groups)
constexpr int SLICE = 4 * DROWS;    // rows per slice
// Nodes and node rows a tile can touch, for steps >= 3 and for steps >= 8
// (checked on the host).  The shared arrays are sized by these caps: the
// smaller ones leave more of the SM's combined L1 / shared memory to the L1
// that serves the gathers.
constexpr int NODE_CAP = 1152, NODE_CAP_S8 = 256;
constexpr int nrow_cap(int dty, int min_step) { return dty / min_step + 4; }

// cell index and weight of a pixel position along one axis of the node grid
// (node i at c0 + i s; positions outside the hull take the border value)
__device__ __forceinline__ void axis_weight(int pos, int n, float c0, int s, int &i0, float &t)
{
    if (n <= 1) {
        i0 = 0;
        t = 0.f;
        return;
    }
    float f = over_step((float)pos - c0, s);
    f = fminf(fmaxf(f, 0.f), (float)(n - 1));
    int ia = (int)floorf(f);
    if (ia > n - 2) ia = n - 2;
    i0 = ia;
    t = f - (float)ia;
}

// Signed integers in the order of the floats they are made of (no NaN), and
// back: a warp's minimum or maximum is then one reduction instruction.
__device__ __forceinline__ int order_key(int bits) { return bits ^ ((bits >> 31) & 0x7fffffff); }
__device__ __forceinline__ float warp_min(float v)
{
    return __int_as_float(order_key(__reduce_min_sync(0xffffffffu, order_key(__float_as_int(v)))));
}
__device__ __forceinline__ float warp_max(float v)
{
    return __int_as_float(order_key(__reduce_max_sync(0xffffffffu, order_key(__float_as_int(v)))));
}

// A pixel as a float plus the format's bias: integers below 2^23 are placed in
// the mantissa under the exponent of 2^23 (one logic instruction instead of a
// conversion), so the bias is 2^23.  Differences of biased pixels are exact.
__device__ __forceinline__ float biased(uint8_t v) { return __uint_as_float(0x4B000000u | (uint32_t)v); }
__device__ __forceinline__ float biased(uint16_t v) { return __uint_as_float(0x4B000000u | (uint32_t)v); }
__device__ __forceinline__ float biased(float v) { return v; }

// floor(d) + 1.5 * 2^23 (|d| < 2^22): the add rounds down at a unit in the last
// place of one.  The integer is the bits minus FLOOR_BITS.
constexpr uint32_t FLOOR_BITS = 0x4B400000u;
constexpr float FLOOR_BIAS = 12582912.f;

// First tap of pixel (x, y) whose floors, plus FLOOR_BITS, are fx and fy.  32-bit
// offsets are formed modulo 2^32, so that the constants of the row fold into one.
template <typename T>
__device__ __forceinline__ const T *tap(const T *base, uint32_t pe, int x, int y, uint32_t fx, uint32_t fy)
{
    const uint32_t row = (uint32_t)y * pe + (uint32_t)x - FLOOR_BITS * (pe + 1u);
    return base + (uint32_t)(fy * pe + fx + row);
}
template <typename T>
__device__ __forceinline__ const T *tap(const T *base, long long pe, int x, int y, uint32_t fx, uint32_t fy)
{
    return base + ((long long)(y + (int)(fy - FLOOR_BITS)) * pe + (x + (int)(fx - FLOOR_BITS)));
}

// The tile in slices of SLICE rows; a thread takes four consecutive rows of a
// slice, unrolled so that their gathers are in flight together; rows and
// columns past the grown image are computed on clamped coordinates and not
// stored.  The kernel is bound by instruction issue (73 % active at six CTAs
// per SM) and the latency of its gathers, so
//   - the rows of a node cell (the same for the whole warp) share its nodes;
//   - taps keep the bias of their format until the blend;
//   - when every lane's four rows have the same integer displacement (a smooth
//     field between its integer steps), their taps are five consecutive source
//     rows: ten loads instead of sixteen.
// 64 pairs of 1 MP, 16 px windows: 193 -> 170 us (0.32 -> 0.36 of the HBM rate); 181
// (0.34) since the launch also interpolates its predictor.
// CLAMP: the taps are clamped to the image (tiles near its border or with a
// displacement range reaching outside); otherwise the taps are read from one
// base pointer.  Off: the integer type of pixel offsets.
template <int DTY, typename T, typename Off, bool CLAMP>
__device__ __forceinline__ void deform_rows(const DeformArgs &a, const T *base, float *out, int djo, Off pe, int x,
                                            int y0, int lx, int ly0, const float2 *cuv, const int2 *rinfo)
{
    // warps whose 32 columns, and slices whose rows, lie past the grown
    // image store nothing: skip them (uniform per warp)
    if (x - (int)(threadIdx.x & 31) >= a.W + a.M) return;
    const float bias = sizeof(T) < 4 ? 8388608.f : 0.f;
    for (int r0 = DROWS * ly0; r0 < DTY; r0 += SLICE) {
        if (y0 + r0 >= a.H + a.M) break;
        const int4 ra = reinterpret_cast<const int4 *>(rinfo + r0)[0], rb = reinterpret_cast<const int4 *>(rinfo + r0)[1];
        const int off[DROWS] = {ra.x, ra.z, rb.x, rb.z};
        const int wgt[DROWS] = {ra.y, ra.w, rb.y, rb.w};
        float res[DROWS];
        float u0 = 0.f, v0 = 0.f, ud = 0.f, vd = 0.f;
        float tx[DROWS], ty[DROWS];
        uint32_t bx[DROWS], by[DROWS];  // floors plus FLOOR_BITS
#pragma unroll
        for (int k = 0; k < DROWS; ++k) {
            if (k == 0 || off[k] != off[k - 1]) {
                const float2 n0 = cuv[off[k] + lx], n1 = cuv[off[k] + djo + lx];
                u0 = n0.x;
                v0 = n0.y;
                ud = n1.x - n0.x;
                vd = n1.y - n0.y;
            }
            const float wy = __int_as_float(wgt[k]);
            float du = fmaf(wy, ud, u0), dv = fmaf(wy, vd, v0);
            if (CLAMP) {
                // NaN or absurd predictor values are clamped so the index math cannot overflow
                du = fminf(fmaxf(du, -1048576.f), 1048576.f);
                dv = fminf(fmaxf(dv, -1048576.f), 1048576.f);
            }
            const float gx = __fadd_rd(du, FLOOR_BIAS), gy = __fadd_rd(dv, FLOOR_BIAS);
            bx[k] = __float_as_uint(gx);
            by[k] = __float_as_uint(gy);
            tx[k] = du - (gx - FLOOR_BIAS);
            ty[k] = dv - (gy - FLOOR_BIAS);
        }
        // a pixel from its two tap rows: left taps (biased) and steps to the right ones
        auto blend = [&](int k, float l0, float s0, float l1, float s1) {
            const float top = (l0 - bias) + tx[k] * s0, bot = (l1 - bias) + tx[k] * s1;
            return top + ty[k] * (bot - top);
        };
        const uint32_t differ = (bx[0] ^ bx[1]) | (bx[0] ^ bx[2]) | (bx[0] ^ bx[3]) | (by[0] ^ by[1]) |
                                (by[0] ^ by[2]) | (by[0] ^ by[3]);
        if (!CLAMP && __all_sync(0xffffffffu, differ == 0u)) {
            const T *q = tap(base, pe, x, y0 + r0, bx[0], by[0]);
            float l[DROWS + 1], s[DROWS + 1];
#pragma unroll
            for (int k = 0; k <= DROWS; ++k) {
                l[k] = biased(__ldg(q + k * pe));
                s[k] = biased(__ldg(q + k * pe + 1)) - l[k];
            }
#pragma unroll
            for (int k = 0; k < DROWS; ++k) res[k] = blend(k, l[k], s[k], l[k + 1], s[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < DROWS; ++k) {
                const int y = y0 + r0 + k;
                float f00, f10, f01, f11;
                if (CLAMP) {
                    const int xl = x + (int)(bx[k] - FLOOR_BITS), yl = y + (int)(by[k] - FLOOR_BITS);
                    const int xa = min(max(xl, 0), a.W - 1), xb = min(max(xl + 1, 0), a.W - 1);
                    const int ya = min(max(yl, 0), a.H - 1), yb = min(max(yl + 1, 0), a.H - 1);
                    const T *ra = base + (Off)ya * pe, *rb = base + (Off)yb * pe;
                    f00 = biased(__ldg(ra + xa));
                    f10 = biased(__ldg(ra + xb));
                    f01 = biased(__ldg(rb + xa));
                    f11 = biased(__ldg(rb + xb));
                } else {
                    const T *q = tap(base, pe, x, y, bx[k], by[k]);
                    f00 = biased(__ldg(q));
                    f10 = biased(__ldg(q + 1));
                    f01 = biased(__ldg(q + pe));
                    f11 = biased(__ldg(q + pe + 1));
                }
                res[k] = blend(k, f00, f10 - f00, f01, f11 - f01);
            }
        }
        if (x < a.W + a.M) {
            float *o = out + (long long)(y0 + r0 + a.M) * a.out_pitch + (x + a.M);
#pragma unroll
            for (int k = 0; k < DROWS; ++k)
                if (y0 + r0 + k < a.H + a.M) o[(long long)k * a.out_pitch] = res[k];
        }
    }
}

template <int DTY, typename T, typename Off>
__device__ __forceinline__ void deform_rows_any(const DeformArgs &a, const T *base, float *out, bool inside, int djo,
                                                Off pe, int x, int y0, int lx, int ly0, const float2 *cuv,
                                                const int2 *rinfo)
{
    if (inside)
        deform_rows<DTY, T, Off, false>(a, base, out, djo, pe, x, y0, lx, ly0, cuv, rinfo);
    else
        deform_rows<DTY, T, Off, true>(a, base, out, djo, pe, x, y0, lx, ly0, cuv, rinfo);
}

// The field is bilinear in the nodes: the tile first interpolates every node
// row it touches along x at each of its columns, already scaled (cuv), and
// stores per row its node-row offset and weight (rinfo), so that a pixel needs
// one interpolation along y.  With a source field (n_src) the tile interpolates
// its nodes from it, and stores them for the pass (as a launch of its own the
// interpolation of a single pair took as long as a small pass).  A tile whose taps provably stay inside the image
// (its displacement lies within the range of its nodes, a convex combination)
// skips the clamping; either way every tap is the clamp-to-edge sample.
template <typename T, int DTY, int MIN_STEP>
__device__ void deform_tile(const DeformArgs &a, const unsigned char *img, float *pu, float *pv, float *out,
                            int pair)
{
    constexpr int NCAP = MIN_STEP >= 8 ? NODE_CAP_S8 : NODE_CAP;
    __shared__ float nu[NCAP], nv[NCAP];
    __shared__ float2 cuv[nrow_cap(DTY, MIN_STEP) * DTX];
    __shared__ __align__(16) int2 rinfo[DTY];
    __shared__ float red[4][8];
    const int x0 = blockIdx.x * DTX - a.M, y0 = blockIdx.y * DTY - a.M;
    const float c0 = 0.5f * (float)(a.w - 1);
    const bool has = pu != nullptr && pv != nullptr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lx = threadIdx.x % DTX, ly0 = threadIdx.x / DTX;
    const int x = x0 + lx;
    float umin = 0.f, umax = 0.f, vmin = 0.f, vmax = 0.f;
    bool any_nan = false;
    int djo = 0;
    if (has) {
        int ilo, ihi, jlo, jhi;
        float t;
        // the cells of the tile's corners, one per lane
        const int corner = lane & 3;
        axis_weight(corner < 2 ? x0 + (corner & 1) * (DTX - 1) : y0 + (corner & 1) * (DTY - 1), corner < 2 ? a.nx : a.ny,
                    c0, a.s, ilo, t);
        jhi = __shfl_sync(0xffffffffu, ilo, 3);
        jlo = __shfl_sync(0xffffffffu, ilo, 2);
        ihi = __shfl_sync(0xffffffffu, ilo, 1);
        ilo = __shfl_sync(0xffffffffu, ilo, 0);
        ihi = min(ihi + 1, a.nx - 1);
        jhi = min(jhi + 1, a.ny - 1);
        const int nwn = ihi - ilo + 1, nhn = jhi - jlo + 1;
        float lu0 = INFINITY, lu1 = -INFINITY, lv0 = INFINITY, lv1 = -INFINITY;
        bool nan_seen = false;
        const FieldSrc &fs = a.src[a.n_src > 1 && resolve(a.src[1].u, pair) && resolve(a.src[1].v, pair) ? 1 : 0];
        const float *su = nullptr, *sv = nullptr;
        if (a.n_src > 0) {
            su = (const float *)resolve(fs.u, pair);
            sv = (const float *)resolve(fs.v, pair);
            if (!sv) su = nullptr;
        }
        for (int e = threadIdx.x; e < nwn * nhn; e += blockDim.x) {
            const int jj = e / nwn, ii = e - jj * nwn;
            const int node = (jlo + jj) * a.nx + ilo + ii;
            float fu, fv;
            if (a.n_src > 0) {
                // the tiles that share a node write the same value
                const float2 d = su ? interp_node(su, sv, fs.nx, fs.ny, fs.w, fs.s, a.w, a.s, fs.levels_up, ilo + ii, jlo + jj)
                                    : make_float2(0.f, 0.f);
                pu[node] = fu = d.x;
                pv[node] = fv = d.y;
            } else {
                fu = pu[node];
                fv = pv[node];
            }
            nu[e] = fu;
            nv[e] = fv;
            nan_seen |= (fu != fu) || (fv != fv);
            lu0 = fminf(lu0, fu);
            lu1 = fmaxf(lu1, fu);
            lv0 = fminf(lv0, fv);
            lv1 = fmaxf(lv1, fv);
        }
        lu0 = warp_min(lu0);
        lu1 = warp_max(lu1);
        lv0 = warp_min(lv0);
        lv1 = warp_max(lv1);
        if (lane == 0) {
            red[0][warp] = lu0;
            red[1][warp] = lu1;
            red[2][warp] = lv0;
            red[3][warp] = lv1;
        }
        for (int e = threadIdx.x; e < DTY; e += blockDim.x) {
            int j0;
            axis_weight(y0 + e, a.ny, c0, a.s, j0, t);
            rinfo[e] = make_int2((j0 - jlo) * DTX, __float_as_int(t));
        }
        any_nan = __syncthreads_or(nan_seen);
        // node rows interpolated along x at this thread's column, scaled
        {
            int i0;
            float tx;
            axis_weight(x, a.nx, c0, a.s, i0, tx);
            const int ci = i0 - ilo, di = a.nx > 1 ? 1 : 0;
            for (int jj = ly0; jj < nhn; jj += blockDim.x / DTX) {
                const float *ru = nu + jj * nwn + ci, *rv = nv + jj * nwn + ci;
                cuv[jj * DTX + lx] = make_float2(a.scale * (ru[0] + tx * (ru[di] - ru[0])),
                                                 a.scale * (rv[0] + tx * (rv[di] - rv[0])));
            }
        }
        umin = red[0][0];
        umax = red[1][0];
        vmin = red[2][0];
        vmax = red[3][0];
        for (int k = 1; k < 8; ++k) {
            umin = fminf(umin, red[0][k]);
            umax = fmaxf(umax, red[1][k]);
            vmin = fminf(vmin, red[2][k]);
            vmax = fmaxf(vmax, red[3][k]);
        }
        // the central warp scales by -1/2 for frame A: the range flips
        const float su0 = a.scale * umin, su1 = a.scale * umax, sv0 = a.scale * vmin, sv1 = a.scale * vmax;
        umin = fminf(su0, su1);
        umax = fmaxf(su0, su1);
        vmin = fminf(sv0, sv1);
        vmax = fmaxf(sv0, sv1);
        djo = a.ny > 1 ? DTX : 0;
        __syncthreads();
    } else {
        // no predictor: one zero node row, weight 0 on every row
        if (threadIdx.x < DTX) cuv[threadIdx.x] = make_float2(0.f, 0.f);
        if (threadIdx.x < DTY) rinfo[threadIdx.x] = make_int2(0, 0);
        __syncthreads();
    }
    // every tap of the tile inside the image, with a pixel to spare against rounding
    const bool inside = !any_nan && umin > -1048576.f && umax < 1048576.f && vmin > -1048576.f &&
                        vmax < 1048576.f && x0 + floorf(umin) - 1.f >= 0.f &&
                        x0 + DTX - 1 + floorf(umax) + 2.f <= (float)(a.W - 1) && y0 + floorf(vmin) - 1.f >= 0.f &&
                        y0 + DTY - 1 + floorf(vmax) + 2.f <= (float)(a.H - 1);
    const T *base = reinterpret_cast<const T *>(img);
    const long long pe = a.pitch / (long long)sizeof(T);  // row pitch in pixels (a multiple of the pixel size)
    // 32-bit pixel offsets when the whole image fits them
    if ((long long)a.H * pe < (1LL << 31))
        deform_rows_any<DTY, T, uint32_t>(a, base, out, inside, djo, (uint32_t)pe, x, y0, lx, ly0, cuv, rinfo);
    else
        deform_rows_any<DTY, T, long long>(a, base, out, inside, djo, pe, x, y0, lx, ly0, cuv, rinfo);
}

// one kernel per pixel type, so that each holds a single copy of the tile's
// shared arrays; MIN_STEP: the smallest node step its caps allow (3 or 8).
// Six CTAs per SM (40 registers; eight, at 32, spill and are no faster, five are
// slower).
template <typename T, int DTY, int MIN_STEP>
__global__ void __launch_bounds__(256, 6) deform_kernel(const DeformArgs a)
{
    const int pair = blockIdx.z;
    const unsigned char *img = (const unsigned char *)resolve(a.img, pair);
    float *pu = (float *)resolve(a.pred_u, pair);
    float *pv = (float *)resolve(a.pred_v, pair);
    float *out = (float *)resolve(a.out, pair);
    deform_tile<T, DTY, MIN_STEP>(a, img, pu, pv, out, pair);
}

// nodes touched by a DTX x dty tile along each axis, plus the neighbour node,
// within the caps of the kernel for steps >= min_step
bool nodes_fit(int s, int nx, int ny, int dty, int min_step)
{
    const int cx = DTX / s + 3, cy = dty / s + 3;
    const int cap = min_step >= 8 ? NODE_CAP_S8 : NODE_CAP;
    return std::min(cx, nx) * std::min(cy, ny) <= cap && std::min(cy, ny) <= nrow_cap(dty, min_step);
}

}  // namespace

bool deform_nodes_fit(int w, int s, int nx, int ny)
{
    (void)w;
    return nodes_fit(s, nx, ny, DTY_MAX, 3);
}

template <int DTY, int MIN_STEP>
static void launch_tiles_caps(const DeformArgs &a, int n_pairs, cudaStream_t st)
{
    const int WE = a.W + 2 * a.M, HE = a.H + 2 * a.M;
    dim3 grid((WE + DTX - 1) / DTX, (HE + DTY - 1) / DTY, n_pairs);
    if (a.fmt == PIX_U8) deform_kernel<uint8_t, DTY, MIN_STEP><<<grid, 256, 0, st>>>(a);
    else if (a.fmt == PIX_U16) deform_kernel<uint16_t, DTY, MIN_STEP><<<grid, 256, 0, st>>>(a);
    else deform_kernel<float, DTY, MIN_STEP><<<grid, 256, 0, st>>>(a);
}

// the small-cap kernel whenever the grid fits its caps (no predictor: one
// zero node row)
template <int DTY>
static void launch_tiles(const DeformArgs &a, int n_pairs, cudaStream_t st)
{
    const bool has = a.pred_u.base != nullptr && a.pred_v.base != nullptr;
    if (!has || nodes_fit(a.s, a.nx, a.ny, DTY, 8)) launch_tiles_caps<DTY, 8>(a, n_pairs, st);
    else launch_tiles_caps<DTY, 3>(a, n_pairs, st);
}

// 64 x 128 tiles when there are ten of them per SM, a wave and two thirds at the
// kernel's six CTAs per SM (the line was drawn at two waves of five: 0.235 ->
// 0.215 ms per 64-pair 1 MP launch); smaller launches take the tallest tile that
// still gives four CTAs per SM, at least 64 x 32
cudaError_t launch_deform(const DeformArgs &a, int n_pairs, cudaStream_t st)
{
    const long long WE = a.W + 2LL * a.M, HE = a.H + 2LL * a.M;
    auto tiles = [&](int dty) { return ((WE + DTX - 1) / DTX) * ((HE + dty - 1) / dty) * n_pairs; };
    if (tiles(DTY_MAX) >= 2LL * device_sm_count() * 5) launch_tiles<DTY_MAX>(a, n_pairs, st);
    else if (tiles(64) >= 4LL * device_sm_count()) launch_tiles<64>(a, n_pairs, st);
    else launch_tiles<32>(a, n_pairs, st);
    return cudaGetLastError();
}

}  // namespace rpiv
