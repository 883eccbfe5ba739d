// Per-node kernels of the vector grid and the image pyramid:
//   - universal outlier detection with median replacement (paper Sec. 2,
//     Westerweel & Scarano 2005; threshold 2 and 0.1 px regulariser, Sec. 3.1)
//   - grid-to-grid bilinear interpolation (pass-to-pass predictor, pyramid)
//   - vorticity omega = dv/dx - du/dy (paper Sec. 1-2, displayed field)
//   - 2x2 box downsampling of the image pyramid (coarse-to-fine predictor)
#include <algorithm>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "grid_interp.cuh"
#include "rpiv_internal.h"

namespace rpiv {

// ------------------------------------------------------------------ UOD --

constexpr int UOD_TILE = 16;
constexpr int UOD_IN = UOD_TILE + 4;    // values with a 2-node halo
constexpr int UOD_FLAG = UOD_TILE + 2;  // flags with a 1-node halo

__device__ __forceinline__ void cswap(float &a, float &b)
{
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    a = lo;
    b = hi;
}

// Sorts 8 values ascending (Batcher's odd-even merge network, 19 exchanges).
__device__ __forceinline__ void sort8(float (&v)[8])
{
    cswap(v[0], v[1]); cswap(v[2], v[3]); cswap(v[4], v[5]); cswap(v[6], v[7]);
    cswap(v[0], v[2]); cswap(v[1], v[3]); cswap(v[4], v[6]); cswap(v[5], v[7]);
    cswap(v[1], v[2]); cswap(v[5], v[6]);
    cswap(v[0], v[4]); cswap(v[1], v[5]); cswap(v[2], v[6]); cswap(v[3], v[7]);
    cswap(v[2], v[4]); cswap(v[3], v[5]);
    cswap(v[1], v[2]); cswap(v[3], v[4]); cswap(v[5], v[6]);
}

// Median of the first c entries (c in 1..8) of v once sorted; the rest must
// be +inf.  v is left sorted.
__device__ __forceinline__ float median_sorted(float (&v)[8], int c)
{
    sort8(v);
    if (c == 8) return 0.5f * (v[3] + v[4]);  // every neighbour present: the usual case
    float m = v[0];
#pragma unroll
    for (int q = 1; q < 8; ++q)
        if (q == c / 2) m = v[q];
    if ((c & 1) == 0) {
        float lo = v[0];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q == c / 2 - 1) lo = v[q];
        m = 0.5f * (lo + m);
    }
    return m;
}

__global__ void __launch_bounds__(256) uod_kernel(const UodArgs a)
{
    __shared__ float su[UOD_IN][UOD_IN], sv[UOD_IN][UOD_IN];
    __shared__ unsigned char sok[UOD_IN][UOD_IN];   // 1 if the node exists
    __shared__ unsigned char sbad[UOD_FLAG][UOD_FLAG];
    const int pair = blockIdx.z;
    const float *u = (const float *)resolve(a.u, pair);
    const float *v = (const float *)resolve(a.v, pair);
    const int32_t *info = (const int32_t *)resolve(a.info, pair);
    float *uo = (float *)resolve(a.u_out, pair);
    float *vo = (float *)resolve(a.v_out, pair);
    uint8_t *mask = (uint8_t *)resolve(a.mask, pair);
    const int i0 = blockIdx.x * UOD_TILE - 2, j0 = blockIdx.y * UOD_TILE - 2;
    const int tid = threadIdx.x;
    for (int e = tid; e < UOD_IN * UOD_IN; e += blockDim.x) {
        const int jj = e / UOD_IN, ii = e % UOD_IN;
        const int i = i0 + ii, j = j0 + jj;
        const bool ok = i >= 0 && j >= 0 && i < a.nx && j < a.ny;
        su[jj][ii] = ok ? u[j * a.nx + i] : 0.f;
        sv[jj][ii] = ok ? v[j * a.nx + i] : 0.f;
        sok[jj][ii] = ok ? 1 : 0;
    }
    __syncthreads();
    // detection on the tile plus a 1-node halo
    for (int e = tid; e < UOD_FLAG * UOD_FLAG; e += blockDim.x) {
        const int jj = e / UOD_FLAG + 1, ii = e % UOD_FLAG + 1;
        const int i = i0 + ii, j = j0 + jj;
        unsigned char bad = 0;
        if (sok[jj][ii]) {
            if (info && !(info[j * a.nx + i] & 1)) bad = 1;
            // the neighbours in a fixed order, +inf where a node is missing:
            // sorting puts the c present values first, in the same order as
            // any packing of them would
            float nu[8], nv[8];
            int c = 0, q = 0;
#pragma unroll
            for (int dj = -1; dj <= 1; ++dj)
#pragma unroll
                for (int di = -1; di <= 1; ++di) {
                    if (di == 0 && dj == 0) continue;
                    const bool ok = sok[jj + dj][ii + di];
                    nu[q] = ok ? su[jj + dj][ii + di] : INFINITY;
                    nv[q] = ok ? sv[jj + dj][ii + di] : INFINITY;
                    c += ok ? 1 : 0;
                    ++q;
                }
            if (c > 0) {
                // nu, nv sorted in place: the residuals of their first c entries
                const float um = median_sorted(nu, c);
                const float vm = median_sorted(nv, c);
#pragma unroll
                for (int q2 = 0; q2 < 8; ++q2) {
                    nu[q2] = q2 < c ? fabsf(nu[q2] - um) : INFINITY;
                    nv[q2] = q2 < c ? fabsf(nv[q2] - vm) : INFINITY;
                }
                const float rmu = median_sorted(nu, c);
                const float rmv = median_sorted(nv, c);
                const float r0u = fabsf(su[jj][ii] - um) / (rmu + a.eps);
                const float r0v = fabsf(sv[jj][ii] - vm) / (rmv + a.eps);
                if (r0u > a.thr || r0v > a.thr) bad = 1;
                // a non-finite value is always an outlier
                if (!isfinite(su[jj][ii]) || !isfinite(sv[jj][ii])) bad = 1;
            }
        }
        sbad[jj - 1][ii - 1] = bad;
    }
    __syncthreads();
    // replacement on the tile
    {
        const int ii = tid % UOD_TILE + 2, jj = tid / UOD_TILE + 2;
        const int i = i0 + ii, j = j0 + jj;
        if (tid < UOD_TILE * UOD_TILE && i < a.nx && j < a.ny) {
            const int k = j * a.nx + i;
            float ru = su[jj][ii], rv = sv[jj][ii];
            const bool bad = sbad[jj - 1][ii - 1];
            if (bad && a.replace) {
                float nu[8], nv[8];
                int c = 0, q = 0;
#pragma unroll
                for (int dj = -1; dj <= 1; ++dj)
#pragma unroll
                    for (int di = -1; di <= 1; ++di) {
                        if (di == 0 && dj == 0) continue;
                        const bool ok = sok[jj + dj][ii + di] && !sbad[jj + dj - 1][ii + di - 1];
                        nu[q] = ok ? su[jj + dj][ii + di] : INFINITY;
                        nv[q] = ok ? sv[jj + dj][ii + di] : INFINITY;
                        c += ok ? 1 : 0;
                        ++q;
                    }
                if (c > 0) {
                    ru = median_sorted(nu, c);
                    rv = median_sorted(nv, c);
                }
            }
            uo[k] = ru;
            vo[k] = rv;
            if (mask) mask[k] = bad ? 0 : 1;
        }
    }
}

cudaError_t launch_uod(const UodArgs &a, int n_pairs, cudaStream_t st)
{
    dim3 grid((a.nx + UOD_TILE - 1) / UOD_TILE, (a.ny + UOD_TILE - 1) / UOD_TILE, n_pairs);
    uod_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// --------------------------------------------------------------- interp --

__global__ void interp_kernel(const InterpArgs a)
{
    const int pair = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.dnx * a.dny) return;
    const float *su = (const float *)resolve(a.su, pair);
    const float *sv = (const float *)resolve(a.sv, pair);
    float *du = (float *)resolve(a.du, pair);
    float *dv = (float *)resolve(a.dv, pair);
    if (!su || !sv) {
        if (a.zero_if_null) {
            du[k] = 0.f;
            dv[k] = 0.f;
        }
        return;
    }
    const int j = k / a.dnx, i = k - j * a.dnx;
    const float2 d = interp_node(su, sv, a.snx, a.sny, a.sw, a.ss, a.dw, a.ds, a.levels_up, i, j);
    du[k] = d.x;
    dv[k] = d.y;
}

cudaError_t launch_interp(const InterpArgs &a, int n_pairs, cudaStream_t st)
{
    const int n = a.dnx * a.dny;
    dim3 grid((n + 255) / 256, n_pairs);
    interp_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------ vorticity --

__global__ void vort_kernel(const VortArgs a)
{
    const int pair = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.nx * a.ny) return;
    const float *u = (const float *)resolve(a.u, pair);
    const float *v = (const float *)resolve(a.v, pair);
    float *o = (float *)resolve(a.out, pair);
    if (!o) return;
    const int j = k / a.nx, i = k - j * a.nx;
    const int nx = a.nx, ny = a.ny;
    const float s = (float)a.s;
    float dvdx = 0.f, dudy = 0.f;
    if (nx > 1) {
        if (i == 0) dvdx = (v[j * nx + 1] - v[j * nx]) / s;
        else if (i == nx - 1) dvdx = (v[j * nx + i] - v[j * nx + i - 1]) / s;
        else dvdx = (v[j * nx + i + 1] - v[j * nx + i - 1]) / (2.f * s);
    }
    if (ny > 1) {
        if (j == 0) dudy = (u[nx + i] - u[i]) / s;
        else if (j == ny - 1) dudy = (u[j * nx + i] - u[(j - 1) * nx + i]) / s;
        else dudy = (u[(j + 1) * nx + i] - u[(j - 1) * nx + i]) / (2.f * s);
    }
    o[k] = dvdx - dudy;
}

__global__ void ema_kernel(const float *__restrict__ x, float *state, size_t n, float alpha, int init)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float xi = x[i];
        state[i] = init ? xi : alpha * xi + (1.f - alpha) * state[i];
    }
}

cudaError_t launch_ema(const float *x, float *state, size_t n, float alpha, int init, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const size_t blocks = std::min<size_t>((n + 255) / 256, (size_t)device_sm_count() * 8);
    ema_kernel<<<(unsigned)blocks, 256, 0, st>>>(x, state, n, alpha, init);
    return cudaGetLastError();
}

cudaError_t launch_vort(const VortArgs &a, int n_pairs, cudaStream_t st)
{
    const int n = a.nx * a.ny;
    dim3 grid((n + 255) / 256, n_pairs);
    vort_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// --------------------------------------------- frames and their pyramid --

// Four consecutive source pixels of a row from pixel p (a multiple of 4): one
// 4-byte (u8), 8-byte (u16) or 16-byte (float) load.
template <typename T>
__device__ __forceinline__ void load4(const unsigned char *row, int p, float (&v)[4])
{
    if (sizeof(T) == 1) {
        const uint32_t u = __ldg(reinterpret_cast<const uint32_t *>(row) + p / 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = (float)((u >> (8 * i)) & 0xffu);
    } else if (sizeof(T) == 2) {
        const uint2 u = __ldg(reinterpret_cast<const uint2 *>(row) + p / 4);
        v[0] = (float)(u.x & 0xffffu);
        v[1] = (float)(u.x >> 16);
        v[2] = (float)(u.y & 0xffffu);
        v[3] = (float)(u.y >> 16);
    } else {
        const float4 f = __ldg(reinterpret_cast<const float4 *>(row) + p / 4);
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    }
}

// The first n of N consecutive floats to d: one vector store where d is aligned
// for it and all are wanted.
template <int N>
__device__ __forceinline__ void store_run(float *d, const float (&v)[N], int n)
{
    if (N == 4 && n >= N && (reinterpret_cast<uintptr_t>(d) & 15) == 0) {
        *reinterpret_cast<float4 *>(d) = make_float4(v[0], v[1], v[N - 2], v[N - 1]);
    } else if (N == 2 && n >= N && (reinterpret_cast<uintptr_t>(d) & 7) == 0) {
        *reinterpret_cast<float2 *>(d) = make_float2(v[0], v[N - 1]);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < n) d[i] = v[i];
    }
}

// A thread takes a patch of 4 x 4 source pixels (one vector load per row where
// the rows are aligned for it): frame A's floats, 2 x 2 pixels of level 1 and
// one of level 2, so that a frame is read once for all three and a warp's
// stores are contiguous.  Each level is the 2x2 box mean of the one below,
// ((a + b) + (c + d)) / 4.  Bound by DRAM: 64 pairs of 1 MP u16, two levels,
// 705 MB in 117 us (0.88 of the measured copy rate); patches of 8 x 4 took 157
// us (half-filled sectors per store), of 4 x 8 134 us (fewer warps).  As five
// launches (frame A, levels 1 and 2 of each frame) it was 195 us, and five of
// the 23 launches of a single pair.
constexpr int FR_ROWS = 4;

template <typename T>
__global__ void __launch_bounds__(256) frames_kernel(const FramesArgs a)
{
    const int pair = blockIdx.z / a.frames, f = blockIdx.z - pair * a.frames;
    const int x0 = 4 * (blockIdx.x * 32 + (threadIdx.x & 31)), y0 = FR_ROWS * (blockIdx.y * 8 + (threadIdx.x >> 5));
    if (x0 >= a.W || y0 >= a.H) return;
    const unsigned char *src = (const unsigned char *)resolve(a.src[f], pair);
    const bool vec = x0 + 4 <= a.W && ((reinterpret_cast<uintptr_t>(src) | (uintptr_t)a.pitch) & (4 * sizeof(T) - 1)) == 0;
    float v[FR_ROWS][4];
#pragma unroll
    for (int r = 0; r < FR_ROWS; ++r) {
        const unsigned char *row = src + (long long)min(y0 + r, a.H - 1) * a.pitch;
        if (vec) {
            load4<T>(row, x0, v[r]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) v[r][k] = (float)__ldg(reinterpret_cast<const T *>(row) + min(x0 + k, a.W - 1));
        }
    }
    if (a.ingest && f == 0) {
        float *d = (float *)resolve(a.full, pair) + (long long)(y0 + a.margin) * a.full_pitch + (x0 + a.margin);
#pragma unroll
        for (int r = 0; r < FR_ROWS; ++r)
            if (y0 + r < a.H) store_run(d + r * a.full_pitch, v[r], a.W - x0);
    }
    if (a.levels < 1) return;
    const int W1 = a.W / 2, H1 = a.H / 2, x1 = x0 / 2, y1 = y0 / 2;
    float p[FR_ROWS / 2][2];
#pragma unroll
    for (int r = 0; r < FR_ROWS / 2; ++r)
#pragma unroll
        for (int i = 0; i < 2; ++i)
            p[r][i] = 0.25f * ((v[2 * r][2 * i] + v[2 * r][2 * i + 1]) + (v[2 * r + 1][2 * i] + v[2 * r + 1][2 * i + 1]));
    float *d1 = (float *)resolve(a.down[0][f], pair) + (long long)(y1 + a.margin) * a.down_pitch[0] + (x1 + a.margin);
#pragma unroll
    for (int r = 0; r < FR_ROWS / 2; ++r)
        if (y1 + r < H1) store_run(d1 + r * a.down_pitch[0], p[r], W1 - x1);
    if (a.levels < 2) return;
    const int W2 = W1 / 2, H2 = H1 / 2, x2 = x1 / 2, y2 = y1 / 2;
    float *d2 = (float *)resolve(a.down[1][f], pair) + (long long)(y2 + a.margin) * a.down_pitch[1] + (x2 + a.margin);
#pragma unroll
    for (int r = 0; r < FR_ROWS / 4; ++r)
        if (y2 + r < H2 && x2 < W2)
            d2[r * a.down_pitch[1]] = 0.25f * ((p[2 * r][0] + p[2 * r][1]) + (p[2 * r + 1][0] + p[2 * r + 1][1]));
}

cudaError_t launch_frames(const FramesArgs &a, int n_pairs, cudaStream_t st)
{
    const dim3 grid((a.W + 4 * 32 - 1) / (4 * 32), (a.H + FR_ROWS * 8 - 1) / (FR_ROWS * 8), n_pairs * a.frames);
    if (a.fmt == PIX_U8) frames_kernel<uint8_t><<<grid, 256, 0, st>>>(a);
    else if (a.fmt == PIX_U16) frames_kernel<uint16_t><<<grid, 256, 0, st>>>(a);
    else frames_kernel<float><<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// A warp copies up to 32 consecutive 16-byte words of a row of one frame of one
// pair.  Every load is an aligned 16-byte word; where a row starts off a 16-byte
// boundary, a word of the destination is the end of one and the start of the next,
// which the next lane holds (the words at a row's ends reach past it, inside the
// 16 bytes that hold its first or last pixel).
// Bound by the link to the host (33.5 MB in 163 us, 205 GB/s, as long as
// cudaMemcpyAsync takes).  Beside other parts' passes about 64 CTAs keep the link
// 93 % busy; more loads in flight only hold up the passes' own (four 2048^2
// pairs end to end: 64 CTAs 702 us, 152 714, 304 750, 32 with four loads per
// thread 717).  Alone, as the first part's is, two CTAs per SM (17 pairs of 407 x 297
// u16 and 64 CTAs for the first part too: 118 us, 110 before the parts).
constexpr int UPLOAD_CTAS = 64;

// the 16 bytes from byte sh (0..15) of lo followed by hi
__device__ __forceinline__ uint4 bytes_from(uint4 lo, uint4 hi, int sh)
{
    uint32_t a[7] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z}, last = hi.w;
    if (sh & 8) {
        a[0] = a[2], a[1] = a[3], a[2] = a[4], a[3] = a[5], a[4] = a[6], a[5] = last;
    }
    if (sh & 4) {
        a[0] = a[1], a[1] = a[2], a[2] = a[3], a[3] = a[4], a[4] = a[5];
    }
    const uint32_t bits = 8u * (sh & 3);
    return make_uint4(__funnelshift_r(a[0], a[1], bits), __funnelshift_r(a[1], a[2], bits),
                      __funnelshift_r(a[2], a[3], bits), __funnelshift_r(a[3], a[4], bits));
}

__global__ void __launch_bounds__(256) upload_kernel(const UploadArgs a)
{
    const int pair = blockIdx.z, which = blockIdx.y, lane = threadIdx.x & 31;
    const unsigned char *src = (const unsigned char *)resolve(which ? a.src_b : a.src_a, pair);
    unsigned char *dst = (unsigned char *)resolve(which ? a.dst_b : a.dst_a, pair);
    const int nw = (a.row_bytes + 15) >> 4, nc = (nw + 31) >> 5, warps = gridDim.x * 8;
    for (long long t = blockIdx.x * 8 + (threadIdx.x >> 5); t < (long long)a.H * nc; t += warps) {
        const int y = (int)(t / nc), x = 32 * (int)(t - (long long)y * nc) + lane;
        const unsigned char *row = src + (long long)y * a.pitch;
        const int sh = (int)(reinterpret_cast<uintptr_t>(row) & 15);
        const uint4 *p = reinterpret_cast<const uint4 *>(row - sh);
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (x < nw) w = p[x];
        if (sh) {  // the same for the whole warp
            uint4 n;
            n.x = __shfl_down_sync(0xffffffffu, w.x, 1);
            n.y = __shfl_down_sync(0xffffffffu, w.y, 1);
            n.z = __shfl_down_sync(0xffffffffu, w.z, 1);
            n.w = __shfl_down_sync(0xffffffffu, w.w, 1);
            // no next lane holds the following word, and this one needs bytes of it
            if (x < nw && (lane == 31 || x + 1 == nw) && sh + min(16, a.row_bytes - 16 * x) > 16) n = p[x + 1];
            w = bytes_from(w, n, sh);
        }
        if (x < nw) reinterpret_cast<uint4 *>(dst + (long long)y * a.dst_pitch)[x] = w;
    }
}

cudaError_t launch_upload(const UploadArgs &a, int n_pairs, cudaStream_t st)
{
    const int tasks = a.H * (((a.row_bytes + 15) / 16 + 31) / 32), frames = 2 * n_pairs;
    const int ctas = a.beside ? UPLOAD_CTAS : 2 * device_sm_count();
    dim3 grid(std::min((tasks + 7) / 8, std::max(1, (ctas + frames - 1) / frames)), 2, n_pairs);
    upload_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace rpiv
