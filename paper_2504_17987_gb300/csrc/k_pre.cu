// Pre-processing before the flow estimate (paper Sec. 2): a high-pass filter
// against the static background, then contrast-limited adaptive histogram
// equalisation (CLAHE).
//
//   high-pass  d = max(0, n I - S), S the clamp-to-edge sum of I over the
//              (2 hp + 1)^2 box around the pixel, n its pixel count (hp = 0:
//              d = I, n = 1); the filtered value is d / n
//   CLAHE      256 bins over [0, vmax + 1), bin = floor(d 256 / (n (vmax + 1)));
//              per tile of N pixels the histogram is clipped at
//              L = max(1, floor(clip% N / (100 * 256))), the excess E spread as
//              E / 256 to every bin and one more to the first E mod 256 bins;
//              map[b] = cdf[b] vmax / N; a pixel blends the maps of the four
//              tiles whose centres surround it, bilinearly
//
// Box sums, bins and cumulative counts are integers, so every bin is exact,
// in whatever order they are formed.
//
// Three launches: high-pass, bins and partial histograms (pre_bins); the maps
// (clahe_maps); the blend (clahe_apply).  A 1 MP frame moves 2 to 8 MB, so the
// launches are bound by latency, not bandwidth, and the work is split to fill
// the chip: a histogram tile is cut into chunks of about 16 rows, one CTA each
// (512 CTAs for 8 x 8 tiles of a 1 MP frame, where one CTA per tile left 88 of
// 152 SMs idle).
#include <algorithm>
#include <cuda_runtime.h>
#include <stdint.h>

#include "rpiv_internal.h"

namespace rpiv {

namespace {

constexpr int NBINS = 256;
constexpr int PRE_THREADS = 256;
constexpr int BATCH = 8;        // rows of vertical sums staged at a time
constexpr int STRIP = 256;      // columns staged at a time
constexpr int CHUNK = 512;      // widest chunk
constexpr int FILTER_COLS = 128;  // widest chunk without equalisation
constexpr int COPIES = 16;      // copies of a chunk's histogram
constexpr int MAX_HP = 64;      // largest box radius
constexpr int RUN = 4;          // consecutive pixels per thread: the horizontal sum slides along them

template <typename T>
__device__ __forceinline__ int px(const unsigned char *img, long long pitch, int x, int y)
{
    return (int)__ldg(reinterpret_cast<const T *>(img + (long long)y * pitch) + x);
}

// Chunks: every tile of the histogram grid (without equalisation: the frame) is cut
// into ncx x ncy chunks of cw x ch pixels (the last ones smaller, possibly empty).
struct PreSplit {
    int tw, th, ncx, ncy, cw, ch;
    long long bin_pitch;  // bytes between rows of the bins, a multiple of 4
};

// One chunk per CTA: d = max(0, n I - S) (hp = 0: d = I) with the box sum S
// from vertical running sums, one column per thread, staged BATCH rows at a
// time, and a horizontal sum that slides along the thread's RUN pixels.  With
// equalisation: the bin of d (one byte per pixel instead of d itself) and the
// chunk's histogram; without: the filtered value d / n.
//
// bin = floor(256 d / den), den = n (vmax + 1), without a division: d is in
// bin b or above exactly when d >= ceil(b den / 256), so a single-precision
// estimate (off by at most one: two roundings of a value below 256) is
// corrected against its two thresholds (at most den <= 129^2 2^16 < 2^31).
//
// Two lanes of a warp share a copy of the histogram, the copies in different
// banks: equal bins, the usual case on a dark background, collide in pairs
// instead of all at once.
template <typename T, bool EQUALISE>
__global__ void __launch_bounds__(PRE_THREADS) pre_bins(const PreArgs a, const PreSplit q, uint8_t *bins, int *parts)
{
    __shared__ int vs[2][BATCH][STRIP + 2 * MAX_HP];
    __shared__ int thr[NBINS + 1];
    __shared__ int hist[EQUALISE ? NBINS * COPIES : 1];
    const int tid = threadIdx.x, lane = tid & 31;
    const int ti = blockIdx.x / q.ncx, cx = blockIdx.x - ti * q.ncx;
    const int tj = blockIdx.y / q.ncy, cy = blockIdx.y - tj * q.ncy;
    const int X0 = ti * q.tw + cx * q.cw, X1 = min(min(a.W, (ti + 1) * q.tw), X0 + q.cw);
    const int Y0 = tj * q.th + cy * q.ch, Y1 = min(min(a.H, (tj + 1) * q.th), Y0 + q.ch);
    const unsigned char *img = static_cast<const unsigned char *>(a.img);
    const int hp = a.hp, n = a.n;
    const long long den = (long long)n * (a.vmax + 1);
    const float scale = 256.f / (float)den;
    if (EQUALISE) {
        for (int b = tid; b <= NBINS; b += PRE_THREADS) thr[b] = (int)((b * den + 255) / 256);
        for (int e = tid; e < NBINS * COPIES; e += PRE_THREADS) hist[e] = 0;
    }
    int buf = 0;
    for (int xs = X0; xs < X1; xs += STRIP) {
        const int w = min(STRIP, X1 - xs), cols = w + 2 * hp;
        // running vertical sums of this thread's columns (at most two)
        constexpr int NC = (STRIP + 2 * MAX_HP + PRE_THREADS - 1) / PRE_THREADS;
        int run[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            run[k] = 0;
            const int c = tid + k * PRE_THREADS;
            if (hp > 0 && c < cols && Y0 < Y1) {
                const int x = min(max(xs - hp + c, 0), a.W - 1);
                for (int dy = -hp; dy <= hp; ++dy) run[k] += px<T>(img, a.pitch, x, min(max(Y0 + dy, 0), a.H - 1));
            }
        }
        for (int yb = Y0; yb < Y1; yb += BATCH) {
            if (hp > 0) {
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    const int c = tid + k * PRE_THREADS;
                    if (c < cols) {
                        const int x = min(max(xs - hp + c, 0), a.W - 1);
                        int in[BATCH], out[BATCH];
#pragma unroll
                        for (int r = 0; r < BATCH; ++r) {
                            in[r] = px<T>(img, a.pitch, x, min(yb + r + hp + 1, a.H - 1));
                            out[r] = px<T>(img, a.pitch, x, min(max(yb + r - hp, 0), a.H - 1));
                        }
#pragma unroll
                        for (int r = 0; r < BATCH; ++r) {
                            vs[buf][r][c] = run[k];
                            run[k] += in[r] - out[r];
                        }
                    }
                }
            }
            __syncthreads();  // also orders the thresholds and the zeroed histogram
            const int nseg = (w + RUN - 1) / RUN, rows = min(BATCH, Y1 - yb);
            for (int it = tid; it < nseg * rows; it += PRE_THREADS) {
                const int r = it / nseg, c0 = (it - r * nseg) * RUN, y = yb + r;
                const int cnt = min(RUN, w - c0);
                const int *v = vs[buf][r] + c0;
                int S = 0;
                if (hp > 0)
                    for (int k = 0; k <= 2 * hp; ++k) S += v[k];
                uint32_t packed = 0;
#pragma unroll
                for (int k = 0; k < RUN; ++k) {
                    if (k < cnt) {
                        const int I = px<T>(img, a.pitch, xs + c0 + k, y);
                        const int d = hp > 0 ? max(n * I - S, 0) : I;
                        if (EQUALISE) {
                            int b = min((int)((float)d * scale), NBINS - 1);
                            if (d < thr[b]) --b;
                            else if (b < NBINS - 1 && d >= thr[b + 1]) ++b;
                            packed |= (uint32_t)b << (8 * k);
                            atomicAdd(&hist[b * COPIES + (lane & (COPIES - 1))], 1);
                        } else {
                            a.out[(long long)y * a.out_pitch + xs + c0 + k] = (float)d / (float)n;
                        }
                        if (hp > 0 && k + 1 < cnt) S += v[2 * hp + 1 + k] - v[k];
                    }
                }
                if (EQUALISE) {
                    uint8_t *o = bins + (long long)y * q.bin_pitch + xs + c0;
                    if (cnt == RUN && ((xs + c0) & 3) == 0)
                        *reinterpret_cast<uint32_t *>(o) = packed;
                    else
                        for (int k = 0; k < cnt; ++k) o[k] = (uint8_t)(packed >> (8 * k));
                }
            }
            buf ^= 1;  // the next batch's sums go to the other buffer: one barrier per batch
        }
        __syncthreads();
    }
    if (EQUALISE) {
        __syncthreads();
        int c = 0;
        for (int k = 0; k < COPIES; ++k) c += hist[tid * COPIES + ((tid + k) & (COPIES - 1))];
        const long long chunk = ((long long)(tj * a.tx + ti) * q.ncy + cy) * q.ncx + cx;
        parts[chunk * NBINS + tid] = c;
    }
}

// One CTA of 256 threads per tile: the chunks' counts summed, clipped, the
// excess spread, the exact integer scan (warp scans, then the warps' totals);
// each bin's map value is then formed on its own.  parts may be the maps' own
// memory when a tile is one chunk (each thread reads its bin before it writes it).
__global__ void __launch_bounds__(NBINS) clahe_maps(const PreArgs a, const PreSplit q, const int *parts, float *maps)
{
    __shared__ int excess;
    __shared__ int wtot[NBINS / 32];
    const int ti = blockIdx.x, tj = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    const int x0 = ti * q.tw, x1 = min(a.W, x0 + q.tw), y0 = tj * q.th, y1 = min(a.H, y0 + q.th);
    const int N = max(x1 - x0, 0) * max(y1 - y0, 0), sub = q.ncx * q.ncy;
    const long long tile = (long long)tj * a.tx + ti;
    if (tid == 0) excess = 0;
    int h = 0;
    for (int k = 0; k < sub; ++k) h += parts[(tile * sub + k) * NBINS + tid];
    __syncthreads();
    int L = (int)((long long)a.clip_pct * N / (100LL * NBINS));
    if (L < 1) L = 1;
    const int over = h > L ? h - L : 0;
    if (over) atomicAdd(&excess, over);
    __syncthreads();
    const int E = excess;
    int c = min(h, L) + E / NBINS + (tid < E % NBINS ? 1 : 0);
    // inclusive scan within the warp, then the totals of the warps before
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) c += t;
    }
    if (lane == 31) wtot[tid >> 5] = c;
    __syncthreads();
    for (int k = 0; k < (tid >> 5); ++k) c += wtot[k];
    maps[tile * NBINS + tid] = N > 0 ? (float)((double)c * a.vmax / (double)N) : 0.f;
}

// tile pair and weight along one axis: centres at t * ts + (width_t - 1) / 2,
// clamped to the outer centres
__device__ __forceinline__ void tile_pair(int p, int ext, int ts, int nt, int &t0, int &t1, float &w)
{
    const float c0 = 0.5f * (float)(ts - 1);
    const int tl = nt - 1;
    const float cl = (float)(tl * ts) + 0.5f * (float)(ext - tl * ts - 1);
    if (nt == 1 || (float)p <= c0) {
        t0 = t1 = 0;
        w = 0.f;
    } else if ((float)p >= cl) {
        t0 = t1 = tl;
        w = 0.f;
    } else {
        int t = (int)floorf(((float)p - c0) / (float)ts);
        if (t > nt - 2) t = nt - 2;
        t0 = t;
        t1 = t + 1;
        const float a0 = (float)(t0 * ts) + 0.5f * (float)(ts - 1);
        const float a1 = (t1 == tl) ? cl : (float)(t1 * ts) + 0.5f * (float)(ts - 1);
        w = ((float)p - a0) / (a1 - a0);
    }
}

// Four pixels per thread (one word of bins, one 16-byte store where the output
// row is aligned for it); the row's blend is shared by the four.
__global__ void __launch_bounds__(PRE_THREADS) clahe_apply(const PreArgs a, const PreSplit q, const uint8_t *bins, const float *maps)
{
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x), y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= a.W || y >= a.H) return;
    const uint32_t packed = *reinterpret_cast<const uint32_t *>(bins + (long long)y * q.bin_pitch + x);
    int j0, j1;
    float wy;
    tile_pair(y, a.H, q.th, a.ty, j0, j1, wy);
    const float *r0 = maps + (long long)j0 * a.tx * NBINS, *r1 = maps + (long long)j1 * a.tx * NBINS;
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int i0, i1;
        float wx;
        tile_pair(min(x + k, a.W - 1), a.W, q.tw, a.tx, i0, i1, wx);
        const int b = (packed >> (8 * k)) & 0xff;
        const float m00 = r0[i0 * NBINS + b], m01 = r0[i1 * NBINS + b];
        const float m10 = r1[i0 * NBINS + b], m11 = r1[i1 * NBINS + b];
        v[k] = (1.f - wy) * ((1.f - wx) * m00 + wx * m01) + wy * ((1.f - wx) * m10 + wx * m11);
    }
    float *o = a.out + (long long)y * a.out_pitch + x;
    if (x + 4 <= a.W && (reinterpret_cast<uintptr_t>(o) & 15) == 0)
        *reinterpret_cast<float4 *>(o) = make_float4(v[0], v[1], v[2], v[3]);
    else
        for (int k = 0; k < 4 && x + k < a.W; ++k) o[k] = v[k];
}

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

// With equalisation: chunks of about 16 rows and at most CHUNK columns, none below 512 pixels
// unless it is a whole tile: the partial histograms (1 KB each) then fit the
// first scratch frame (4 bytes per pixel); if rounding up the tiles of an odd
// size says otherwise, one chunk per tile, whose counts sit where its map goes.
// Without: the tiles mean nothing, and the frame is cut into chunks of at most
// FILTER_COLS columns and 16 rows (391 x 277 u8, radius 64: cut by 64 x 64 tiles
// it took 41 us, by one tile 38, now 14: the host).
PreSplit split_tiles(const PreArgs &a)
{
    PreSplit q;
    q.bin_pitch = (a.W + 3) / 4 * 4;
    if (a.clip_pct <= 0) {
        q.tw = a.W;
        q.th = a.H;
        q.ncx = (a.W + FILTER_COLS - 1) / FILTER_COLS;
        q.cw = (a.W + q.ncx - 1) / q.ncx;
        q.ch = 16;
        q.ncy = (a.H + q.ch - 1) / q.ch;
        return q;
    }
    q.tw = (a.W + a.tx - 1) / a.tx;
    q.th = (a.H + a.ty - 1) / a.ty;
    q.ncx = (q.tw + CHUNK - 1) / CHUNK;
    q.cw = (q.tw + q.ncx - 1) / q.ncx;
    const int rows = std::max(16, (CHUNK + q.cw - 1) / q.cw);
    q.ncy = std::max(1, q.th / rows);
    if ((size_t)a.tx * a.ty * q.ncx * q.ncy * NBINS * 4 > up256((size_t)a.W * a.H * 4)) {
        q.ncx = q.ncy = 1;
        q.cw = q.tw;
    }
    q.ch = (q.th + q.ncy - 1) / q.ncy;
    return q;
}

template <typename T>
void launch_bins(const PreArgs &a, const PreSplit &q, uint8_t *bins, int *parts, cudaStream_t st)
{
    if (a.clip_pct > 0) pre_bins<T, true><<<dim3(a.tx * q.ncx, a.ty * q.ncy), PRE_THREADS, 0, st>>>(a, q, bins, parts);
    else pre_bins<T, false><<<dim3(q.ncx, q.ncy), PRE_THREADS, 0, st>>>(a, q, bins, parts);
}

}  // namespace

// two float frames and the maps: the partial histograms, the bins (a byte per
// pixel) and the maps sit in them
size_t preprocess_scratch_bytes(int W, int H, int tx, int ty)
{
    return 2 * up256((size_t)W * H * 4) + up256((size_t)tx * ty * NBINS * 4);
}

cudaError_t launch_preprocess(const PreArgs &a, void *scratch, cudaStream_t st)
{
    char *s = static_cast<char *>(scratch);
    const size_t frame = up256((size_t)a.W * a.H * 4);
    const PreSplit q = split_tiles(a);
    float *maps = reinterpret_cast<float *>(s + 2 * frame);
    int *parts = q.ncx * q.ncy > 1 ? reinterpret_cast<int *>(s) : reinterpret_cast<int *>(maps);
    uint8_t *bins = reinterpret_cast<uint8_t *>(s + frame);
    if (a.fmt == PIX_U8) launch_bins<uint8_t>(a, q, bins, parts, st);
    else launch_bins<uint16_t>(a, q, bins, parts, st);
    if (a.clip_pct > 0) {
        clahe_maps<<<dim3(a.tx, a.ty), NBINS, 0, st>>>(a, q, parts, maps);
        const int quads = (a.W + 3) / 4, bx = std::min(PRE_THREADS, (quads + 31) / 32 * 32), by = PRE_THREADS / bx;
        clahe_apply<<<dim3((quads + bx - 1) / bx, (a.H + by - 1) / by), dim3(bx, by), 0, st>>>(a, q, bins, maps);
    }
    return cudaGetLastError();
}

}  // namespace rpiv
