// Bilinear interpolation of a source grid's field at the nodes of another grid
// (pass-to-pass predictor, pyramid), shared by the interpolation kernel and the
// deformation, which interpolates the nodes it needs itself.
#pragma once

#include "rpiv_internal.h"

namespace rpiv {

// x / s for a positive integer s.  The reciprocal of a power of two is exact, so
// the product equals the quotient bit for bit; any other step is divided by
// (its rounded reciprocal would bias every weight the same way, up to 1e-5 px
// at 4k columns).  s is the same for the whole launch: the branch is uniform.
__device__ __forceinline__ float over_step(float x, int s)
{
    return (s & (s - 1)) == 0 ? x * __uint_as_float((uint32_t)(127 - (31 - __clz(s))) << 23) : x / (float)s;
}

__device__ __forceinline__ void axis_wf(float pos, int n, float c0, int s, int &i0, int &i1, float &t)
{
    if (n <= 1) {
        i0 = i1 = 0;
        t = 0.f;
        return;
    }
    float f = over_step(pos - c0, s);
    f = fminf(fmaxf(f, 0.f), (float)(n - 1));
    int ia = (int)floorf(f);
    if (ia > n - 2) ia = n - 2;
    i0 = ia;
    i1 = ia + 1;
    t = f - (float)ia;
}

// Field (su, sv) of a grid (snx x sny, window sw, step ss) at node (i, j) of a
// grid (window dw, step ds) whose image is levels_up pyramid levels finer.
__device__ __forceinline__ float2 interp_node(const float *su, const float *sv, int snx, int sny, int sw, int ss, int dw,
                                              int ds, int levels_up, int i, int j)
{
    const float f = (float)(1 << levels_up);
    const float X = (float)(i * ds) + 0.5f * (float)(dw - 1);
    const float Y = (float)(j * ds) + 0.5f * (float)(dw - 1);
    const float xs = over_step(X + 0.5f, 1 << levels_up) - 0.5f, ys = over_step(Y + 0.5f, 1 << levels_up) - 0.5f;
    const float c0 = 0.5f * (float)(sw - 1);
    int i0, i1, j0, j1;
    float tx, ty;
    axis_wf(xs, snx, c0, ss, i0, i1, tx);
    axis_wf(ys, sny, c0, ss, j0, j1, ty);
    const float u00 = su[j0 * snx + i0], u10 = su[j0 * snx + i1], u01 = su[j1 * snx + i0], u11 = su[j1 * snx + i1];
    const float v00 = sv[j0 * snx + i0], v10 = sv[j0 * snx + i1], v01 = sv[j1 * snx + i0], v11 = sv[j1 * snx + i1];
    float t0 = u00 + tx * (u10 - u00);
    float t1 = u01 + tx * (u11 - u01);
    const float u = f * (t0 + ty * (t1 - t0));
    t0 = v00 + tx * (v10 - v00);
    t1 = v01 + tx * (v11 - v01);
    return make_float2(u, f * (t0 + ty * (t1 - t0)));
}

}  // namespace rpiv
