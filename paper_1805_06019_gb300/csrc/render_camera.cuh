// Camera geometry of native-size rendering, shared by its kernels: the grid
// cell of a camera, its four neighbour views, and the stencil each of them
// contributes (Section 3.6).
#pragma once

#include <climits>

#include "rlfc_internal.h"

namespace rlfc {

struct Grid {
    uint32_t U, V, W, H;
    uint32_t cells_u, cells_v;   // cells of neighbouring cameras (one where an axis has one camera)
};

inline Grid make_grid(uint32_t U, uint32_t V, uint32_t W, uint32_t H)
{
    return Grid{U, V, W, H, U > 1 ? U - 1 : 1, V > 1 ? V - 1 : 1};
}

__device__ __forceinline__ void camera_axis(float u, uint32_t G, uint32_t &i0, float &f)
{
    u = fminf(fmaxf(u, 0.0f), (float)(G - 1));
    if (G == 1) {
        i0 = 0;
        f = 0.0f;
        return;
    }
    i0 = (uint32_t)min((int)floorf(u), (int)G - 2);
    f = u - (float)i0;
}

struct CameraCell {
    uint32_t ci, cj;   // cell: neighbours (ci, cj) .. (ci + 1, cj + 1)
    float u, v;        // position, clamped to the grid
    float fu, fv;
};

__device__ __forceinline__ void camera_cell(const Grid &g, const float *uv, uint32_t r, CameraCell &c)
{
    c.u = fminf(fmaxf(uv[2 * r], 0.0f), (float)(g.U - 1));
    c.v = fminf(fmaxf(uv[2 * r + 1], 0.0f), (float)(g.V - 1));
    camera_axis(c.u, g.U, c.ci, c.fu);
    camera_axis(c.v, g.V, c.cj, c.fv);
}

__device__ __forceinline__ uint32_t neighbour_view(const Grid &g, uint32_t ci, uint32_t cj, int k)
{
    const uint32_t i = g.U == 1 ? 0u : ci + (uint32_t)(k & 1), j = g.V == 1 ? 0u : cj + (uint32_t)(k >> 1);
    return j * g.U + i;
}

struct Stencil {
    int ox, oy;       // integer part of the neighbour's shift
    float fx, fy;     // fractional part
    float sx, sy;     // the shift
};

// The neighbours' blend weights and shifts for focus disparity d.
__device__ __forceinline__ void camera_stencils(const Grid &g, const CameraCell &c, float d, float w[4], Stencil st[4])
{
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int ia = k & 1, jb = k >> 1;
        const int i = g.U == 1 ? 0 : (int)c.ci + ia, j = g.V == 1 ? 0 : (int)c.cj + jb;
        w[k] = (ia ? c.fu : 1.0f - c.fu) * (jb ? c.fv : 1.0f - c.fv);
        // a shift beyond twice the image size samples only the clamped edge
        // either way; bounding it keeps the integer pixel arithmetic in range
        const float lim = 2.0f * (float)max(g.W, g.H) + 4.0f;
        const float sx = fminf(fmaxf(d * ((float)i - c.u), -lim), lim);
        const float sy = fminf(fmaxf(d * ((float)j - c.v), -lim), lim);
        const float flx = floorf(sx), fly = floorf(sy);
        st[k].ox = (int)flx;
        st[k].oy = (int)fly;
        st[k].fx = sx - flx;
        st[k].fy = sy - fly;
        st[k].sx = sx;
        st[k].sy = sy;
    }
}

// ray of an output pixel, bilinear taps along one axis with clamp-to-edge
__device__ __forceinline__ float ray_s(uint32_t x, uint32_t W, uint32_t out_w)
{
    return ((float)x + 0.5f) * (float)W / (float)out_w - 0.5f;
}
__device__ __forceinline__ void taps(float xs, uint32_t W, int &xa, int &xb, float &fx)
{
    const float x0 = floorf(xs);
    fx = xs - x0;
    const int xi = (int)x0;
    xa = min(max(xi, 0), (int)W - 1);
    xb = min(max(xi + 1, 0), (int)W - 1);
}

// x / 255, correctly rounded, for x = 0 and normal x whose quotient is
// normal: 1/255 as the sum of two floats (Brisebarre, Muller and Raina,
// "Accelerating correctly rounded floating-point division when the divisor is
// known in advance", 2004; checked for every mantissa).  Two instructions
// instead of a division, twelve times a pixel: the sampled renderer takes 79
// instead of 89 us for eight 800 x 600 views.
__device__ __forceinline__ float div255(float x)
{
    constexpr float hi = 1.0f / 255.0f, lo = (float)(1.0 / 255.0 - (double)hi);
    return fmaf(x, hi, x * lo);
}

// One neighbour's bilinear sample at any output size, weighted and added.
__device__ __forceinline__ void sample_add(float w, float fx, float fy, uint32_t p00, uint32_t p10, uint32_t p01, uint32_t p11,
                                           float acc[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const auto v = [c](uint32_t rgb) { return (float)((rgb >> (8 * c)) & 255u); };
        const float top = (1.0f - fx) * v(p00) + fx * v(p10);
        const float bot = (1.0f - fx) * v(p01) + fx * v(p11);
        acc[c] += w * div255((1.0f - fy) * top + fy * bot);
    }
}

}  // namespace rlfc
