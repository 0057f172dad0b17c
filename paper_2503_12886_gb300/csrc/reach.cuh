// Which pixels a splat can reach: bounds of its alpha 1/255 ellipse, for the block masks of the tile
// lists (binsort.cu) and the pixel halves of a block (render.cu).
#pragma once
#include "rgba_internal.cuh"

namespace rgba {

// The region where a splat reaches alpha 1/255: the ellipse a dx^2 + 2 b dx dy + c dy^2 <= s,
// s = -2 alpha_cut(o), around (u, v).
struct Reach {
    bool none, all;  // never reaches it (decides over all); too elongated to bound tightly
    float u, v, ia, b, det, as, ys, hy;
};

// The square roots and quotients are the hardware's approximate ones: the widening below covers
// their few ulp many times over.
__device__ __forceinline__ float sqrt_fast(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// s is widened by 2 % and each block by 0.05 px, so that whatever is excluded fails the per-pixel
// FP32 test with room to spare: that test's power is off by at most a few 2^-24 (a dx^2 + c dy^2),
// which on the ellipse is a few 2^-24 s / (1 - b^2 / ac). Beyond ac / det = 10^4 (a splat a hundred
// times longer than wide) neither bound is trusted and every block is taken.
__device__ __forceinline__ Reach reach_of(const float4 &r0, const float2 &r1) {
    Reach e;
    const float a = r0.z, b = r0.w, c = r1.x, tau = alpha_cut(r1.y);
    // by fixed operations, so that whoever asks gets the same none
    const float det = __fmaf_rn(a, c, -__fmul_rn(b, b));
    e.none = !(tau < 0.0f && det > 0.0f);
    e.all = !(a * c < 1e4f * det);
    const float s = -2.04f * tau, id = __fdividef(1.0f, det);
    e.u = r0.x;
    e.v = r0.y;
    e.ia = __fdividef(1.0f, a);
    e.b = b;
    e.det = det;
    e.as = a * s;
    e.hy = sqrt_fast(e.as * id);
    const float hx = sqrt_fast(s * c * id);
    e.ys = -__fdividef(b, c) * hx;  // dy where the ellipse is furthest right (minus it: furthest left)
    return e;
}

// The x extent [xl, xr] of the ellipse over pixel-centre rows y0 .. y1, widened (empty: xl > xr).
// The right end over the rows is where dy is closest to ys, the left end closest to -ys.
__device__ __forceinline__ void reach_rows(const Reach &e, float y0, float y1, float &xl, float &xr) {
    const float d0 = y0 - 0.05f - e.v, d1 = y1 + 0.05f - e.v;
    xl = 1.0f;
    xr = -1.0f;
    if (d0 > e.hy || d1 < -e.hy) return;
    const float yr = fminf(fmaxf(e.ys, d0), d1), yl = fminf(fmaxf(-e.ys, d0), d1);
    xr = e.u + 0.05f + (sqrt_fast(fmaxf(0.0f, e.as - e.det * yr * yr)) - e.b * yr) * e.ia;
    xl = e.u - 0.05f - (sqrt_fast(fmaxf(0.0f, e.as - e.det * yl * yl)) + e.b * yl) * e.ia;
}

}  // namespace rgba
