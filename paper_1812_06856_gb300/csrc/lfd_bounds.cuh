// Bounds of FP32 rounding that let the kernels leave work out, as plain
// arithmetic that also compiles for the host (u = 2^-24, the rounding of one
// operation).
#pragma once
#include <math.h>
#include <string.h>
#ifdef __CUDACC__
#define LFD_HD __host__ __device__ __forceinline__
#else
#define LFD_HD inline
#endif

namespace lfd {

// ---------------------------------------------------------------------------
// window tests of energy samples: nearest pixel, positions relative to an anchor
// ---------------------------------------------------------------------------
//
// A homography takes a box in front of the camera into the hull of its
// corners, so exact corners would decide for every pixel of the box; the margin
// covers that corners and pixels are each rounded.
//
// A pixel's offset f from the anchor pixel is ex / Nw, both affine in the
// pixel.  With |f| <= F at the corners and Nw within a factor 16 over the box,
// which holds the anchor, one evaluation errs by at most 36 u F (two roundings
// of ex and of Nw, their inner sums up to 16 times the result, and 2 u of the
// reciprocal); corner and pixel together, with the corner's sum anchor + f, by
// 75 u F.  INSIDE_MARGIN covers that up to F = INSIDE_REACH, 0.293 px; boxes
// further from the anchor (the anchor follows the current plane and may lie
// 2^20 px outside the view) are left to the tested samples.
constexpr float INSIDE_REACH = 65536.f, INSIDE_MARGIN = 0.3f;

struct CornerSides {
    bool in;                     // inside the window by the margin
    bool x0, x1, y0, y1;         // outside it by the margin: left, right, above, below
};

// corner at ex / Nw, ey / Nw (r = 1 / Nw) from the anchor pixel (xa, ya) of a
// Wi x Hi view; hw: the anchor's own homogeneous coordinate
LFD_HD CornerSides corner_sides(float ex, float ey, float r, float Nw, float hw, int xa, int ya, int Wi, int Hi)
{
    const float fx = ex * r, fy = ey * r, x = (float)xa + fx, y = (float)ya + fy;
    const float lo = -0.5f - INSIDE_MARGIN, xe = (float)Wi - 0.5f + INSIDE_MARGIN, ye = (float)Hi - 0.5f + INSIDE_MARGIN;
    const float xi = (float)Wi - 0.5f - INSIDE_MARGIN, yi = (float)Hi - 0.5f - INSIDE_MARGIN;
    const bool fit = hw > 0.f && Nw > 0.25f * hw && Nw < 4.f * hw && fabsf(fx) <= INSIDE_REACH &&
                     fabsf(fy) <= INSIDE_REACH;
    CornerSides c;
    c.in = fit && x >= -0.5f + INSIDE_MARGIN && x <= xi && y >= -0.5f + INSIDE_MARGIN && y <= yi;
    c.x0 = fit && x < lo;
    c.x1 = fit && x > xe;
    c.y0 = fit && y < lo;
    c.y1 = fit && y > ye;
    return c;
}

// Nearest pixels by adding 1.5 * 2^23: t carries the offset from the anchor
// pixel in its low bits, a_m is the anchor pixel minus the bits of 1.5 * 2^23.
// Modulo 2^32: an offset out of range (|f| >= 2^22, infinite, NaN) gives a
// coordinate that no view has.
LFD_HD unsigned float_bits(float t)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(t);
#else
    unsigned u;
    memcpy(&u, &t, 4);
    return u;
#endif
}

LFD_HD unsigned pixel_coord(float t, int a_m) { return float_bits(t) + (unsigned)a_m; }

// index of an inside pixel in a view of width Wi, base = pixel_base(xa_m, ya_m, Wi)
LFD_HD unsigned pixel_base(int xa_m, int ya_m, int Wi) { return (unsigned)ya_m * (unsigned)Wi + (unsigned)xa_m; }

LFD_HD unsigned pixel_index(float tx, float ty, int Wi, unsigned base)
{
    return float_bits(ty) * (unsigned)Wi + (float_bits(tx) + base);
}

}  // namespace lfd
