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

// 1 / x to one unit of the last place (the device's estimate)
LFD_HD float reciprocal(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

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

// ---------------------------------------------------------------------------
// window tests of sweep samples: bilinear, positions in image coordinates
// ---------------------------------------------------------------------------
//
// A sample's position is X / Z with X = c + (a0 du + a1 dv), Z likewise (or Z
// constant): near the neighbour's principal plane, or far from the
// superpixel's anchor, terms much larger than X cancel in it.  With MX and MZ
// the largest sums of the terms' magnitudes over the box and Z >= zmin, one
// evaluation errs by at most 3 u MX / zmin + |x| (3 u MZ / zmin + 3 u), two of
// them by 12 u (MX + W MZ) / zmin, which is below BOX_MARGIN (0.215 px) where
// MX + W MZ <= BOX_REACH zmin.  A sample that is admitted so reads the texture
// from the entries -1 to W - 1 that the view has.
constexpr float BOX_REACH = 3e5f, BOX_MARGIN = 0.25f;

// the offsets [x0, x1] x [y0, y1] all sample inside a Wi x Hi view.  general:
// cz is the anchor's homogeneous coordinate; else Z is constant, cz = 1 / Z
LFD_HD bool box_inside(bool general, float a00, float a01, float a10, float a11, float a20, float a21, float cx,
                       float cy, float cz, int Wi, int Hi, int x0, int x1, int y0, int y1)
{
    const float mu = fmaxf(fabsf((float)x0), fabsf((float)x1)), mv = fmaxf(fabsf((float)y0), fabsf((float)y1));
    const float xe = (float)Wi - 0.5f - BOX_MARGIN, ye = (float)Hi - 0.5f - BOX_MARGIN;
    float zmin = INFINITY;
    bool in = true;
    for (int c = 0; c < 4; c++) {
        const float du = (float)((c & 1) ? x1 : x0), dv = (float)((c & 2) ? y1 : y0);
        const float X = fmaf(a00, du, fmaf(a01, dv, cx)), Y = fmaf(a10, du, fmaf(a11, dv, cy));
        float r = cz;
        if (general) {
            const float Z = fmaf(a20, du, fmaf(a21, dv, cz));
            zmin = fminf(zmin, Z);
            r = reciprocal(Z);
        }
        const float x = X * r, y = Y * r;
        in = in && x >= BOX_MARGIN - 0.5f && x <= xe && y >= BOX_MARGIN - 0.5f && y <= ye;
    }
    const float MX = fmaf(fabsf(a00), mu, fmaf(fabsf(a01), mv, fabsf(cx)));
    const float MY = fmaf(fabsf(a10), mu, fmaf(fabsf(a11), mv, fabsf(cy)));
    if (!general) return in && MX * cz + (float)Wi <= BOX_REACH && MY * cz + (float)Hi <= BOX_REACH;
    const float MZ = fmaf(fabsf(a20), mu, fmaf(fabsf(a21), mv, fabsf(cz)));
    return in && zmin > 0.f && fmaf((float)Wi, MZ, MX) <= BOX_REACH * zmin && fmaf((float)Hi, MZ, MY) <= BOX_REACH * zmin;
}

// ---------------------------------------------------------------------------
// sums of a label's costs in two orders
// ---------------------------------------------------------------------------
//
// Relative bound of the difference between two FP32 sums of the n * nnb
// non-negative samples of a label.  In the full sweep's order a sample goes
// through up to chunk * nnb additions of its chunk and one per chunk; in the
// order of the lanes (incumbent and last labels) through n / chunk * nnb of
// its lane, and fewer than 16 of the lanes and warps.  x: one rounding of u per
// addition of either order and 8 for the comparisons; 2 x^2 covers that
// roundings multiply.  Not doubled: labels closer than this are summed again,
// in the full sweep's order by few lanes, which large superpixels feel (48 of
// 25600 pixels, 33 labels, FP32 views: 28.3 ms with 2 x, 21.2 with x).
LFD_HD float sweep_eps(int n, int nnb, int chunk)
{
    const float chunks = (float)(n / chunk + 1);
    const float x = ((float)(chunk * nnb) + chunks * (float)(nnb + 1) + 24.f) * 5.9605e-8f;
    return fmaf(2.f * x, x, x);
}

}  // namespace lfd
