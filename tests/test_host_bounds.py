"""The samples taken without a window test stay inside the view: random
hypotheses that land on the image border, far outside the anchor of the
current plane and near the neighbour's principal plane, through the corner
tests that admit them (csrc/lfd_bounds.cuh, compiled for the host)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1812_06856_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <random>
#include "lfd_bounds.cuh"
using namespace lfd;

// a rotation of the neighbour by angle a about y and b about x
static void pair(double f, int W, int H, double a, double b, const double t[3], double P[9], double q[3])
{
    const double R[9] = {cos(a), 0, sin(a), sin(a) * sin(b), cos(b), -cos(a) * sin(b), -sin(a) * cos(b), sin(b), cos(a) * cos(b)};
    const double K[9] = {f, 0, (W - 1) / 2.0, 0, f, (H - 1) / 2.0, 0, 0, 1};
    const double Ki[9] = {1 / f, 0, -K[2] / f, 0, 1 / f, -K[5] / f, 0, 0, 1};
    double KR[9];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            KR[3 * i + j] = 0;
            for (int k = 0; k < 3; k++) KR[3 * i + j] += K[3 * i + k] * R[3 * k + j];
        }
    for (int i = 0; i < 3; i++) {
        q[i] = 0;
        for (int k = 0; k < 3; k++) q[i] += K[3 * i + k] * t[k];
        for (int j = 0; j < 3; j++) {
            P[3 * i + j] = 0;
            for (int k = 0; k < 3; k++) P[3 * i + j] += KR[3 * i + k] * Ki[3 * k + j];
        }
    }
}

static float as_float(uint32_t u) { float f; __builtin_memcpy(&f, &u, 4); return f; }
static uint32_t as_bits(float f) { uint32_t u; __builtin_memcpy(&u, &f, 4); return u; }
// 1 / x within one unit of the last place, as the device's estimate
static float rcp(float x, int ulp) { return as_float(as_bits(1.0f / x) + ulp); }

// out: boxes admitted as inside, as outside, and those of each with a pixel that is not
extern "C" void refine_boxes(uint64_t seed, long trials, long out[4])
{
    std::mt19937_64 g(seed);
    auto U = [&](double lo, double hi) { return lo + (hi - lo) * (g() >> 11) * 0x1p-53; };
    for (int k = 0; k < 4; k++) out[k] = 0;
    const int sizes[4][2] = {{640, 480}, {1920, 1080}, {3840, 2160}, {32767, 400}};
    for (long it = 0; it < trials; it++) {
        const int *sz = sizes[g() & 3], W = sz[0], H = sz[1], side = 1 + (int)(g() % 24);
        const double f = W * U(0.5, 1.2), rs = U(0.01, 10.0);
        const double t[3] = {U(-2, 2), U(-0.2, 0.2), U(-2, 2)};
        double P[9], q[3];
        pair(f, W, H, U(-1.5, 1.5), U(-0.1, 0.1), t, P, q);
        const int rx = (int)U(0, W), ry = (int)U(0, H);
        double pr[3];
        for (int k = 0; k < 3; k++) pr[k] = P[3 * k] * rx + P[3 * k + 1] * ry + P[3 * k + 2];
        // anchor of the current plane: homogeneous coordinate from 1e-5 to 1; candidate: its own
        // position on the left or right border
        const double hwa = exp(U(-11.5, 0)), za = (hwa - pr[2]) / q[2];
        const double edge = (g() & 1 ? W - 0.5 : -0.5) + U(-1.2, 1.2);
        const double z1 = (edge * pr[2] - pr[0]) / (q[0] - edge * q[2]);
        if (!(z1 > 0) || !(za > 0) || z1 > 100 || za > 100) continue;
        const double g0 = U(-1, 1) * z1 / W, g1 = U(-1, 1) * z1 / W;
        const double hx = q[0] * za + pr[0], hy = q[1] * za + pr[1], hw = q[2] * za + pr[2];
        const double xa = fmin(fmax(floor(hx / hw), -1048576.0), 1048576.0), ya = fmin(fmax(floor(hy / hw), -1048576.0), 1048576.0);
        const float dgr = (float)(z1 - za), g0f = (float)g0, g1f = (float)g1;
        const float hwc = fmaf((float)(q[2] * rs), dgr, (float)(hw * rs));
        const float cx = fmaf((float)((q[0] - xa * q[2]) * rs), dgr, (float)((hx - xa * hw) * rs));
        const float cy = fmaf((float)((q[1] - ya * q[2]) * rs), dgr, (float)((hy - ya * hw) * rs));
        const float dx = (float)((q[0] - xa * q[2]) * rs), dy = (float)((q[1] - ya * q[2]) * rs), qw = (float)(q[2] * rs);
        const float b0 = fmaf(dx, g0f, (float)((P[0] - xa * P[6]) * rs)), b1 = fmaf(dx, g1f, (float)((P[1] - xa * P[7]) * rs));
        const float c0 = fmaf(dy, g0f, (float)((P[3] - ya * P[6]) * rs)), c1 = fmaf(dy, g1f, (float)((P[4] - ya * P[7]) * rs));
        const float a20 = fmaf(qw, g0f, (float)(P[6] * rs)), a21 = fmaf(qw, g1f, (float)(P[7] * rs));
        const int lo = -(int)(g() % (side + 1)), hi = lo + side;
        bool in = true, x0 = true, x1 = true, y0 = true, y1 = true;
        for (int c = 0; c < 4; c++) {
            const float du = (float)(c & 1 ? hi : lo), dv = (float)(c & 2 ? hi : lo);
            const float Nw = fmaf(a20, du, fmaf(a21, dv, hwc));
            const float ex = fmaf(b0, du, fmaf(b1, dv, cx)), ey = fmaf(c0, du, fmaf(c1, dv, cy));
            const CornerSides s = corner_sides(ex, ey, rcp(Nw, (int)(g() % 3) - 1), Nw, hwc, (int)xa, (int)ya, W, H);
            in = in && s.in;
            x0 = x0 && s.x0; x1 = x1 && s.x1; y0 = y0 && s.y0; y1 = y1 && s.y1;
        }
        const bool off = x0 || x1 || y0 || y1;
        if (!in && !off) continue;
        out[in ? 0 : 1]++;
        bool wrong = false;
        for (int v = lo; v <= hi; v++)
            for (int u = lo; u <= hi; u++) {
                const float du = (float)u, dv = (float)v, Nw = fmaf(a20, du, fmaf(a21, dv, hwc));
                const float ex = fmaf(b0, du, fmaf(b1, dv, cx)), ey = fmaf(c0, du, fmaf(c1, dv, cy));
                const float r = rcp(Nw, (int)(g() % 3) - 1);
                const float tx = fmaf(ex, r, 12582912.f), ty = fmaf(ey, r, 12582912.f);      // 1.5 * 2^23: nearest integer
                const uint32_t ix = as_bits(tx) - 0x4B400000u + (uint32_t)(int)xa, iy = as_bits(ty) - 0x4B400000u + (uint32_t)(int)ya;
                const bool pixel = Nw > 0.f && ix < (uint32_t)W && iy < (uint32_t)H;
                wrong = wrong || pixel != in;
            }
        if (wrong) out[in ? 2 : 3]++;
    }
}

// chunks of a superpixel in one neighbour view, near its border and its principal plane;
// out: boxes admitted, and those with a sample outside the window
extern "C" void sweep_boxes(uint64_t seed, long trials, long out[2])
{
    std::mt19937_64 g(seed);
    auto U = [&](double lo, double hi) { return lo + (hi - lo) * (g() >> 11) * 0x1p-53; };
    out[0] = out[1] = 0;
    const int sizes[4][2] = {{640, 480}, {1920, 1080}, {3840, 2160}, {32767, 400}};
    for (long it = 0; it < trials; it++) {
        const int *sz = sizes[g() & 3], W = sz[0], H = sz[1];
        const double f = W * U(0.5, 1.2), t[3] = {U(-2, 2), U(-0.2, 0.2), U(-2, 0)};
        const bool general = g() & 3;
        double P[9], q[3];
        pair(f, W, H, general ? U(-1.5, 1.5) : 0.0, general ? U(-0.1, 0.1) : 0.0, t, P, q);
        // the chunk's box, at any offset from the superpixel's anchor
        const int far = 1 << (g() % 12), x0 = (int)U(-far, far), y0 = (int)U(-far, far), w = (int)(g() % 12), h = (int)(g() % 12);
        const double px = U(0, W), py = U(0, H);
        const int rx = (int)px - x0, ry = (int)py - y0;
        double pr[3], pp[3];
        for (int k = 0; k < 3; k++) {
            pr[k] = P[3 * k] * rx + P[3 * k + 1] * ry + P[3 * k + 2];
            pp[k] = P[3 * k] * (rx + x0) + P[3 * k + 1] * (ry + y0) + P[3 * k + 2];
        }
        // a camera that has the box's first pixel on the window's edge, at 1e-4 to 1 of its depth
        const double edge = (g() & 1 ? W - 0.5 : -0.5) + U(-0.6, 0.6), z = U(0.1, 2), near = exp(U(-9, 0)), at = U(0, H);
        if (general) {
            q[0] = (edge * near - pp[0]) / z;
            q[1] = (at * near - pp[1]) / z;
            q[2] = (near - pp[2]) / z;
        }
        const float a00 = (float)P[0], a01 = (float)P[1], a10 = (float)P[3], a11 = (float)P[4], a20 = (float)P[6], a21 = (float)P[7];
        const float cx = (float)(z * q[0] + pr[0]), cy = (float)(z * q[1] + pr[1]), cw = (float)(z * q[2] + pr[2]);
        if (!general && !(cw > 0.f)) continue;
        const float rc = general ? cw : rcp(cw, (int)(g() % 3) - 1);
        if (!box_inside(general, a00, a01, a10, a11, a20, a21, cx, cy, rc, W, H, x0, x0 + w, y0, y0 + h)) continue;
        out[0]++;
        bool wrong = false;
        for (int v = y0; v <= y0 + h; v++)
            for (int u = x0; u <= x0 + w; u++) {
                const float fu = (float)u, fv = (float)v;
                const float A = fmaf(a00, fu, a01 * fv), B = fmaf(a10, fu, a11 * fv), wz = fmaf(a20, fu, a21 * fv) + cw;
                const float r = general ? rcp(wz, (int)(g() % 3) - 1) : rc, x = (A + cx) * r, y = (B + cy) * r;
                wrong = wrong || (general && !(wz > 0.f)) ||
                        !(x >= -0.5f && x < (float)W - 0.5f && y >= -0.5f && y < (float)H - 0.5f);
            }
        out[1] += wrong;
    }
}

extern "C" float bound_of_sums(int n, int nnb) { return sweep_eps(n, nnb, 128); }
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("inside")
    src, lib = d / "probe.cpp", d / "probe.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC, "-o", str(lib),
                           str(src)])
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_boxes_of_the_refinement_are_on_the_side_they_are_taken_for(probe, seed):
    out = (ctypes.c_long * 4)()
    probe.refine_boxes(ctypes.c_uint64(seed), ctypes.c_long(4_000_000), out)
    inside, outside, wrong_in, wrong_out = out
    assert inside > 1000 and outside > 1000
    assert (wrong_in, wrong_out) == (0, 0)


INDEX = r"""
#include <cstdio>
#include <random>
#include "lfd_bounds.cuh"
using namespace lfd;

int main()
{
    std::mt19937_64 g(1);
    for (int it = 0; it < 2000000; it++) {
        const int W = 1 + (int)(g() % 32767), H = 1 + (int)(g() % 32767), x = (int)(g() % W), y = (int)(g() % H);
        const int xa = (int)(g() % 2097153) - 1048576, ya = (int)(g() % 2097153) - 1048576;
        const float tx = (float)(x - xa) + 12582912.f, ty = (float)(y - ya) + 12582912.f;
        const int xm = xa - 0x4B400000, ym = ya - 0x4B400000;
        if (pixel_coord(tx, xm) != (unsigned)x || pixel_coord(ty, ym) != (unsigned)y) return 1;
        if (pixel_index(tx, ty, W, pixel_base(xm, ym, W)) != (unsigned)(y * W + x)) return 2;
        // an offset out of range is no pixel of any view
        unsigned bits = (unsigned)g();
        float f;
        memcpy(&f, &bits, 4);
        if (!(fabsf(f) < 4194304.f) && pixel_coord(f + 12582912.f, xm) < 32767u) return 3;
    }
    printf("ok");
    return 0;
}
"""


def test_pixel_indices_are_taken_modulo_two_to_the_32(tmp_path):
    (tmp_path / "index.cpp").write_text(INDEX)
    exe = tmp_path / "index"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fsanitize=signed-integer-overflow",
                           "-fsanitize-undefined-trap-on-error", "-I", CSRC, "-o", str(exe), str(tmp_path / "index.cpp")])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert (r.returncode, r.stdout) == (0, "ok")


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_boxes_of_the_sweep_are_inside(probe, seed):
    out = (ctypes.c_long * 2)()
    probe.sweep_boxes(ctypes.c_uint64(seed), ctypes.c_long(4_000_000), out)
    assert out[0] > 1000 and out[1] == 0


@pytest.mark.parametrize("nnb", [1, 2, 4, 8])
@pytest.mark.parametrize("n", [1, 127, 128, 256, 4096, 22_000, 65_536, 1 << 20, 1 << 24, (1 << 30) - 1])
def test_bound_of_sums_covers_every_addition(probe, n, nnb):
    """One rounding of 2^-24 for each addition a sample goes through: up to 128 nnb of its chunk and one per chunk in
    the full sweep's order; nnb per chunk of 128 pixels in a lane, 4 slots, 5 steps of a butterfly and 4 warps in the
    other."""
    probe.bound_of_sums.restype = ctypes.c_float
    chunks = -(-n // 128)
    additions = (128 * nnb + chunks) + (chunks * nnb + 4 + 5 + 4)
    assert probe.bound_of_sums(n, nnb) >= additions * 2.0 ** -24
