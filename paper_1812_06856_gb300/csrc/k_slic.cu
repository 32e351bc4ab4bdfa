// SLIC superpixels on the GPU (Achanta et al. 2012; the segmentation step the
// method runs before Section III-A), with the grid-indexed labels the rest of
// the path expects (label = cell_y * grid_w + cell_x of the winning centre).
//
// Colour space CIELAB (sRGB companding, D65 white); seeds at the centres of
// the grid cells (boundaries at round(k W / grid_w), half up); a pixel of cell
// (cx, cy) compares the centres of the 3x3 cells around its own by
// D^2 = |lab - lab_c|^2 + (m / S)^2 |xy - xy_c|^2, ties to the first cell in
// row-major order; a centre becomes the mean of its pixels (kept when it has
// none).  No connectivity post-processing: the superpixel builder accepts any
// label map.  Deterministic: the update's sums are integers (Lab in fixed
// point), so their order does not matter.  Up to SLIC_BATCH
// views go through the same launches (blockIdx.y = view).
#include "lfd_slic.cuh"

namespace lfd {

__device__ __forceinline__ float srgb_linear(float c)
{
    return c <= 0.04045f ? c * (1.0f / 12.92f) : powf((c + 0.055f) * (1.0f / 1.055f), 2.4f);
}

__device__ __forceinline__ float lab_f(float t)
{
    return t > (216.0f / 24389.0f) ? cbrtf(t) : ((24389.0f / 27.0f) * t + 16.0f) * (1.0f / 116.0f);
}

__device__ __forceinline__ float3 linear_to_lab(float r, float g, float b)
{
    const float X = (0.4124564f * r + 0.3575761f * g + 0.1804375f * b) * (1.0f / 0.95047f);
    const float Y = 0.2126729f * r + 0.7151522f * g + 0.0721750f * b;
    const float Z = (0.0193339f * r + 0.1191920f * g + 0.9503041f * b) * (1.0f / 1.08883f);
    const float fx = lab_f(X), fy = lab_f(Y), fz = lab_f(Z);
    return make_float3(116.0f * fy - 16.0f, 500.0f * (fx - fy), 200.0f * (fy - fz));
}

__device__ __forceinline__ void texel_rgb(int fmt, const char *row, int x, float &r, float &g, float &b)
{
    if (fmt == LFD_RGBA8) {
        const uchar4 t = ((const uchar4 *)row)[x];
        r = t.x * (1.0f / 255.0f); g = t.y * (1.0f / 255.0f); b = t.z * (1.0f / 255.0f);
    } else if (fmt == LFD_RGBA_F16) {
        const __half *t = (const __half *)row + 4 * x;
        r = __half2float(t[0]); g = __half2float(t[1]); b = __half2float(t[2]);
    } else if (fmt == LFD_RGBA_BF16) {
        const __nv_bfloat16 *t = (const __nv_bfloat16 *)row + 4 * x;
        r = __bfloat162float(t[0]); g = __bfloat162float(t[1]); b = __bfloat162float(t[2]);
    } else {
        const float4 t = ((const float4 *)row)[x];
        r = t.x; g = t.y; b = t.z;
    }
}

// boundary k of n cells over `size` pixels: round(k size / n), half up
// (32-bit unsigned: 2 k size + n < 2^32 for sizes up to LFD_MAX_DIM)
__device__ __forceinline__ int cell_edge(int k, int size, int n)
{
    return (int)((2u * (unsigned)k * (unsigned)size + (unsigned)n) / (2u * (unsigned)n));
}

// The scratch is cell-major: cell c = cy GW + cx holds its pixels, row by row,
// at entries c stride .. of `lab`, so that a warp reads
// it as one contiguous run.  A Lab entry's
// fourth word is (y << 16 | x).  The entries past a cell's last pixel hold a
// NaN colour and a negative fourth word: they pick no centre.
//
// A CTA's 8 warps take 8 / wpc cells, wpc warps each (wpc a power of two, see
// launch_slic).
constexpr int SLIC_WARPS = 8;

// The 256 values a byte channel can take go through powf once per CTA instead
// of three times per pixel (8 x 1024x768 RGBA8: 70 -> 42 us).
__global__ void __launch_bounds__(32 * SLIC_WARPS) k_slic_lab(const __grid_constant__ SlicBatch b, int wpc)
{
    const SlicView &s = b.v[blockIdx.y];
    __shared__ float lut[256];
    if (s.fmt == LFD_RGBA8) {
        lut[threadIdx.x] = srgb_linear(threadIdx.x * (1.0f / 255.0f));
        __syncthreads();
    }
    const int wid = threadIdx.x >> 5;
    const int c = blockIdx.x * (SLIC_WARPS / wpc) + wid / wpc;
    if (c >= s.GW * s.GH) return;
    const int cx = c % s.GW, cy = c / s.GW;
    const int x0 = cell_edge(cx, s.W, s.GW), cw = cell_edge(cx + 1, s.W, s.GW) - x0;
    const int y0 = cell_edge(cy, s.H, s.GH), n = cw * (cell_edge(cy + 1, s.H, s.GH) - y0);
    float4 *lab = s.lab + (long long)c * s.stride;
    for (int i = (wid % wpc) * 32 + (threadIdx.x & 31); i < s.stride; i += 32 * wpc) {
        if (i >= n) {
            const float nan = __int_as_float(0x7fffffff);
            lab[i] = make_float4(nan, nan, nan, __int_as_float(-1));
            continue;
        }
        const int x = x0 + i % cw, y = y0 + i / cw;
        const char *row = (const char *)s.img + (long long)y * s.pitch;
        float3 l;
        if (s.fmt == LFD_RGBA8) {
            const uchar4 t = ((const uchar4 *)row)[x];
            l = linear_to_lab(lut[t.x], lut[t.y], lut[t.z]);
        } else {
            float r, g, bl;
            texel_rgb(s.fmt, row, x, r, g, bl);
            l = linear_to_lab(srgb_linear(r), srgb_linear(g), srgb_linear(bl));
        }
        lab[i] = make_float4(l.x, l.y, l.z, __int_as_float((y << 16) | x));
    }
}

__global__ void k_slic_seeds(const __grid_constant__ SlicBatch b)
{
    const SlicView &s = b.v[blockIdx.y];
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.GW * s.GH) return;
    const int cx = c % s.GW, cy = c / s.GW;
    const float x = 0.5f * (float)(cell_edge(cx, s.W, s.GW) + cell_edge(cx + 1, s.W, s.GW) - 1);
    const float y = 0.5f * (float)(cell_edge(cy, s.H, s.GH) + cell_edge(cy + 1, s.H, s.GH) - 1);
    const int px = min((int)floorf(x + 0.5f), s.W - 1), py = min((int)floorf(y + 0.5f), s.H - 1);
    const int x0 = cell_edge(cx, s.W, s.GW), cw = cell_edge(cx + 1, s.W, s.GW) - x0, y0 = cell_edge(cy, s.H, s.GH);
    const float4 l = s.lab[(long long)c * s.stride + (py - y0) * cw + (px - x0)];    // a pixel of the own cell
    float *o = s.centres + 5 * (long long)c;
    o[0] = l.x; o[1] = l.y; o[2] = l.z; o[3] = x; o[4] = y;
}

// Fixed-point scale of the Lab sums: 2^18 (a power of two, so v * 2^18 is
// exact and the rounding error of one value is at most 2^-19), on values
// clamped to [-256, 256] (every sRGB colour is inside).  Integer sums are associative: the update does not depend on
// the order of its sums.
constexpr float SLIC_FIX = 262144.0f;
constexpr float SLIC_LAB_MAX = 256.0f;

__device__ __forceinline__ int slic_fix(float v)
{
    return __float2int_rn(fminf(fmaxf(v, -SLIC_LAB_MAX), SLIC_LAB_MAX) * SLIC_FIX);
}

// A cell's pixels pick the nearest of the 3x3 cells' centres (ties to the
// first in row-major order; the own cell, and no mean, when every distance is
// NaN).  FINAL writes the labels; otherwise the picks go into the sums {L, a, b
// in fixed point, x, y, count} of the cell's pixels per centre picked,
// s.sums[cell][9][6], which k_slic_update adds up centre by centre: no atomics.
//
// Lanes take pixels in pairs: a centre's shared-memory broadcast, every
// component twice, feeds the packed FP32 operations for both; each operation
// rounds as the scalar one.  After 128 pixels (four a lane) the warp sums the
// picks of one centre after the other, of those present: lane sums fit 32 bits
// (four values below 2^26), a REDUX each for their low and high halves, and
// lane j keeps centre j's totals.  Offsets in the cell are summed as one word
// (dy << 16 | dx) unless WIDE (cells above 256 pixels across).
//
// 8 x 1024x768 RGBA8, 4015 cells of 14 x 14 pixels per view, 10 iterations:
// 103 us an assignment with its sums, 8 us an update, 1.30 ms in all; with one
// byte per pixel out and the sums gathered by a warp per centre from its 3x3
// cells 46 and 80 us, 1.43 ms; with one CTA per cell, REDUX per quantity and
// winner and 64-bit atomics 272 us an iteration, 3.02 ms.  Bound by issue; 3
// CTAs per SM at 80 registers (4 at 64 spill: 1.34 ms).
template <bool FINAL, bool WIDE>
__global__ void __launch_bounds__(32 * SLIC_WARPS, 3) k_slic_assign(const __grid_constant__ SlicBatch b, int parity,
                                                                    int wpc)
{
    const SlicView &s = b.v[blockIdx.y];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int c = blockIdx.x * (SLIC_WARPS / wpc) + wid / wpc;
    __shared__ float4 cen[SLIC_WARPS][9][3];     // {L, L, a, a}, {b, b, x, x}, {y, y, -, -}
    __shared__ long long part[FINAL ? 1 : SLIC_WARPS][9][6];
    const bool here = c < s.GW * s.GH;           // whole warp
    long long tot[6] = {0, 0, 0, 0, 0, 0};       // lane j: centre j's sums
    if (here) {
        const float *centres = parity ? s.centres2 : s.centres;
        const float2 wxy = dup2(b.wxy[blockIdx.y]);
        const int cx = c % s.GW, cy = c / s.GW;
        const int x0 = cell_edge(cx, s.W, s.GW), y0 = cell_edge(cy, s.H, s.GH);
        if (lane < 9) {
            const int nx = cx + lane % 3 - 1, ny = cy + lane / 3 - 1;
            const bool in = nx >= 0 && ny >= 0 && nx < s.GW && ny < s.GH;
            const float *o = centres + 5 * (long long)(in ? ny * s.GW + nx : c);
            const float L = in ? o[0] : INFINITY;    // no cell there: an infinite distance wins nothing
            cen[wid][lane][0] = make_float4(L, L, o[1], o[1]);
            cen[wid][lane][1] = make_float4(o[2], o[2], o[3], o[3]);
            cen[wid][lane][2] = make_float4(o[4], o[4], 0.f, 0.f);
        }
        __syncwarp();
        const float4 *lab = s.lab + (long long)c * s.stride;
#pragma unroll 1
        for (int base = (wid % wpc) * 128; base < s.stride; base += 128 * wpc) {
            float4 px[4];
            int pick[4];
#pragma unroll
            for (int u = 0; u < 4; u++) px[u] = __ldg(lab + min(base + 32 * u + lane, s.stride - 1));
            float2 vl[2], va[2], vb[2], vx[2], vy[2], best[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const float4 l0 = px[2 * h], l1 = px[2 * h + 1];
                const int p0 = __float_as_int(l0.w), p1 = __float_as_int(l1.w);
                vl[h] = make_float2(l0.x, l1.x);
                va[h] = make_float2(l0.y, l1.y);
                vb[h] = make_float2(l0.z, l1.z);
                vx[h] = make_float2((float)(p0 & 0xffff), (float)(p1 & 0xffff));
                vy[h] = make_float2((float)(p0 >> 16), (float)(p1 >> 16));
                best[h] = make_float2(INFINITY, INFINITY);
                pick[2 * h] = pick[2 * h + 1] = 255;
            }
#pragma unroll
            for (int j = 0; j < 9; j++) {
                const float4 q0 = cen[wid][j][0], q1 = cen[wid][j][1];
                const float2 q2 = *(const float2 *)&cen[wid][j][2];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const float2 dl = fsub2(vl[h], make_float2(q0.x, q0.y)), da = fsub2(va[h], make_float2(q0.z, q0.w));
                    const float2 db = fsub2(vb[h], make_float2(q1.x, q1.y)), dx = fsub2(vx[h], make_float2(q1.z, q1.w));
                    const float2 dy = fsub2(vy[h], q2);
                    const float2 col = ffma2(dl, dl, ffma2(da, da, fmul2(db, db)));
                    const float2 D = ffma2(wxy, ffma2(dx, dx, fmul2(dy, dy)), col);
                    if (D.x < best[h].x) { best[h].x = D.x; pick[2 * h] = j; }
                    if (D.y < best[h].y) { best[h].y = D.y; pick[2 * h + 1] = j; }
                }
            }
            // past the cell's entries (the clamped loads): no pick
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (base + 32 * u + lane >= s.stride) pick[u] = 256;
            if (FINAL) {
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int p = __float_as_int(px[u].w), j = pick[u] == 255 ? 4 : pick[u];
                    if (pick[u] < 256 && p >= 0)
                        s.labels[(long long)(p >> 16) * s.W + (p & 0xffff)] = c + (j / 3 - 1) * s.GW + j % 3 - 1;
                }
                continue;
            }
            int q[4][3], off[4];
            unsigned mine = 0;
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int p = __float_as_int(px[u].w);
                q[u][0] = slic_fix(px[u].x);
                q[u][1] = slic_fix(px[u].y);
                q[u][2] = slic_fix(px[u].z);
                off[u] = (((p >> 16) - y0) << 16) | ((p & 0xffff) - x0);
                mine |= pick[u] < 9 ? 1u << pick[u] : 0u;
            }
            unsigned present = __reduce_or_sync(0xffffffffu, mine);
            while (present) {
                const int j = __ffs(present) - 1;
                present &= present - 1;
                int t[3] = {0, 0, 0}, xy = 0, yy = 0, n = 0;
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (pick[u] == j) {
                        t[0] += q[u][0];
                        t[1] += q[u][1];
                        t[2] += q[u][2];
                        if (WIDE) {
                            xy += off[u] & 0xffff;
                            yy += off[u] >> 16;
                        } else {
                            xy += off[u];
                        }
                        n++;
                    }
                long long r[6];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)t[k] & 0xffffu);
                    const int hi = __reduce_add_sync(0xffffffffu, t[k] >> 16);
                    r[k] = ((long long)hi << 16) + lo;
                }
                const unsigned sxy = __reduce_add_sync(0xffffffffu, (unsigned)xy);
                const unsigned sn = __reduce_add_sync(0xffffffffu, (unsigned)n);
                const unsigned sy = WIDE ? __reduce_add_sync(0xffffffffu, (unsigned)yy) : sxy >> 16;
                r[3] = (long long)(WIDE ? sxy : sxy & 0xffffu) + (long long)sn * x0;
                r[4] = (long long)sy + (long long)sn * y0;
                r[5] = sn;
                if (lane == j)
#pragma unroll
                    for (int k = 0; k < 6; k++) tot[k] += r[k];
            }
        }
    }
    if (FINAL) return;
    if (wpc > 1) {                               // the warps that share the cell
        if (lane < 9)
#pragma unroll
            for (int k = 0; k < 6; k++) part[wid][lane][k] = tot[k];
        __syncthreads();
        if (wid % wpc) return;
        if (lane < 9)
            for (int o = 1; o < wpc; o++)
#pragma unroll
                for (int k = 0; k < 6; k++) tot[k] += part[wid + o][lane][k];
    }
    if (here && lane < 9) {
        longlong2 *out = (longlong2 *)(s.sums + 54 * (long long)c + 6 * lane);
        out[0] = make_longlong2(tot[0], tot[1]);
        out[1] = make_longlong2(tot[2], tot[3]);
        out[2] = make_longlong2(tot[4], tot[5]);
    }
}

// a centre becomes the mean of the pixels that picked it in its 3x3 cells
// (kept when there are none)
__global__ void __launch_bounds__(128) k_slic_update(const __grid_constant__ SlicBatch b, int parity)
{
    const SlicView &s = b.v[blockIdx.y];
    const int c = blockIdx.x * 128 + threadIdx.x;
    if (c >= s.GW * s.GH) return;
    const int cx = c % s.GW, cy = c / s.GW;
    long long t[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 9; q++) {
        const int nx = cx + q % 3 - 1, ny = cy + q / 3 - 1;
        if (nx < 0 || ny < 0 || nx >= s.GW || ny >= s.GH) continue;
        // this centre as that cell numbers it
        const longlong2 *in = (const longlong2 *)(s.sums + 54 * (long long)(ny * s.GW + nx) + 6 * (8 - q));
        const longlong2 u = __ldg(in), v = __ldg(in + 1), w = __ldg(in + 2);
        t[0] += u.x; t[1] += u.y; t[2] += v.x; t[3] += v.y; t[4] += w.x; t[5] += w.y;
    }
    const float *cin = (parity ? s.centres2 : s.centres) + 5 * (long long)c;
    float *o = (parity ? s.centres : s.centres2) + 5 * (long long)c;
    if (t[5] > 0) {
        const double r = 1.0 / (double)t[5];
        for (int j = 0; j < 3; j++) o[j] = (float)((double)t[j] * r * (1.0 / SLIC_FIX));
        o[3] = (float)((double)t[3] * r);
        o[4] = (float)((double)t[4] * r);
    } else {
        for (int j = 0; j < 5; j++) o[j] = cin[j];
    }
}

cudaError_t launch_slic(const SlicBatch &b, const float *const *centres_in, int iterations,
                        float *const *centres_out, cudaStream_t st)
{
    // warps per cell: one as long as that fills the chip (152 SMs, 32 warps
    // each), more for few or large cells while each warp keeps a step of 128 pixels
    int wpc = 1;
    while (wpc < SLIC_WARPS && b.max_stride > 128 * wpc &&
           (b.max_stride > 1024 * wpc || (long long)b.max_cells * b.n * wpc < 152 * 32))
        wpc *= 2;
    const int per_cta = SLIC_WARPS / wpc;
    const dim3 grid((b.max_cells + per_cta - 1) / per_cta, b.n);
    constexpr int threads = 32 * SLIC_WARPS;
    const dim3 g_cells((b.max_cells + 127) / 128, b.n);
    bool wide = false;                       // (dy << 16 | dx) sums of 128 pixels fit below 256 x 256
    for (int v = 0; v < b.n; v++)
        wide = wide || b.v[v].W > 256 * b.v[v].GW || b.v[v].H > 256 * b.v[v].GH;
    k_slic_lab<<<grid, threads, 0, st>>>(b, wpc);
    bool seeds = false;
    for (int v = 0; v < b.n; v++) {
        const SlicView &s = b.v[v];
        const size_t S = (size_t)s.GW * s.GH;
        if (!(centres_in && centres_in[v])) {
            seeds = true;
            continue;
        }
        cudaError_t e = cudaMemcpyAsync(s.centres, centres_in[v], sizeof(float) * 5 * S, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
    }
    if (seeds) {
        // views with given centres keep them: seed only the others
        SlicBatch bs = b;
        int k = 0;
        for (int v = 0; v < b.n; v++)
            if (!(centres_in && centres_in[v])) bs.v[k++] = b.v[v];
        bs.n = k;
        k_slic_seeds<<<dim3((b.max_cells + 127) / 128, k), 128, 0, st>>>(bs);
    }
    for (int it = 0; it < iterations; it++) {
        if (wide) k_slic_assign<false, true><<<grid, threads, 0, st>>>(b, it & 1, wpc);
        else k_slic_assign<false, false><<<grid, threads, 0, st>>>(b, it & 1, wpc);
        k_slic_update<<<g_cells, 128, 0, st>>>(b, it & 1);
    }
    const int parity = iterations & 1;
    k_slic_assign<true, false><<<grid, threads, 0, st>>>(b, parity, wpc);
    for (int v = 0; v < b.n && centres_out; v++) {
        if (!centres_out[v]) continue;
        const SlicView &s = b.v[v];
        cudaError_t e = cudaMemcpyAsync(centres_out[v], parity ? s.centres2 : s.centres,
                                        sizeof(float) * 5 * (size_t)s.GW * s.GH, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace lfd
