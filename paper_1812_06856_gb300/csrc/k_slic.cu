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
// at entries c stride .. of `lab` and `code`, so that a warp reads a cell, or
// the three cells of a window's row, as one contiguous run.  A Lab entry's
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
// first in row-major order): code 0..8, or 255 when every distance is NaN (a
// colour that is not finite keeps its own cell and enters no mean).  FINAL
// writes the labels instead.  Lanes take pixels in pairs: a centre's
// shared-memory broadcast, every component twice, feeds the packed FP32
// operations for both; each operation rounds as the scalar one.
//
// 8 x 1024x768 RGBA8, 4015 cells of 14 x 14 pixels per view, 10 iterations:
// 46 us an assignment and 80 us an update, 1.44 ms in all; one CTA per cell
// that also added every pixel to its winner's sums (REDUX per quantity and
// winner, 64-bit atomics) took 272 us an iteration, 3.02 ms in all.  Both
// kernels are bound by issue and latency together (63 % issue-active at 40
// warps per SM); the Lab entries (108 MB) come from HBM once per iteration,
// 2.2 TB/s.
template <bool FINAL>
__global__ void __launch_bounds__(32 * SLIC_WARPS, 5) k_slic_assign(const __grid_constant__ SlicBatch b, int parity,
                                                                 int wpc)
{
    const SlicView &s = b.v[blockIdx.y];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int c = blockIdx.x * (SLIC_WARPS / wpc) + wid / wpc;
    if (c >= s.GW * s.GH) return;                // whole warp
    const float *centres = parity ? s.centres2 : s.centres;
    const float2 wxy = dup2(b.wxy[blockIdx.y]);
    __shared__ float4 cen[SLIC_WARPS][9][3];     // {L, L, a, a}, {b, b, x, x}, {y, y, -, -}
    const int cx = c % s.GW, cy = c / s.GW;
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
    unsigned char *code = s.code + (long long)c * s.stride;
    for (int i0 = (wid % wpc) * 64 + lane; i0 - lane < s.stride; i0 += 64 * wpc) {
        const int i1 = i0 + 32;
        const float4 l0 = __ldg(lab + min(i0, s.stride - 1)), l1 = __ldg(lab + min(i1, s.stride - 1));
        const int p0 = __float_as_int(l0.w), p1 = __float_as_int(l1.w);
        const float2 vl = make_float2(l0.x, l1.x), va = make_float2(l0.y, l1.y), vb = make_float2(l0.z, l1.z);
        const float2 vx = make_float2((float)(p0 & 0xffff), (float)(p1 & 0xffff));
        const float2 vy = make_float2((float)(p0 >> 16), (float)(p1 >> 16));
        float best0 = INFINITY, best1 = INFINITY;
        int k0 = 255, k1 = 255;
#pragma unroll
        for (int j = 0; j < 9; j++) {
            const float4 q0 = cen[wid][j][0], q1 = cen[wid][j][1];
            const float2 q2 = *(const float2 *)&cen[wid][j][2];
            const float2 dl = fsub2(vl, make_float2(q0.x, q0.y)), da = fsub2(va, make_float2(q0.z, q0.w));
            const float2 db = fsub2(vb, make_float2(q1.x, q1.y)), dx = fsub2(vx, make_float2(q1.z, q1.w));
            const float2 dy = fsub2(vy, q2);
            const float2 col = ffma2(dl, dl, ffma2(da, da, fmul2(db, db)));
            const float2 D = ffma2(wxy, ffma2(dx, dx, fmul2(dy, dy)), col);
            if (D.x < best0) { best0 = D.x; k0 = j; }
            if (D.y < best1) { best1 = D.y; k1 = j; }
        }
        if (FINAL) {
            const int j0 = k0 == 255 ? 4 : k0, j1 = k1 == 255 ? 4 : k1;
            if (i0 < s.stride && p0 >= 0)
                s.labels[(long long)(p0 >> 16) * s.W + (p0 & 0xffff)] = c + (j0 / 3 - 1) * s.GW + j0 % 3 - 1;
            if (i1 < s.stride && p1 >= 0)
                s.labels[(long long)(p1 >> 16) * s.W + (p1 & 0xffff)] = c + (j1 / 3 - 1) * s.GW + j1 % 3 - 1;
        } else {
            if (i0 < s.stride) code[i0] = (unsigned char)k0;
            if (i1 < s.stride) code[i1] = (unsigned char)k1;
        }
    }
}

// exact sum over the warp of 64-bit values below 2^62 in magnitude: three
// 22-bit limbs, one REDUX each (the top one signed)
__device__ __forceinline__ long long warp_sum64(long long v)
{
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x3fffffu);
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 22) & 0x3fffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 44));
    return ((long long)hi << 44) + ((long long)mid << 22) + (long long)lo;
}

// A centre becomes the mean of the pixels that picked it (kept when there are
// none): its warps find them among the codes of the centre's 3x3 cells, four a
// word and a window row (three cells) as one run, list them in shared memory
// and sum them with full lanes, {L, a, b} in fixed point.
constexpr int SLIC_LIST = 512;

__global__ void __launch_bounds__(32 * SLIC_WARPS, 5) k_slic_update(const __grid_constant__ SlicBatch b, int parity,
                                                                 int wpc)
{
    const SlicView &s = b.v[blockIdx.y];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int c = blockIdx.x * (SLIC_WARPS / wpc) + wid / wpc;
    __shared__ int list[SLIC_WARPS][SLIC_LIST];
    __shared__ long long tot[SLIC_WARPS][6];
    const bool here = c < s.GW * s.GH;           // whole warp
    long long sum[6] = {0, 0, 0, 0, 0, 0};       // L, a, b (fixed point), x, y, count
    if (here) {
        const int cx = c % s.GW, cy = c / s.GW;
        const unsigned lt = (1u << lane) - 1u;
        const int words = s.stride >> 2;
        int have = 0;
        auto drain = [&]() {                     // at most 16 entries a lane: 32-bit sums
            __syncwarp();
            int q[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 4
            for (int e = lane; e < have; e += 32) {
                const float4 l = __ldg(s.lab + list[wid][e]);
                const int p = __float_as_int(l.w);
                q[0] += slic_fix(l.x);
                q[1] += slic_fix(l.y);
                q[2] += slic_fix(l.z);
                q[3] += p & 0xffff;
                q[4] += p >> 16;
                q[5]++;
            }
#pragma unroll
            for (int k = 0; k < 6; k++) sum[k] += q[k];
            have = 0;
            __syncwarp();
        };
        const int xl = max(cx - 1, 0), cells = min(cx + 1, s.GW - 1) - xl + 1;   // of a window row
        const int run = cells * words;
        for (int ny = max(cy - 1, 0); ny <= min(cy + 1, s.GH - 1); ny++) {
            const int first = (ny * s.GW + xl) * s.stride;
            const unsigned *code = (const unsigned *)(s.code + first);
            // this centre as the row's first cell numbers it; one less per cell to the right
            const int want = (cy - ny + 1) * 3 + (cx - xl + 1);
#pragma unroll 2
            for (int w0 = (wid % wpc) * 32; w0 < run; w0 += 32 * wpc) {
                const int wi = w0 + lane;
                const int at = want - (wi >= words ? 1 : 0) - (wi >= 2 * words ? 1 : 0);
                const unsigned m = wi < run ? __vcmpeq4(__ldg(code + min(wi, run - 1)), (unsigned)at * 0x01010101u) : 0u;
                if (have + 128 > SLIC_LIST) drain();
#pragma unroll
                for (int y = 0; y < 4; y++) {
                    const bool hit = (m >> (8 * y)) & 1u;
                    const unsigned bal = __ballot_sync(0xffffffffu, hit);
                    if (hit) list[wid][have + __popc(bal & lt)] = first + 4 * wi + y;
                    have += __popc(bal);
                }
            }
        }
        drain();
#pragma unroll
        for (int q = 0; q < 6; q++) sum[q] = warp_sum64(sum[q]);
    }
    if (lane < 6) {
        long long v = 0;
#pragma unroll
        for (int q = 0; q < 6; q++) v = lane == q ? sum[q] : v;
        tot[wid][lane] = v;
    }
    __syncthreads();
    // the means, one lane per centre of the CTA: FP64 is taken once for all of
    // them (its pipe is 16 times narrower than FP32's)
    const int per = SLIC_WARPS / wpc, cl = blockIdx.x * per + lane;
    if (wid == 0 && lane < per && cl < s.GW * s.GH) {
        long long t[6];
        for (int q = 0; q < 6; q++) {
            t[q] = 0;
            for (int k = 0; k < wpc; k++) t[q] += tot[lane * wpc + k][q];
        }
        const float *cin = (parity ? s.centres2 : s.centres) + 5 * (long long)cl;
        float *o = (parity ? s.centres : s.centres2) + 5 * (long long)cl;
        if (t[5] > 0) {
            const double r = 1.0 / (double)t[5];
            for (int j = 0; j < 3; j++) o[j] = (float)((double)t[j] * r * (1.0 / SLIC_FIX));
            o[3] = (float)((double)t[3] * r);
            o[4] = (float)((double)t[4] * r);
        } else {
            for (int j = 0; j < 5; j++) o[j] = cin[j];
        }
    }
}

cudaError_t launch_slic(const SlicBatch &b, const float *const *centres_in, int iterations,
                        float *const *centres_out, cudaStream_t st)
{
    // warps per cell: one as long as that fills the chip (152 SMs, 32 warps
    // each), more for few or large cells while each warp keeps a step of 64 pixels
    int wpc = 1;
    while (wpc < SLIC_WARPS && b.max_stride > 64 * wpc &&
           (b.max_stride > 1024 * wpc || (long long)b.max_cells * b.n * wpc < 152 * 32))
        wpc *= 2;
    const int per_cta = SLIC_WARPS / wpc;
    const dim3 grid((b.max_cells + per_cta - 1) / per_cta, b.n);
    constexpr int threads = 32 * SLIC_WARPS;
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
        k_slic_assign<false><<<grid, threads, 0, st>>>(b, it & 1, wpc);
        k_slic_update<<<grid, threads, 0, st>>>(b, it & 1, wpc);
    }
    const int parity = iterations & 1;
    k_slic_assign<true><<<grid, threads, 0, st>>>(b, parity, wpc);
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
