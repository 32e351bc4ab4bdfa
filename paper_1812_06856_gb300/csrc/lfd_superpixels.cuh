// Step a1: launch entries of k_superpixels.cu, and the device code that it
// shares with the allocation-free statistics (k_noalloc.cu): pixel counts and
// bounding boxes of a label map, and the sums over a superpixel's pixels.
#pragma once
#include "lfd_internal.cuh"

namespace lfd {

// ---------------------------------------------------------------------------
// counts and bounding boxes
// ---------------------------------------------------------------------------
//
// A warp walks a strip of 32 columns x SP_STRIP rows.  While no lane's label
// changes from one row to the next, nothing is written; on a change (or the
// strip's end) the lanes form runs of equal labels, all of the same height,
// and each run's first lane adds it: one set of atomics per run and change
// instead of one per label and row (8 x 1024x768: 64 -> 12.6 us; MATCH and
// five atomics per 14 pixels before).
constexpr int SP_STRIP = 32;

__host__ __device__ inline int label_strips(int W, int H) { return ((W + 31) / 32) * ((H + SP_STRIP - 1) / SP_STRIP); }

// strip `strip` of a W x H label map: cnt[l] += pixels, bbox[l] = {min x, min
// y, max x, max y} over labels l in [0, S); returns a pixel whose label is
// outside that range (-1: none), per lane
__device__ __forceinline__ int label_runs(const int *labels, int W, int H, int S, int *cnt, int4 *bbox, int strip)
{
    const int lane = threadIdx.x & 31;
    const int across = (W + 31) / 32;
    const int x0 = (strip % across) * 32, y0 = (strip / across) * SP_STRIP;
    if (y0 >= H) return -1;                  // whole warp
    const int x = x0 + lane, y1 = min(y0 + SP_STRIP, H);
    int bad = -1, cur = -2, from = y0;       // cur: the lane's label since row `from`, -1 outside the range
    auto flush = [&](int to) {               // rows from .. to - 1
        const int left = __shfl_up_sync(0xffffffffu, cur, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || left != cur);
        if (((heads >> lane) & 1u) && cur >= 0) {
            const unsigned after = lane == 31 ? 0u : heads >> (lane + 1);
            const int len = after ? __ffs(after) : 32 - lane;
            atomicAdd(&cnt[cur], len * (to - from));
            atomicMin(&bbox[cur].x, x);
            atomicMin(&bbox[cur].y, from);
            atomicMax(&bbox[cur].z, x + len - 1);
            atomicMax(&bbox[cur].w, to - 1);
        }
    };
    for (int y = y0; y < y1; y += 4) {
        int l[4];
#pragma unroll
        for (int r = 0; r < 4; r++) l[r] = x < W && y + r < y1 ? __ldg(labels + (long long)(y + r) * W + x) : -1;
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (y + r >= y1) break;
            const bool ok = l[r] >= 0 && l[r] < S;
            if (x < W && !ok) bad = (y + r) * W + x;
            const int v = ok ? l[r] : -1;
            if (__any_sync(0xffffffffu, v != cur)) {
                if (cur != -2) flush(y + r);
                cur = v;
                from = y + r;
            }
        }
    }
    flush(y1);
    return bad;
}

// ---------------------------------------------------------------------------
// sums over a superpixel's pixels
// ---------------------------------------------------------------------------

// Coordinates and colours as exact integers where the format allows: RGBA8
// bytes, FP16 values below 64 in units of 2^-24 (every such half is a
// multiple); the rest in FP64.  FP64 runs at a sixteenth of the FP32 rate.
template <int FMT>
struct SuperpixelSums {
    long long x = 0, y = 0, qr = 0, qg = 0, qb = 0;
    double r = 0.0, g = 0.0, b = 0.0;

    __device__ __forceinline__ static void fixed(float v, long long &q, double &d)
    {
        if (fabsf(v) < 64.f) q += __float2int_rn(v * 16777216.f);
        else d += v;
    }
    __device__ __forceinline__ void pixel(int px, int py, const char *row)
    {
        x += px;
        y += py;
        if (FMT == LFD_RGBA8) {
            const uchar4 t = ((const uchar4 *)row)[px];
            qr += t.x; qg += t.y; qb += t.z;
        } else if (FMT == LFD_RGBA_F16) {
            const __half *t = (const __half *)row + 4 * px;
            fixed(__half2float(t[0]), qr, r);
            fixed(__half2float(t[1]), qg, g);
            fixed(__half2float(t[2]), qb, b);
        } else if (FMT == LFD_RGBA_BF16) {
            const __nv_bfloat16 *t = (const __nv_bfloat16 *)row + 4 * px;
            r += __bfloat162float(t[0]); g += __bfloat162float(t[1]); b += __bfloat162float(t[2]);
        } else {
            const float4 t = ((const float4 *)row)[px];
            r += t.x; g += t.y; b += t.z;
        }
    }
    __device__ __forceinline__ static long long wsum(long long v)
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    __device__ __forceinline__ static double wsum(double v)
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    // the warp's sums, in every lane
    __device__ __forceinline__ void reduce()
    {
        x = wsum(x);
        y = wsum(y);
        if (FMT == LFD_RGBA8 || FMT == LFD_RGBA_F16) { qr = wsum(qr); qg = wsum(qg); qb = wsum(qb); }
        if (FMT == LFD_RGBA_BF16 || FMT == LFD_RGBA_F32 ||
            (FMT == LFD_RGBA_F16 && __any_sync(0xffffffffu, !(r == 0.0 && g == 0.0 && b == 0.0)))) {
            r = wsum(r); g = wsum(g); b = wsum(b);
        }
    }
    __device__ __forceinline__ void add(const SuperpixelSums &o)
    {
        x += o.x; y += o.y; qr += o.qr; qg += o.qg; qb += o.qb;
        r += o.r; g += o.g; b += o.b;
    }
    // centroid and mean colour in [0,1] units of n pixels
    __device__ __forceinline__ void mean(int n, double &cx, double &cy, double &mr, double &mg, double &mb) const
    {
        const double unit = FMT == LFD_RGBA_F16 ? 1.0 / 16777216.0 : 1.0, sc = FMT == LFD_RGBA8 ? 1.0 / 255.0 : 1.0;
        cx = (double)x / n;
        cy = (double)y / n;
        mr = ((double)qr * unit + r) * sc / n;
        mg = ((double)qg * unit + g) * sc / n;
        mb = ((double)qb * unit + b) * sc / n;
    }
};

// The warp's scan of box bb (pixels i = first + lane, step 32 * step) of label
// s: sums into t and, with LIST, the pixels to pix in row-major order (at most
// cap).  Returns the pixels found, in every lane.
template <int FMT, bool LIST>
__device__ __forceinline__ int scan_box(const int *labels, const void *img, long long pitch, int W, int s, int4 bb,
                                        int first, int step, int lane, unsigned *pix, int cap,
                                        SuperpixelSums<FMT> &t)
{
    const int bw = bb.z - bb.x + 1;
    const int area = bw * (bb.w - bb.y + 1);             // below 2^30 (LFD_MAX_DIM)
    int found = 0;
    // position kept incrementally: 32 * step = adv_y rows and adv_x columns
    const int adv_y = 32 * step / bw, adv_x = 32 * step - adv_y * bw;
    const int i0 = first + lane;
    int y = bb.y + i0 / bw, x = bb.x + i0 % bw;
    constexpr int U = 4;
    for (int i = first; i < area; i += 32 * step * U) {
        int px[U], py[U];
        bool f[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            px[u] = x;
            py[u] = y;
            f[u] = y <= bb.w && __ldg(labels + (long long)y * W + x) == s;
            x += adv_x;
            y += adv_y;
            if (x > bb.z) {
                x -= bw;
                y++;
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const unsigned bal = __ballot_sync(0xffffffffu, f[u]);
            if (f[u]) {
                const int at = found + __popc(bal & ((1u << lane) - 1u));
                if (LIST && at < cap) pix[at] = ((unsigned)py[u] << 16) | (unsigned)px[u];
                t.pixel(px[u], py[u], (const char *)img + (long long)py[u] * pitch);
            }
            found += __popc(bal);
        }
    }
    return found;
}

// Superpixels per CTA of 8 warps, from their number and the pixels they share:
// a warp's each, unless large boxes are likely (2500 pixels on average).  Those
// go through the CTA one after another, so there a CTA takes as many as one wave
// of CTAs (152 SMs x 8) leaves to each.  Statistics of one view, us, eight per
// CTA and by this rule (a CTA of their own for all superpixels before): 640x480
// in cells of 60 x 60 118 and 74 (81), 150 x 150 286 and 78 (163), 24 labels
// scattered over the image 2489 and 662 (1018); below that the split only leaves
// warps idle (1920x1080 in cells of 46 x 46 84 and 96, 1280x720 of 16 x 16 41
// and 46).
inline int superpixels_per_cta(int S, long long px)
{
    if (px < 2500ll * S) return 8;
    const int per = (S + 152 * 8 - 1) / (152 * 8);
    return per < 1 ? 1 : (per > 8 ? 8 : per);
}

// ---------------------------------------------------------------------------
// launch entries
// ---------------------------------------------------------------------------

// counts, boxes and the view of every superpixel; max_strips: largest label_strips of the views
cudaError_t launch_sp_count(const Workspace &w, int V, int max_strips, int *cnt, int4 *bbox, int *sp_view,
                            cudaStream_t st);

// a work order: `order` receives the superpixels of `in` (NULL = index order)
// stably sorted by the key of `mode` (0 propagation: pixel-slot class, band; 1
// sweep: power-of-two size class, band; 2: sweep class).  hist: scratch of
// ORDER_KEYS * order_tiles(S_total) ints (at most 2.2 S_total), unused for a
// single tile
constexpr int ORDER_TILE = 1024;
static_assert(ORDER_KEYS <= ORDER_TILE, "k_order_small scans a key per thread");
__host__ __device__ inline int order_tiles(int S_total) { return (S_total + ORDER_TILE - 1) / ORDER_TILE; }
int order_kernels(int S_total);              // kernels a launch_sp_orders enqueues
struct SuperpixelOrder {
    int *order, *hist;
    const int *in;
    int mode;
};
// n <= 2 orders in the same launches
cudaError_t launch_sp_orders(const Workspace &w, int n, const SuperpixelOrder *o, int bands, cudaStream_t st);

}  // namespace lfd
