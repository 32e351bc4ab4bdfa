// Step a1: superpixel pixel lists (CSR) and statistics, and the per-view
// bilinear sampling textures.
//
// Section III-A: each view is over-segmented into compact superpixels laid out
// as a regular grid with an 8-neighbour system; each superpixel's plane is
// anchored at its centroid and its colour is the mean colour of its pixels
// (Section III-C1).  Eq. 11 needs the minimum colour similarity to the
// neighbours, which is fixed per superpixel and computed here once.
//
// The pixel lists are built without sorting and without atomics on the list
// itself: one warp per superpixel (a CTA for large ones) scans the
// superpixel's bounding box in row-major order and compacts the matching
// pixels by ballots, so the list order (row-major) and every sum are
// deterministic.  The cost is the sum of bounding-box areas, about the image
// area for compact superpixels.
#include "lfd_superpixels.cuh"

namespace lfd {

// ---------------------------------------------------------------------------
// 1. counts and bounding boxes (label_runs, lfd_superpixels.cuh)
// ---------------------------------------------------------------------------

// blockIdx.y = view; one warp per strip of 32 columns x SP_STRIP rows
__global__ void __launch_bounds__(256) k_sp_count(Workspace w, int *cnt, int4 *bbox)
{
    const int v = blockIdx.y;
    const ViewDev &vd = w.views[v];
    const int bad = label_runs(vd.labels, vd.W, vd.H, vd.S, cnt + vd.sp_base, bbox + vd.sp_base,
                               blockIdx.x * 8 + (threadIdx.x >> 5));
    if (bad >= 0 && atomicOr(&w.ctr->status, DEV_ERR_LABEL) == 0) {
        w.ctr->bad_view = v;
        w.ctr->bad_index = bad;
    }
}

// per superpixel: empty count and box, and its view (the last one whose first
// superpixel is not behind it)
__global__ void k_sp_init(Workspace w, int V, int *cnt, int4 *bbox, int *sp_view)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= w.S_total) return;
    cnt[i] = 0;
    bbox[i] = make_int4(0x7fffffff, 0x7fffffff, -1, -1);
    int lo = 0, hi = V - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (w.views[mid].sp_base <= i) lo = mid;
        else hi = mid - 1;
    }
    sp_view[i] = lo;
}

cudaError_t launch_sp_count(const Workspace &w, int V, int max_strips, int *cnt, int4 *bbox, int *sp_view,
                            cudaStream_t st)
{
    k_sp_init<<<(w.S_total + 255) / 256, 256, 0, st>>>(w, V, cnt, bbox, sp_view);
    k_sp_count<<<dim3((max_strips + 7) / 8, V), 256, 0, st>>>(w, cnt, bbox);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 2. exclusive scan of the counts of each view -> global list offsets
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(1024) k_sp_scan(Workspace w, int V, const int *cnt, int *off)
{
    const int v = blockIdx.x;
    const ViewDev &vd = w.views[v];
    __shared__ int warp_tot[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = (int)vd.px_base;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int base = 0; base < vd.S; base += 1024) {
        const int s = base + threadIdx.x;
        const int c = s < vd.S ? cnt[vd.sp_base + s] : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_tot[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int t = warp_tot[lane];
            int ti = t;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int u = __shfl_up_sync(0xffffffffu, ti, o);
                if (lane >= o) ti += u;
            }
            warp_tot[lane] = ti - t;   // exclusive prefix of warp totals
        }
        __syncthreads();
        const int excl = carry + warp_tot[wid] + incl - c;
        if (s < vd.S) off[vd.sp_base + s] = excl;
        __syncthreads();
        if (threadIdx.x == 1023) carry = excl + c;
        __syncthreads();
    }
    if (v == V - 1 && threadIdx.x == 0) off[w.S_total] = carry;
}

cudaError_t launch_sp_scan(const Workspace &w, int V, const int *cnt, int *off, cudaStream_t st)
{
    k_sp_scan<<<V, 1024, 0, st>>>(w, V, cnt, off);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 3. ordered compaction of each superpixel's pixels + centroid and colour sums
// ---------------------------------------------------------------------------

// One warp per superpixel; a superpixel whose box exceeds SP_WARP_AREA pixels
// is left to a second pass of whole CTAs over the same grid.
//
// 8 x 1024x768 RGBA8 (32120 superpixels of 14 x 14): 590 -> 63 us; one CTA of
// 256 threads per superpixel spent its time in five block-wide trees of FP64
// and 64-bit sums.  Latency-bound (label, then texel); the lists, labels and
// texels are 38 MB, 6 us at the HBM rate.
constexpr int SP_WARP_AREA = 4096;

template <int FMT>
__global__ void __launch_bounds__(256) k_sp_collect(Workspace w, int per, const int4 *bbox, const int *cnt,
                                                    unsigned *pix, double2 *cen, int2 *ref, float4 *col)
{
    __shared__ SuperpixelSums<FMT> part[8];
    __shared__ int wcnt[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto finish = [&](int gs, const SuperpixelSums<FMT> &t, int n) {     // one lane
        double cx, cy, r, g, b;
        t.mean(n, cx, cy, r, g, b);
        cen[gs] = make_double2(cx, cy);
        ref[gs] = make_int2(__double2int_rn(cx), __double2int_rn(cy));
        col[gs] = make_float4((float)r, (float)g, (float)b, 1.0f);
    };
    const int gs0 = blockIdx.x * per, gs = gs0 + wid;
    bool large = false;
    if (wid < per && gs < w.S_total) {
        const int n = cnt[gs];
        if (n == 0) {
            if (lane == 0) {
                cen[gs] = make_double2(0.0, 0.0);
                ref[gs] = make_int2(0, 0);
                col[gs] = make_float4(0.f, 0.f, 0.f, 1.f);
            }
        } else {
            const int4 bb = bbox[gs];
            large = (long long)(bb.z - bb.x + 1) * (bb.w - bb.y + 1) > SP_WARP_AREA;
            if (!large) {
                const ViewDev &vd = w.views[__ldg(w.sp_view + gs)];
                SuperpixelSums<FMT> t;
                const int got = scan_box<FMT, true>(vd.labels, vd.img, vd.pitch, vd.W, gs - vd.sp_base, bb, 0, 1, lane,
                                                    pix + w.sp_off[gs], n, t);
                t.reduce();
                if (lane == 0) {
                    part[wid] = t;
                    if (got != n && atomicOr(&w.ctr->status, DEV_ERR_COUNT) == 0) {
                        w.ctr->bad_view = __ldg(w.sp_view + gs);
                        w.ctr->bad_index = gs - vd.sp_base;
                    }
                }
            }
        }
        if (lane == 0) wcnt[wid] = large ? -1 : n;
    } else if (lane == 0) {
        wcnt[wid] = 0;
    }
    const bool any_large = __syncthreads_or(large);
    // the warps' means, one lane each: FP64 divisions once per CTA
    if (threadIdx.x < 8 && wcnt[threadIdx.x] > 0) finish(gs0 + threadIdx.x, part[threadIdx.x], wcnt[threadIdx.x]);
    if (!any_large) return;
    for (int k = 0; k < per; k++) {
        __syncthreads();
        if (wcnt[k] >= 0) continue;          // uniform
        const int g = gs0 + k, n = cnt[g], v = __ldg(w.sp_view + g);
        const ViewDev &vd = w.views[v];
        const int s = g - vd.sp_base;
        const int4 bb = bbox[g];
        // rows of the box split between the warps; a warp's place in the list follows from the warps before it
        const int rows = bb.w - bb.y + 1, per = (rows + 7) / 8;
        const int4 mine = make_int4(bb.x, min(bb.y + wid * per, bb.w + 1), bb.z, min(bb.y + (wid + 1) * per - 1, bb.w));
        __shared__ int start[9];
        SuperpixelSums<FMT> t;
        const int got = mine.w < mine.y ? 0 : scan_box<FMT, false>(vd.labels, vd.img, vd.pitch, vd.W, s, mine, 0, 1,
                                                                   lane, nullptr, 0, t);
        if (lane == 0) start[wid + 1] = got;
        __syncthreads();
        int before = 0, total = 0;
        for (int q = 0; q < 8; q++) {
            before += q < wid ? start[q + 1] : 0;
            total += start[q + 1];
        }
        if (mine.w >= mine.y && before < n) {
            SuperpixelSums<FMT> dummy;
            scan_box<FMT, true>(vd.labels, vd.img, vd.pitch, vd.W, s, mine, 0, 1, lane, pix + w.sp_off[g] + before,
                                n - before, dummy);
        }
        t.reduce();
        if (lane == 0) part[wid] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < 8; q++) part[0].add(part[q]);
            if (total != n && atomicOr(&w.ctr->status, DEV_ERR_COUNT) == 0) {
                w.ctr->bad_view = v;
                w.ctr->bad_index = s;
            }
            finish(g, part[0], n);
        }
    }
}

cudaError_t launch_sp_collect(const Workspace &w, const Consts &c, const int4 *bbox, const int *cnt, unsigned *pix,
                              double2 *cen, int2 *ref, float4 *col, cudaStream_t st)
{
    const int per = superpixels_per_cta(w.S_total, w.px_total), blocks = (w.S_total + per - 1) / per;
    switch (c.fmt) {
    case LFD_RGBA8: k_sp_collect<LFD_RGBA8><<<blocks, 256, 0, st>>>(w, per, bbox, cnt, pix, cen, ref, col); break;
    case LFD_RGBA_F16: k_sp_collect<LFD_RGBA_F16><<<blocks, 256, 0, st>>>(w, per, bbox, cnt, pix, cen, ref, col); break;
    case LFD_RGBA_BF16: k_sp_collect<LFD_RGBA_BF16><<<blocks, 256, 0, st>>>(w, per, bbox, cnt, pix, cen, ref, col); break;
    default: k_sp_collect<LFD_RGBA_F32><<<blocks, 256, 0, st>>>(w, per, bbox, cnt, pix, cen, ref, col); break;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 4. minimum colour similarity to the present 8-neighbours (Eq. 11)
// ---------------------------------------------------------------------------

__global__ void k_sp_minw(Workspace w, Consts c, float4 *col)
{
    const int gs = blockIdx.x * blockDim.x + threadIdx.x;
    if (gs >= w.S_total) return;
    const int v = w.sp_view[gs];
    const ViewDev &vd = w.views[v];
    const int s = gs - vd.sp_base;
    const int gx = s % vd.GW, gy = s / vd.GW;
    const float4 cs = col[gs];
    const double k_col = vd.k_col;   // log2(e) / (2 alpha^2): omega = 2^(-|dC|^2 k_col)
    // the smallest similarity 2^-x is that of the largest x: one exponential
    // instead of eight (FP64; 8 x 1024x768: 18.6 -> 10 us)
    double far = 0.0;
    bool any = false;
    for (int d = 0; d < 8; d++) {
        int dx, dy;
        ring_dir(d, dx, dy);
        const int x = gx + dx, y = gy + dy;
        if (x < 0 || y < 0 || x >= vd.GW || y >= vd.GH) continue;
        const int j = vd.sp_base + y * vd.GW + x;
        if (w.sp_cnt[j] == 0) continue;
        const float4 cj = col[j];
        const double dr = (double)cj.x - cs.x, dg = (double)cj.y - cs.y, db = (double)cj.z - cs.z;
        const double q = (dr * dr + dg * dg + db * db) * k_col;
        if (!any || q > far) far = q;
        any = true;
    }
    col[gs].w = (float)(any ? exp2(-far) : 1.0);
}

cudaError_t launch_sp_minw(const Workspace &w, const Consts &c, float4 *col, cudaStream_t st)
{
    k_sp_minw<<<(w.S_total + 127) / 128, 128, 0, st>>>(w, c, col);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 5. sampling textures: per pixel the 2x2 bilinear footprint in one record
// ---------------------------------------------------------------------------
//   RGBA8, F16, BF16: red/green of t00, t10, t01, t11 as     24 B / pixel
//          four 16-bit pairs (16-B records for all entries), then
//          blue of (t00, t01), (t10, t11) as two pairs (8-B records);
//          RGBA8 bytes are stored as exact halves
//   F32: 3 x float4 RGB of t00, t10, t01, t11                48 B / pixel
//   (W + 1) x (H + 1) entries per view, see k_quads

__device__ __forceinline__ unsigned pack_h2(float lo, float hi)
{
    __half2 h = __floats2half2_rn(lo, hi);   // small integers: exact
    return *reinterpret_cast<unsigned *>(&h);
}

// The texture has a border of one quad on the left and top: entry
// (y + 1) (W + 1) + (x + 1) holds the quad of pixel (x, y) for x in [-1, W-1],
// y in [-1, H-1], every texel index clamped to the image.  A bilinear sample
// anywhere in the texture area -1/2 <= x < W - 1/2 then reads the quad at
// floor(x) with no clamping of the coordinates: where a texel is clamped its
// difference to the neighbour is 0, which gives clamp-to-edge exactly.
__global__ void __launch_bounds__(256) k_quads(Workspace w, int fmt)
{
    const int v = blockIdx.y;
    const ViewDev &vd = w.views[v];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int Wp = vd.W + 1;
    if (p >= Wp * (vd.H + 1)) return;
    const int qx = p % Wp - 1, qy = p / Wp - 1;
    const int x = max(qx, 0), y = max(qy, 0);
    const int x1 = min(qx + 1, vd.W - 1), y1 = min(qy + 1, vd.H - 1);
    const char *base = (const char *)vd.img;
    const long long pitch = vd.pitch;
    const char *r0 = base + (long long)y * pitch;
    const char *r1 = base + (long long)y1 * pitch;
    if (fmt == LFD_RGBA8) {
        // the byte texels as halves (0..255 exact) in the FP16 layout below
        const uchar4 *a = (const uchar4 *)r0, *b = (const uchar4 *)r1;
        const uchar4 t00 = a[x], t10 = a[x1], t01 = b[x], t11 = b[x1];
        const long long npx = (long long)Wp * (vd.H + 1);
        ((uint4 *)vd.quad)[p] = make_uint4(pack_h2(t00.x, t00.y), pack_h2(t10.x, t10.y), pack_h2(t01.x, t01.y),
                                           pack_h2(t11.x, t11.y));
        ((uint2 *)((uint4 *)vd.quad + npx))[p] = make_uint2(pack_h2(t00.z, t01.z), pack_h2(t10.z, t11.z));
    } else if (fmt == LFD_RGBA_F16 || fmt == LFD_RGBA_BF16) {
        // a texel is {red|green, blue|alpha} as two 16-bit pairs
        const uint2 *a = (const uint2 *)r0, *b = (const uint2 *)r1;
        const uint2 t00 = a[x], t10 = a[x1], t01 = b[x], t11 = b[x1];
        const long long npx = (long long)Wp * (vd.H + 1);
        ((uint4 *)vd.quad)[p] = make_uint4(t00.x, t10.x, t01.x, t11.x);
        ((uint2 *)((uint4 *)vd.quad + npx))[p] =
            make_uint2((t00.y & 0xffffu) | (t01.y << 16), (t10.y & 0xffffu) | (t11.y << 16));
    } else {
        const float4 *a = (const float4 *)r0, *b = (const float4 *)r1;
        const float4 t00 = a[x], t10 = a[x1], t01 = b[x], t11 = b[x1];
        float4 *q = (float4 *)vd.quad + 3 * (long long)p;
        q[0] = make_float4(t00.x, t00.y, t00.z, t10.x);
        q[1] = make_float4(t10.y, t10.z, t01.x, t01.y);
        q[2] = make_float4(t01.z, t11.x, t11.y, t11.z);
    }
}

cudaError_t launch_quads(const Workspace &w, int V, int max_px, int fmt, cudaStream_t st)
{
    dim3 grid((max_px + 255) / 256, V);       // max_px: largest (W + 1) (H + 1) of the views
    k_quads<<<grid, 256, 0, st>>>(w, fmt);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 6. work orders of the persistent launches: a stable counting sort of all
//    superpixels by size class, largest first, index order inside a class.
//    Propagation (mode 0) uses pixel-slot classes ceil(n/32), capped at 16:
//    superpixels of one class run the same compiled evaluation, so the warps
//    resident on an SM at any time execute one code body (measured on the
//    8-view 1024x768 case: 23.3 ms per frame in this order, 47 ms with the
//    classes sorted per view, 53 ms in plain index order, from
//    instruction-fetch stalls).  The sweep (mode 1) has one code body and
//    uses coarser power-of-two classes floor(log2 n): expensive superpixels
//    still go first, while superpixels of similar size keep index order, so
//    concurrently swept superpixels are neighbours and share L2 lines (slot
//    classes there interleaved 14- and 15-pixel grid cells across all views
//    and read 6x more DRAM).  Deterministic.
// ---------------------------------------------------------------------------

//    Inside a class the superpixels go by row band (up to ORDER_BANDS
//    bands of each view's grid rows, a launch-shape option) and then in
//    index order: the superpixels in flight at any time cover the same rows
//    of every view, so the rows of the sampling textures and rasterised maps
//    they gather from (their own band, shifted by the disparity, in each
//    neighbour view) stay in L2 together instead of spanning whole views.
//    The sweep's order is finally partitioned, stably, by sweep class (mode
//    2: the label-count class of each superpixel's light field and the pair
//    form of its view): one sweep launch per class, its CTAs as wide as the
//    class's label count, compiled for the class's pair form.

__device__ __forceinline__ int order_key(const Workspace &w, int gs, int mode, int bands)
{
    if (mode == 2) return w.views[__ldg(w.sp_view + gs)].sclass;
    const int n = __ldg(w.sp_cnt + gs);
    const int cls = mode == 0 ? (n + 31) >> 5 : 31 - __clz(max(n, 1));
    const ViewDev &vd = w.views[__ldg(w.sp_view + gs)];
    const int gy = (gs - vd.sp_base) / vd.GW;
    const int band = min(bands - 1, (int)(((long long)gy * bands) / vd.GH));
    return (ORDER_CLASSES - 1 - min(cls, ORDER_CLASSES - 1)) * ORDER_BANDS + band;   // 0 = largest class, top band
}

// Three launches: per tile of ORDER_TILE superpixels a histogram of the keys
// (hist[key][tile]), one exclusive scan of it (key-major: the tile's first
// slot of each key), and the scatter, where a superpixel's slot is its tile's
// start of the key + the count of equal keys before it in the tile.  Both
// orders go through the same launches (blockIdx.y): 13 us on 8 x 1024x768,
// where a walk of one CTA over all tiles took 75 us per order.
struct OrderJob {
    int *order;
    int *hist;
    const int *in;
    int mode;
};

struct OrderJobs {
    OrderJob j[2];
};

__global__ void __launch_bounds__(ORDER_TILE) k_order_hist(Workspace w, const __grid_constant__ OrderJobs jobs,
                                                           int tiles, int bands)
{
    const OrderJob &q = jobs.j[blockIdx.y];
    __shared__ int h[ORDER_KEYS];
    for (int k = threadIdx.x; k < ORDER_KEYS; k += ORDER_TILE) h[k] = 0;
    __syncthreads();
    const int i = blockIdx.x * ORDER_TILE + threadIdx.x;
    if (i < w.S_total) atomicAdd(&h[order_key(w, q.in ? __ldg(q.in + i) : i, q.mode, bands)], 1);
    __syncthreads();
    for (int k = threadIdx.x; k < ORDER_KEYS; k += ORDER_TILE) q.hist[k * tiles + blockIdx.x] = h[k];
}

// exclusive scan of ORDER_KEYS * tiles counts by one CTA, a contiguous run per thread
__global__ void __launch_bounds__(1024) k_order_scan(const __grid_constant__ OrderJobs jobs, int tiles)
{
    int *hist = jobs.j[blockIdx.y].hist;
    __shared__ int warp_tot[32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int total = ORDER_KEYS * tiles, per = (total + 1023) / 1024, first = t * per, last = min(first + per, total);
    int sum = 0;
    for (int i = first; i < last; i++) sum += hist[i];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int x = warp_tot[lane];
        int y = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
        warp_tot[lane] = y - x;
    }
    __syncthreads();
    int run = warp_tot[wid] + incl - sum;
    for (int i = first; i < last; i++) {
        const int x = hist[i];
        hist[i] = run;
        run += x;
    }
}

__global__ void __launch_bounds__(ORDER_TILE) k_order_scatter(Workspace w, const __grid_constant__ OrderJobs jobs,
                                                              int tiles, int bands)
{
    const OrderJob &q = jobs.j[blockIdx.y];
    __shared__ unsigned short wcnt[ORDER_TILE / 32][ORDER_KEYS];     // per-warp counts of the tile
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int i = t; i < (ORDER_TILE / 32) * ORDER_KEYS / 2; i += ORDER_TILE) ((unsigned *)wcnt)[i] = 0u;
    __syncthreads();
    const int pos = blockIdx.x * ORDER_TILE + t;
    const bool ok = pos < w.S_total;
    const int gs = ok ? (q.in ? __ldg(q.in + pos) : pos) : 0;
    const int key = ok ? order_key(w, gs, q.mode, bands) : ORDER_KEYS;   // out-of-range lanes: a key of their own
    const unsigned same = __match_any_sync(0xffffffffu, key);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (ok && rank == 0) wcnt[wid][key] = (unsigned short)__popc(same);
    __syncthreads();
    if (!ok) return;
    int before = 0;
    for (int u = 0; u < wid; u++) before += wcnt[u][key];
    q.order[q.hist[key * tiles + blockIdx.x] + before + rank] = gs;
}

// up to one tile of superpixels: the whole sort in one CTA per order
__global__ void __launch_bounds__(ORDER_TILE) k_order_small(Workspace w, const __grid_constant__ OrderJobs jobs,
                                                            int bands)
{
    const OrderJob &q = jobs.j[blockIdx.y];
    __shared__ unsigned short wcnt[ORDER_TILE / 32][ORDER_KEYS];
    __shared__ int start[ORDER_TILE];
    __shared__ int warp_tot[ORDER_TILE / 32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int i = t; i < (ORDER_TILE / 32) * ORDER_KEYS / 2; i += ORDER_TILE) ((unsigned *)wcnt)[i] = 0u;
    __syncthreads();
    const bool ok = t < w.S_total;
    const int gs = ok ? (q.in ? __ldg(q.in + t) : t) : 0;
    const int key = ok ? order_key(w, gs, q.mode, bands) : ORDER_KEYS;
    const unsigned same = __match_any_sync(0xffffffffu, key);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (ok && rank == 0) wcnt[wid][key] = (unsigned short)__popc(same);
    __syncthreads();
    // exclusive scan of the keys' totals, thread t = key t
    int total = 0;
    if (t < ORDER_KEYS)
        for (int u = 0; u < ORDER_TILE / 32; u++) total += wcnt[u][t];
    int incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    int before = 0;
    for (int u = 0; u < wid; u++) before += warp_tot[u];
    start[t] = before + incl - total;
    __syncthreads();
    if (!ok) return;
    before = start[key];
    for (int u = 0; u < wid; u++) before += wcnt[u][key];
    q.order[before + rank] = gs;
}

int order_kernels(int S_total) { return order_tiles(S_total) > 1 ? 3 : 1; }

cudaError_t launch_sp_orders(const Workspace &w, int n, const SuperpixelOrder *o, int bands, cudaStream_t st)
{
    bands = max(1, min(bands, ORDER_BANDS));
    const int tiles = order_tiles(w.S_total);
    OrderJobs jobs = {};
    for (int k = 0; k < n; k++) jobs.j[k] = {o[k].order, o[k].hist, o[k].in, o[k].mode};
    if (tiles <= 1) {
        k_order_small<<<dim3(1, n), ORDER_TILE, 0, st>>>(w, jobs, bands);
        return cudaGetLastError();
    }
    k_order_hist<<<dim3(tiles, n), ORDER_TILE, 0, st>>>(w, jobs, tiles, bands);
    k_order_scan<<<dim3(1, n), 1024, 0, st>>>(jobs, tiles);
    k_order_scatter<<<dim3(tiles, n), ORDER_TILE, 0, st>>>(w, jobs, tiles, bands);
    return cudaGetLastError();
}

}  // namespace lfd
