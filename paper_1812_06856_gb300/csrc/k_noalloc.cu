// lfd_superpixel_stats_noalloc: the superpixel statistics of one view (the
// per-label counts, centroids, mean colours and minimum neighbour colour
// similarity that lfd_set_input builds) computed without allocating any
// memory.
//
// Some callers cannot allocate device memory on the path where they need
// these statistics: code running inside a CUDA graph being captured (stream
// capture forbids cudaMalloc/cudaFree), real-time or embedded loops that have
// a fixed memory plan and may not touch the allocator once started, and hosts
// whose allocator is owned by another framework.  This entry point therefore
// takes only caller-provided inputs and outputs; its scratch (per-label pixel
// counts and bounding boxes) lives in a file-scope device array of a fixed
// size that exists for as long as the library is loaded.
//
// Limits and sharing rules:
//  - at most LFD_NOALLOC_MAX_LABELS (65536) labels per call (grid_w*grid_h);
//  - the scratch array is shared by every call on a device and keeps the last
//    call's contents; each call clears the part it uses first;
//  - calls whose GPU work overlaps (different streams, or different host
//    threads without ordering) race on the scratch array and give wrong
//    results: serialise them;
//  - the first call on each device looks up the array's device address
//    (cudaGetSymbolAddress) with that device current; make that first call
//    before any stream capture.
#include <mutex>

#include "lfd_superpixels.cuh"

namespace {

constexpr int NOALLOC_MAX_LABELS = LFD_NOALLOC_MAX_LABELS;
constexpr int NOALLOC_MAX_DEVICES = 64;

struct NoallocScratch {
    int cnt[NOALLOC_MAX_LABELS];
    int4 bbox[NOALLOC_MAX_LABELS];
};

// 1.25 MiB per device, held while the library is loaded
static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

std::mutex g_noalloc_mutex;
NoallocScratch *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

__global__ void k_na_clear(NoallocScratch *sc, int S)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S) {
        sc->cnt[i] = 0;
        sc->bbox[i] = make_int4(0x7fffffff, 0x7fffffff, -1, -1);
    }
}

__global__ void __launch_bounds__(256) k_na_count(NoallocScratch *sc, const int *labels, int W, int H, int S)
{
    // labels outside the grid are ignored
    lfd::label_runs(labels, W, H, S, sc->cnt, sc->bbox, blockIdx.x * 8 + (threadIdx.x >> 5));
}

// One warp per label (8 per CTA at most) sums over the label's bounding box, a large
// box (more than NA_WARP_AREA pixels) is summed by the whole CTA; the means by
// one lane each.  1280x720 FP16, 3600 labels: 72 -> 21 us (a CTA per label and
// its block-wide FP64 trees before); latency-bound.
constexpr int NA_WARP_AREA = 4096;

template <int FMT>
__global__ void __launch_bounds__(256) k_na_stats(const NoallocScratch *sc, const int *labels, const void *img,
                                                  long long pitch, int W, int S, int per, float *stats)
{
    __shared__ lfd::SuperpixelSums<FMT> part[8];
    __shared__ int wcnt[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int s0 = blockIdx.x * per, s = s0 + wid;
    const int n = wid < per && s < S ? sc->cnt[s] : -1;
    bool large = false;
    if (n > 0) {
        const int4 bb = sc->bbox[s];
        large = (long long)(bb.z - bb.x + 1) * (bb.w - bb.y + 1) > NA_WARP_AREA;
        if (!large) {
            lfd::SuperpixelSums<FMT> t;
            lfd::scan_box<FMT, false>(labels, img, pitch, W, s, bb, 0, 1, lane, nullptr, 0, t);
            t.reduce();
            if (lane == 0) part[wid] = t;
        }
    }
    if (lane == 0) wcnt[wid] = large ? -n : n;
    const bool any_large = __syncthreads_or(large);
    auto write = [&](int l, int cnt, const lfd::SuperpixelSums<FMT> &t) {
        float *out = stats + 8 * (long long)l;
        if (cnt == 0) {   // as the regular path: centroid and colour 0, minw filled in by k_na_minw
            for (int k = 0; k < 8; k++) out[k] = k == 5 ? 1.f : 0.f;
            return;
        }
        double cx, cy, r, g, b;
        t.mean(cnt, cx, cy, r, g, b);
        out[0] = (float)cx;
        out[1] = (float)cy;
        out[2] = (float)r;
        out[3] = (float)g;
        out[4] = (float)b;
        out[5] = 1.f;
        out[6] = (float)cnt;
        out[7] = 0.f;
    };
    if (threadIdx.x < 8 && s0 + threadIdx.x < S && wcnt[threadIdx.x] >= 0)
        write(s0 + threadIdx.x, wcnt[threadIdx.x], part[threadIdx.x]);
    if (!any_large) return;
    for (int k = 0; k < per; k++) {
        __syncthreads();
        if (s0 + k >= S || wcnt[k] >= 0) continue;   // uniform
        lfd::SuperpixelSums<FMT> t;
        lfd::scan_box<FMT, false>(labels, img, pitch, W, s0 + k, sc->bbox[s0 + k], 32 * wid, 8, lane, nullptr, 0, t);
        t.reduce();
        if (lane == 0) part[wid] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < 8; q++) part[0].add(part[q]);
            write(s0 + k, -wcnt[k], part[0]);
        }
    }
}

// minimum colour similarity to the present (non-empty) 8-neighbours, from the
// colours just written; an empty label gets the value the regular path gives
// it (its colour is 0), so both report the same slot 5 for every label
__global__ void k_na_minw(float *stats, int GW, int GH, double k_col)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= GW * GH) return;
    const float *me = stats + 8 * (long long)s;
    const int gx = s % GW, gy = s / GW;
    const int dxs[8] = {1, 1, 0, -1, -1, -1, 0, 1}, dys[8] = {0, -1, -1, -1, 0, 1, 1, 1};
    double far = 0.0;    // the smallest similarity 2^-x is that of the largest x
    bool any = false;
    for (int d = 0; d < 8; d++) {
        const int x = gx + dxs[d], y = gy + dys[d];
        if (x < 0 || y < 0 || x >= GW || y >= GH) continue;
        const float *nb = stats + 8 * (long long)(y * GW + x);
        if (nb[6] == 0.f) continue;
        const double dr = (double)nb[2] - me[2], dg = (double)nb[3] - me[3], db = (double)nb[4] - me[4];
        const double q = (dr * dr + dg * dg + db * db) * k_col;
        if (!any || q > far) far = q;
        any = true;
    }
    // written into a separate slot first would need a second buffer; the
    // neighbours read only colours and counts (slots 2..4, 6), never slot 5
    stats[8 * (long long)s + 5] = (float)(any ? exp2(-far) : 1.0);
}

}  // namespace

extern "C" lfd_status lfd_superpixel_stats_noalloc(const int32_t *labels, const void *image, int32_t width,
                                                   int32_t height, int64_t pitch_bytes, int32_t fmt, int32_t grid_w,
                                                   int32_t grid_h, double alpha, float *stats_out, void *stream)
{
    int texel = fmt == LFD_RGBA8 ? 4 : (fmt == LFD_RGBA_F16 || fmt == LFD_RGBA_BF16) ? 8 : fmt == LFD_RGBA_F32 ? 16 : 0;
    if (!labels || !image || !stats_out || texel == 0) return LFD_ERR_INVALID_ARG;
    if (width < 1 || height < 1 || width > LFD_MAX_DIM || height > LFD_MAX_DIM || grid_w < 1 || grid_h < 1)
        return LFD_ERR_INVALID_ARG;
    if ((long long)grid_w * grid_h > NOALLOC_MAX_LABELS) return LFD_ERR_INVALID_ARG;   // beyond the scratch size
    const long long pitch = pitch_bytes ? pitch_bytes : (long long)width * texel;
    if (pitch < (long long)width * texel || pitch % texel || !(alpha > 0)) return LFD_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
        cudaGetLastError();
        return LFD_ERR_CUDA;
    }
    NoallocScratch *sc = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return LFD_ERR_CUDA;
            }
            g_noalloc_ptr[dev] = (NoallocScratch *)p;
        }
        sc = g_noalloc_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int S = grid_w * grid_h;
    const int strips = lfd::label_strips(width, height);
    // An error left pending on this thread by earlier, unrelated work is not
    // this call's: a launch of this call has failed only when the pending
    // error changes from what it was on entry.  (The earlier error stays
    // pending for its owner.)
    const cudaError_t before = cudaPeekAtLastError();
    auto launch_failed = [before]() {
        const cudaError_t e = cudaPeekAtLastError();
        return e != cudaSuccess && e != before;
    };
    const double log2e = 1.4426950408889634;
    k_na_clear<<<(S + 255) / 256, 256, 0, st>>>(sc, S);
    if (!launch_failed()) k_na_count<<<(strips + 7) / 8, 256, 0, st>>>(sc, labels, width, height, S);
    if (!launch_failed()) {
        const int per = lfd::superpixels_per_cta(S, (long long)width * height), blocks = (S + per - 1) / per;
        switch (fmt) {
        case LFD_RGBA8: k_na_stats<LFD_RGBA8><<<blocks, 256, 0, st>>>(sc, labels, image, pitch, width, S, per, stats_out); break;
        case LFD_RGBA_F16:
            k_na_stats<LFD_RGBA_F16><<<blocks, 256, 0, st>>>(sc, labels, image, pitch, width, S, per, stats_out);
            break;
        case LFD_RGBA_BF16:
            k_na_stats<LFD_RGBA_BF16><<<blocks, 256, 0, st>>>(sc, labels, image, pitch, width, S, per, stats_out);
            break;
        default: k_na_stats<LFD_RGBA_F32><<<blocks, 256, 0, st>>>(sc, labels, image, pitch, width, S, per, stats_out); break;
        }
    }
    if (!launch_failed())
        k_na_minw<<<(S + 127) / 128, 128, 0, st>>>(stats_out, grid_w, grid_h, log2e / (2.0 * alpha * alpha));
    if (launch_failed()) {
        if (before == cudaSuccess) cudaGetLastError();   // clear only what this call raised
        return LFD_ERR_CUDA;
    }
    return LFD_OK;
}
