// Stability-based depth fusion (Section III-D), one light field at a time.
//
// Every pixel of every view that carries a depth is lifted to a 3-D point and
// projected into each other view of its light field (nearest pixel, the
// refinement step's validity window); per (reference view, source view) the
// point of smallest depth wins a reference pixel through an integer atomicMin
// on the float bits (positive floats order as integers, so the result does
// not depend on the order of the atomics).  Then every reference pixel
// counts, for each of its depth candidates (its own depth and one per other
// view), the candidates agreeing within tau (relative) minus those that do
// not, and keeps the closest candidate whose count is not negative.
//
// Layout: the reference views are taken in groups whose z-buffers fit
// FUSE_GROUP_BYTES together.  zbuf holds, per reference view r of a group,
// (V_l - 1) planes of its pixel count (source slot = i, or i - 1 past r), +inf
// bits where no point landed; select leaves the planes at +inf again, so they
// are cleared once, when they are allocated, and not by a pass of their own
// per call (131 of 683 us on 9 views of 1280x720).  The per-pair projection is
// x_r ~ d M (x, y, 1) + e with M = K_r R_r R_i^T K_i^-1 and e = K_r (t_r - R_r
// R_i^T t_i), composed in FP64 on the host and applied in FP32; row 3 of K is
// (0, 0, 1), so the third component is the camera-r depth.
#include "lfd_fuse.cuh"

namespace lfd {

__global__ void k_fuse_clear(uint4 *zbuf, long long n)
{
    const unsigned inf = 0x7f800000u;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        zbuf[k] = make_uint4(inf, inf, inf, inf);
}

cudaError_t launch_fuse_clear(unsigned *zbuf, size_t bytes, cudaStream_t st)
{
    k_fuse_clear<<<2048, 256, 0, st>>>((uint4 *)zbuf, (long long)(bytes / 16));
    return cudaGetLastError();
}

// One thread per source pixel (blocks of 64 x 4; blockIdx.z = source view i),
// projected into every reference of the group: depth and position serve them
// all, the group's projections are read from shared memory as broadcasts.
constexpr int FUSE_BX = 64, FUSE_BY = 4;

__global__ void __launch_bounds__(FUSE_BX * FUSE_BY) k_fuse_project(FuseArgs a, int first, int count)
{
    struct Proj {
        float4 x, y, z;                      // rows of M and e: X = d (x.x px + x.y py + x.z) + x.w
        unsigned *zbuf;
        int W, H;
    };
    __shared__ Proj proj[FUSE_MAX_GROUP];
    const int i = blockIdx.z;
    const int tid = threadIdx.y * FUSE_BX + threadIdx.x;
    if (tid < count) {
        const int r = first + tid;
        const float *m = a.mats + 12 * (i * a.V + r);
        Proj q;
        q.x = make_float4(m[0], m[1], m[2], m[9]);
        q.y = make_float4(m[3], m[4], m[5], m[10]);
        q.z = make_float4(m[6], m[7], m[8], m[11]);
        q.W = a.W[r];
        q.H = a.H[r];
        q.zbuf = r == i ? nullptr : a.zbuf + a.zoff[r] + (long long)(i < r ? i : i - 1) * q.W * q.H;
        proj[tid] = q;
    }
    __syncthreads();
    const int W = a.W[i], H = a.H[i];
    const int ix = blockIdx.x * FUSE_BX + threadIdx.x, iy = blockIdx.y * FUSE_BY + threadIdx.y;
    if (ix >= W || iy >= H) return;
    const float d = __ldg(a.depth_in[i] + (long long)iy * W + ix);
    if (!(d > 0.f) || !isfinite(d)) return;
    const float x = (float)ix, y = (float)iy;
    for (int k = 0; k < count; k++) {
        const Proj &q = proj[k];
        if (!q.zbuf) continue;               // its own reference
        const float X = fmaf(d, fmaf(q.x.x, x, fmaf(q.x.y, y, q.x.z)), q.x.w);
        const float Y = fmaf(d, fmaf(q.y.x, x, fmaf(q.y.y, y, q.y.z)), q.y.w);
        const float Z = fmaf(d, fmaf(q.z.x, x, fmaf(q.z.y, y, q.z.z)), q.z.w);
        if (!(Z > 0.f)) continue;
        const float rz = 1.0f / Z;
        const float u = X * rz, v = Y * rz;
        if (!(u >= 0.f && u <= (float)(q.W - 1) && v >= 0.f && v <= (float)(q.H - 1))) continue;
        // floor(u + 0.5) by adding 1.5 * 2^23 towards -inf: exact below 2^22
        const int qx = __float_as_int(__fadd_rd(u + 0.5f, 12582912.f)) - 0x4B400000;
        const int qy = __float_as_int(__fadd_rd(v + 0.5f, 12582912.f)) - 0x4B400000;
        atomicMin(q.zbuf + (qy * q.W + qx), __float_as_uint(Z));
    }
}

// One thread per reference pixel; blockIdx.y = reference of the group.  The
// candidates (own depth, one per other view) stay in NC registers, NaN where
// there is none, so a missing one agrees with nothing.  With n candidates of
// which A (itself included) agree with z_c, its stability is 2 (A - 1) -
// (n - 1).  They are tried from the closest on: the first with stability >= 0
// is the answer, which is mostly the first tried, instead of scoring all n
// (9 views of 1280x720: 97 us including the clearing, 5.5 TB/s of z-buffer;
// 330 us with the candidates in a local array).
template <int NC>
__global__ void __launch_bounds__(256) k_fuse_select(FuseArgs a, int first)
{
    const int r = first + blockIdx.y;
    const int W = __ldg(a.W + r), H = __ldg(a.H + r);
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= W * H) return;
    const long long np = (long long)W * H;
    unsigned *z = a.zbuf + __ldg(a.zoff + r) + q;
    const float nan = __int_as_float(0x7fffffff), inf = __int_as_float(0x7f800000);
    const int ns = a.V - 1;
    float c[NC];
    const float own = __ldg(a.depth_in[r] + q);
    c[0] = own > 0.f && isfinite(own) ? own : nan;
    int n = c[0] > 0.f ? 1 : 0;
#pragma unroll
    for (int k = 0; k < NC - 1; k++) c[k + 1] = k < ns ? __uint_as_float(z[k * np]) : inf;
#pragma unroll
    for (int k = 0; k < NC - 1; k++) {
        if (c[k + 1] < inf) {
            z[k * np] = 0x7f800000u;
            n++;
        } else {
            c[k + 1] = nan;
        }
    }
    float zc = 0.f;
    for (;;) {
        float next = inf;                    // the closest candidate behind the last one tried
#pragma unroll
        for (int k = 0; k < NC; k++) next = c[k] > zc ? fminf(next, c[k]) : next;
        zc = next;
        if (!(zc < inf)) break;
        const float lim = a.tau * zc;
        int agree = 0;
#pragma unroll
        for (int k = 0; k < NC; k++) agree += fabsf(c[k] - zc) <= lim ? 1 : 0;
        if (2 * agree >= n + 1) break;
    }
    a.depth_out[r][q] = zc < inf ? zc : 0.f;
}

// many views: the candidates are re-read from the z-buffer (own depth is index -1)
__global__ void __launch_bounds__(256) k_fuse_select_many(FuseArgs a, int first)
{
    const int r = first + blockIdx.y;
    const int W = a.W[r], H = a.H[r];
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= W * H) return;
    const long long np = (long long)W * H;
    unsigned *z = a.zbuf + a.zoff[r] + q;
    const int ns = a.V - 1;
    const float own = __ldg(a.depth_in[r] + q);
    float best = 0.f;
    bool have = false;
    for (int s = -1; s < ns; s++) {
        const float zc = s < 0 ? own : __uint_as_float(z[s * np]);
        if (!(zc > 0.f) || !isfinite(zc)) continue;
        const float lim = a.tau * zc;
        int stab = 0;
        for (int b = -1; b < ns; b++) {
            if (b == s) continue;
            const float zb = b < 0 ? own : __uint_as_float(z[b * np]);
            if (!(zb > 0.f) || !isfinite(zb)) continue;
            stab += fabsf(zb - zc) <= lim ? 1 : -1;
        }
        if (stab >= 0 && (!have || zc < best)) {
            best = zc;
            have = true;
        }
    }
    for (int s = 0; s < ns; s++) z[s * np] = 0x7f800000u;
    a.depth_out[r][q] = have ? best : 0.f;
}

cudaError_t launch_fuse_group(const FuseArgs &a, int first, int count, int max_w, int max_h, int max_px,
                              cudaStream_t st)
{
    const unsigned blocks = (unsigned)((max_px + 255) / 256);
    k_fuse_project<<<dim3((max_w + FUSE_BX - 1) / FUSE_BX, (max_h + FUSE_BY - 1) / FUSE_BY, a.V),
                     dim3(FUSE_BX, FUSE_BY), 0, st>>>(a, first, count);
    const dim3 g(blocks, count);
    if (a.V <= 4) k_fuse_select<4><<<g, 256, 0, st>>>(a, first);
    else if (a.V <= 6) k_fuse_select<6><<<g, 256, 0, st>>>(a, first);
    else if (a.V <= 9) k_fuse_select<9><<<g, 256, 0, st>>>(a, first);
    else if (a.V <= 12) k_fuse_select<12><<<g, 256, 0, st>>>(a, first);
    else if (a.V <= 16) k_fuse_select<16><<<g, 256, 0, st>>>(a, first);
    else if (a.V <= 32) k_fuse_select<32><<<g, 256, 0, st>>>(a, first);
    else k_fuse_select_many<<<g, 256, 0, st>>>(a, first);
    return cudaGetLastError();
}

}  // namespace lfd
