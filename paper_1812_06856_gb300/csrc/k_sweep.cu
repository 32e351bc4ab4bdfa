// Steps a2-a4: partly randomised fronto-parallel plane sweep (Section III-B).
//
// For superpixel Omega of view v and label k the plane is fronto-parallel at
// inverse depth z_k = 1/d_max + (k + u_k) * delta with u_k uniform in [0,1)
// per superpixel and label (the jitter of Section III-B).  Its cost is
// Eq. 2's double sum over the neighbour views N(v) and the superpixel's
// pixels of the truncated SSD of Eq. 1, sampled bilinearly through the
// plane-induced homography; the lowest cost wins.
//
// Mapping: one CTA per superpixel, one thread per label.  The superpixel's
// pixels are staged in shared memory and read as broadcasts, so every thread
// walks the same pixel list while its own label shifts the projection along
// the epipolar line; neighbouring labels therefore gather from neighbouring
// texels (coalesced, L1-resident).  No reduction is needed per sample: each
// thread owns its label's cost; a single block arg-min ends the CTA.  This
// full sweep serves cost_out, world-frame sweeps, more than 256 labels, the
// non-persistent launch shape and sizes at which it is the faster one; the
// others take the bounded sweep below.
//
// Homography per (label, view): for the plane g = z_k * gh (gh = (0,0,1) for
// camera-frame sweeps) A = P + q g^T; its superpixel-anchored third column
// (P + q g^T) (ref,1) is composed in FP64 and rounded to FP32.  In the camera
// frame the rest, P (du, dv, 0) on the pixel's offset from the anchor, does not
// depend on the label: it is computed once per pixel and view of a chunk into
// shared memory and each sample adds the label's column (3 FP32 adds).  In the
// world frame the label also scales the pixel terms: 6 FP32 FMAs per sample.
#include <type_traits>

#include "lfd_bounds.cuh"
#include "lfd_sample.cuh"

namespace lfd {

constexpr int SWEEP_CHUNK = 128;

// Pair forms of the homography of a (view, neighbour view) pair, the kernels'
// template argument PF:
//   PF_GENERAL  any pair;
//   PF_AFFINE   P row 3 = (0, 0, P22) and q_z = 0 (parallel optical axes at
//               equal depth): the sample's homogeneous coordinate is the same
//               for every pixel of a label;
//   PF_SHIFT    affine with P's upper 2 x 2 block = P22 I as well (rectified
//               parallel cameras with equal intrinsics, e.g. a planar array):
//               a fronto-parallel plane moves every pixel by the same vector
//               (X0, Y0), so the integer part and the bilinear fractions are
//               per label and view, and a sample is an integer offset, a
//               window test on it and the gather.
constexpr int PF_GENERAL = 0, PF_AFFINE = 1, PF_SHIFT = 2;

struct SweepPair {
    float a00, a01, a10, a11, a20, a21;   // FP32 columns 0,1 of P (camera frame: not label dependent)
    int Wi, Hi;
    double pref[3];                       // P (ref,1) in FP64
    double q[3];
    double p0[3], p1[3];                  // columns 0,1 of P in FP64 (world-frame sweeps)
    double icw;                           // 1 / P (ref,1)_z (translation pairs: every label's w)
    const void *tex;
};

template <int THREADS, bool WORLD>
struct SweepShared {
    float2 d[SWEEP_CHUNK];
    float4 ref[SWEEP_CHUNK];
    // camera-frame sweeps: the label-independent part of each pixel's projection into
    // each neighbour view, P (du, dv, 0) (the label adds q z_k at the anchor)
    float4 xyw[WORLD ? 1 : LFD_MAXN][SWEEP_CHUNK];
    SweepPair pair[LFD_MAXN];
    double gh[4];                         // gh and gh.(ref,1)
    float n[3];                           // sweep plane normal (camera frame)
    float bc[THREADS / 32];
    int bk[THREADS / 32];
    int item;
};

// the whole sweep of superpixel gs by one CTA (threads = labels)
template <int FMT, bool WORLD, int THREADS, int PF>
__device__ __forceinline__ void sweep_sp(const Workspace &w, const Consts &c, int gs, SweepShared<THREADS, WORLD> &sh,
                                         float4 *planes, int *label_out, float *cost_out)
{
    const int v = __ldg(w.sp_view + gs);
    const ViewDev &vd = w.views[v];
    if (vd.sweep_skip) return;               // warm-started view: its planes are given
    const int s = gs - vd.sp_base;
    const int n = __ldg(w.sp_cnt + gs);
    if (n == 0) {
        if (threadIdx.x == 0) {
            planes[gs] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (label_out) label_out[gs] = -1;
        }
        return;
    }
    const int2 ref = __ldg(w.sp_ref + gs);
    const int nnb = vd.nnb;
    const int off = __ldg(w.sp_off + gs);
    const void *own_tex = vd.quad;
    const int L = vd.L;

    if (threadIdx.x == 0) {
        // sweep plane normal: fronto-parallel to the camera (gh = (0,0,1)) or to the
        // world z axis; gh = K^-T n / (n . K^-1 (c,1)) so that g = z * gh
        double gh0 = 0.0, gh1 = 0.0, gh2 = 1.0;
        if (WORLD) {
            const double2 cc = __ldg(w.sp_cen + gs);
            const double *Ki = vd.Kinv;
            double nn[3] = {vd.wz[0], vd.wz[1], vd.wz[2]};
            const double ray[3] = {Ki[0] * cc.x + Ki[1] * cc.y + Ki[2], Ki[3] * cc.x + Ki[4] * cc.y + Ki[5],
                                   Ki[6] * cc.x + Ki[7] * cc.y + Ki[8]};
            double nr = nn[0] * ray[0] + nn[1] * ray[1] + nn[2] * ray[2];
            if (nr > 0) { nn[0] = -nn[0]; nn[1] = -nn[1]; nn[2] = -nn[2]; nr = -nr; }
            gh0 = (Ki[0] * nn[0] + Ki[3] * nn[1] + Ki[6] * nn[2]) / nr;
            gh1 = (Ki[1] * nn[0] + Ki[4] * nn[1] + Ki[7] * nn[2]) / nr;
            gh2 = (Ki[2] * nn[0] + Ki[5] * nn[1] + Ki[8] * nn[2]) / nr;
            sh.n[0] = (float)nn[0]; sh.n[1] = (float)nn[1]; sh.n[2] = (float)nn[2];
        } else {
            sh.n[0] = 0.f; sh.n[1] = 0.f; sh.n[2] = -1.f;
        }
        sh.gh[0] = gh0; sh.gh[1] = gh1; sh.gh[2] = gh2;
        sh.gh[3] = gh0 * ref.x + gh1 * ref.y + gh2;
    }
    if (threadIdx.x < nnb) {
        const PairDev &pd = w.pairs[v * LFD_MAXN + threadIdx.x];
        SweepPair sp;
        sp.a00 = pd.Pf[0]; sp.a01 = pd.Pf[1];
        sp.a10 = pd.Pf[3]; sp.a11 = pd.Pf[4];
        sp.a20 = pd.Pf[6]; sp.a21 = pd.Pf[7];
        sp.Wi = pd.Wi; sp.Hi = pd.Hi;
        for (int r = 0; r < 3; r++) {
            sp.pref[r] = pd.P[3 * r] * ref.x + pd.P[3 * r + 1] * ref.y + pd.P[3 * r + 2];
            sp.q[r] = pd.q[r];
            sp.p0[r] = pd.P[3 * r];
            sp.p1[r] = pd.P[3 * r + 1];
        }
        sp.icw = sp.pref[2] > 0.0 ? 1.0 / sp.pref[2] : 0.0;
        sp.tex = pd.quad_i;
        sh.pair[threadIdx.x] = sp;
    }
    __syncthreads();

    const float T = vd.T;
    float best_cost = INFINITY;
    int best_k = 0x7fffffff;
    for (int k0 = 0; k0 < L; k0 += THREADS) {
        const int k = k0 + threadIdx.x;
        const bool active = k < L;
        const double u = vd.jitter ? jitter_u(vd.seed, vd.lf_index, vd.lv, s, active ? k : 0) : 0.5;
        const double z = vd.inv_dmax + ((double)(active ? k : 0) + u) * vd.delta;
        // the label's cost is summed per chunk (at most 128 pixels times the
        // neighbour views) and the chunk sums are added up, which keeps the
        // FP32 sum within ~1e-5 relative for superpixels of any size
        float total = 0.f;
        for (int pc = 0; pc < n; pc += SWEEP_CHUNK) {
            float cost = 0.f;
            const int cn = min(SWEEP_CHUNK, n - pc);
            __syncthreads();
            for (int i = threadIdx.x; i < cn; i += THREADS) {
                const unsigned pk = __ldg(w.sp_pix + off + pc + i);
                const int x = pk & 0xffff, y = pk >> 16;
                sh.d[i] = make_float2((float)(x - ref.x), (float)(y - ref.y));
                const float3 rc = texel_colour<FMT>(own_tex, x, y, vd.W, vd.H);
                float front = 1.f;
                if (WORLD) front = (sh.gh[0] * x + sh.gh[1] * y + sh.gh[2]) > 0.0 ? 1.f : 0.f;
                sh.ref[i] = make_float4(rc.x, rc.y, rc.z, front);
            }
            if (!WORLD) {
                __syncthreads();
                for (int t = threadIdx.x; t < cn * nnb; t += THREADS) {
                    const int j = t / cn, i = t - j * cn;
                    const SweepPair &sp = sh.pair[j];
                    const float2 d = sh.d[i];
                    if (PF == PF_SHIFT) {
                        // the pixel offset and, for 16-bit textures, the pixel's colour in
                        // the texture's format (one broadcast per sample instead of two),
                        // else its offset in view j's sampling texture
                        const int du = (int)d.x, dv = (int)d.y;
                        if constexpr (tex_fmt<FMT>() != LFD_RGBA_F32) {
                            const float4 rc = sh.ref[i];
                            sh.xyw[j][i] = make_float4(__int_as_float(du), __int_as_float(dv),
                                                       __uint_as_float(pack2<tex_fmt<FMT>()>(rc.x, rc.y)),
                                                       __uint_as_float(pack2<tex_fmt<FMT>()>(rc.z, 0.f)));
                        } else {
                            sh.xyw[j][i] = make_float4(__int_as_float(du), __int_as_float(dv),
                                                       __int_as_float(dv * (sp.Wi + 1) + du), 0.f);
                        }
                    } else {
                        sh.xyw[j][i] = make_float4(fmaf(sp.a00, d.x, sp.a01 * d.y), fmaf(sp.a10, d.x, sp.a11 * d.y),
                                                   fmaf(sp.a20, d.x, sp.a21 * d.y), 0.f);
                    }
                }
            }
            __syncthreads();
            for (int j = 0; j < nnb; j++) {
                const SweepPair &sp = sh.pair[j];
                // FP64 composition of the label's homography, anchored at ref
                const double zq0 = z * sp.q[0], zq1 = z * sp.q[1], zq2 = z * sp.q[2];
                const float cx = (float)fma(zq0, sh.gh[3], sp.pref[0]);
                const float cy = (float)fma(zq1, sh.gh[3], sp.pref[1]);
                const float cw = (float)fma(zq2, sh.gh[3], sp.pref[2]);
                float a00 = sp.a00, a01 = sp.a01, a10 = sp.a10, a11 = sp.a11, a20 = sp.a20, a21 = sp.a21;
                if (WORLD) {
                    a00 = (float)fma(zq0, sh.gh[0], sp.p0[0]); a01 = (float)fma(zq0, sh.gh[1], sp.p1[0]);
                    a10 = (float)fma(zq1, sh.gh[0], sp.p0[1]); a11 = (float)fma(zq1, sh.gh[1], sp.p1[1]);
                    a20 = (float)fma(zq2, sh.gh[0], sp.p0[2]); a21 = (float)fma(zq2, sh.gh[1], sp.p1[2]);
                }
                const void *tex = sp.tex;
                const int Wi = sp.Wi, Hi = sp.Hi;
                if (WORLD) {
#pragma unroll 4
                    for (int i = 0; i < cn; i++) {
                        const float2 d = sh.d[i];
                        const float4 rc = sh.ref[i];
                        const float X = fmaf(a00, d.x, fmaf(a01, d.y, cx));
                        const float Y = fmaf(a10, d.x, fmaf(a11, d.y, cy));
                        const float Wz = fmaf(a20, d.x, fmaf(a21, d.y, cw));
                        float t = tssd_sample<FMT>(tex, Wi, Hi, X, Y, Wz, make_float3(rc.x, rc.y, rc.z), T);
                        if (rc.w == 0.f) t = T;
                        cost += t;
                    }
                } else if (PF == PF_SHIFT) {
                    // translation pair: pixel offset (du, dv) samples at (du + X0, dv + Y0);
                    // with ix = du + floor(X0) and fx = X0 - floor(X0) the texture-area
                    // test -1/2 <= ix + fx < Wi - 1/2 is lo <= ix <= lo + Wi - 1, lo = -1
                    // when fx >= 1/2 and 0 otherwise (the same for y)
                    // The shift (X0, Y0) = (cx, cy) / w is split into its integer part and
                    // its fraction in FP64 (w = P (ref,1)_z for every label: q_z = 0), so
                    // the fraction is exact to FP32 rounding of a number below 1 whatever
                    // the image size (an absolute FP32 position near x = 2000 would carry
                    // ~1e-4 px).
                    const float4 *xyw = sh.xyw[WORLD ? 0 : j];
                    const double X0 = fma(zq0, sh.gh[3], sp.pref[0]) * sp.icw;
                    const double Y0 = fma(zq1, sh.gh[3], sp.pref[1]) * sp.icw;
                    if (sp.icw > 0.0 && fabs(X0) < 1e9 && fabs(Y0) < 1e9) {
                        const int ixk = __double2int_rd(X0), iyk = __double2int_rd(Y0);
                        const float fx = (float)(X0 - (double)ixk), fy = (float)(Y0 - (double)iyk);
                        const int ox = ixk + (fx >= 0.5f ? 1 : 0), oy = iyk + (fy >= 0.5f ? 1 : 0);
                        const unsigned spx = (unsigned)(Wi - 1), spy = (unsigned)(Hi - 1);
                        const long long koff = quad_index(ixk, iyk, Wi), npx = quad_entries(Wi, Hi);
#pragma unroll 4
                        for (int i = 0; i < cn; i++) {
                            const float4 q = xyw[i];
                            const int du = __float_as_int(q.x), dv = __float_as_int(q.y);
                            const bool in = (unsigned)(du + ox) <= spx && (unsigned)(dv + oy) <= spy;
                            // branch-free: a sample off the texture area reads entry 0
                            float t;
                            if constexpr (tex_fmt<FMT>() != LFD_RGBA_F32) {
                                const long long e = in ? koff + (dv * (Wi + 1) + du) : 0;
                                t = tssd_quad_href<FMT>(tex, e, npx, fx, fy, __float_as_uint(q.z),
                                                        __float_as_uint(q.w), T);
                            } else {
                                const float4 rc = sh.ref[i];
                                const long long e = in ? koff + __float_as_int(q.z) : 0;
                                t = tssd_quad<FMT>(tex, e, npx, fx, fy, make_float3(rc.x, rc.y, rc.z), T);
                            }
                            cost += in ? t : T;
                        }
                    } else {
                        for (int i = 0; i < cn; i++) cost += T;
                    }
                } else if (PF == PF_AFFINE) {
                    // affine pair: the homogeneous coordinate is cw for every pixel
                    // (P row 3 = (0, 0, P22), q_z = 0), one reciprocal per label and view;
                    // the same arithmetic as the general loop, value for value
                    const float4 *xyw = sh.xyw[WORLD ? 0 : j];
                    const float rw = rcp_approx(cw);
                    if (cw > 0.f) {
#pragma unroll 4
                        for (int i = 0; i < cn; i++) {
                            const float4 q = xyw[i];
                            const float4 rc = sh.ref[i];
                            cost += tssd_at<FMT>(tex, Wi, Hi, (q.x + cx) * rw, (q.y + cy) * rw,
                                                 make_float3(rc.x, rc.y, rc.z), T);
                        }
                    } else {
                        for (int i = 0; i < cn; i++) cost += T;
                    }
                } else {
                    const float4 *xyw = sh.xyw[WORLD ? 0 : j];
#pragma unroll 4
                    for (int i = 0; i < cn; i++) {
                        const float4 q = xyw[i];
                        const float4 rc = sh.ref[i];
                        cost += tssd_sample<FMT>(tex, Wi, Hi, q.x + cx, q.y + cy, q.z + cw,
                                                 make_float3(rc.x, rc.y, rc.z), T);
                    }
                }
            }
            total += cost;
        }
        const float cost = total;
        if (active) {
            if (cost_out) cost_out[(long long)gs * c.L + k] = cost * c.col_scale * c.col_scale;
            if (cost < best_cost) {   // k increases within a thread: strict < keeps the lowest k
                best_cost = cost;
                best_k = k;
            }
        }
    }
    // block arg-min, lowest k on ties
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float oc = __shfl_xor_sync(0xffffffffu, best_cost, o);
        const int ok = __shfl_xor_sync(0xffffffffu, best_k, o);
        if (oc < best_cost || (oc == best_cost && ok < best_k)) {
            best_cost = oc;
            best_k = ok;
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sh.bc[wid] = best_cost;
        sh.bk[wid] = best_k;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float bc = sh.bc[0];
        int bk = sh.bk[0];
        for (int i = 1; i < THREADS / 32; i++)
            if (sh.bc[i] < bc || (sh.bc[i] == bc && sh.bk[i] < bk)) {
                bc = sh.bc[i];
                bk = sh.bk[i];
            }
        const double u = vd.jitter ? jitter_u(vd.seed, vd.lf_index, vd.lv, s, bk) : 0.5;
        const double z = vd.inv_dmax + ((double)bk + u) * vd.delta;
        planes[gs] = make_float4((float)(1.0 / z), sh.n[0], sh.n[1], sh.n[2]);
        if (label_out) label_out[gs] = bk;
        atomicAdd(&w.ctr->hyp, (unsigned long long)L);
        atomicAdd(&w.ctr->samples, (unsigned long long)L * n * nnb);
        atomicAdd(&w.ctr->taken_sweep, (unsigned long long)L * n * nnb);
    }
}

// ---------------------------------------------------------------------------
// bounded sweep: the winning label without every label's full cost
// ---------------------------------------------------------------------------
//
// lfd_plane_sweep without cost_out and the frames need the arg-min label only.
// Every sample costs between 0 and T, so a label's partial sum is a lower
// bound of its cost: once it exceeds the cost of any one label, the label is
// out.  One CTA of NW warps sweeps one superpixel:
//   1. lanes over labels (32 a pass, the passes split between the warps), the
//      first (chunk of pixels, view) for all labels;
//   2. the label with the lowest partial sum is summed in full, threads over
//      pixels (the incumbent): its cost plus rounding is the bound B;
//   3. the labels still at or below B are listed and carried on (chunk, view)
//      by (chunk, view), the list compacted after each;
//   4. with at most BS_LANES left, each is summed to the end by one warp,
//      lanes over pixels, and left at the first view after which it exceeds B;
//      B falls with every better label;
//   5. if several labels end within the rounding of the two summation orders
//      of each other, these alone are carried on as in 3 to their exact sums.
// The result is the label that the full sums choose, lowest label on ties:
// sums that decide are taken in k_sweep's order, sums in another order only
// exclude, with the margin of their rounding (sweep_eps).
//
// Samples in the image's interior take a loop without window tests, when the
// superpixel's box lands inside for all 32 labels of the pass.  FP64 (the
// labels' projections) is taken lane-parallel over labels or (label, view)
// pairs: its pipe is 16 times narrower than FP32's here.
//
// Measured against the full sweep (one thread per label): 16 x 1080p FP16,
// 256 labels, 4 x 4 grid 104.6 -> 25.9 ms (24 % of the samples taken; other
// scenes of this size 21.9 to 27.5 ms with 20 to 25 %);
// 8 x 1024x768 RGBA8, 256 labels, 30-degree arc 20.2 -> 13.5 ms (58 %: wide
// baselines leave the best label a high cost, and the others go later).  What
// bounds it: issue (64 % of the cycles) with the L1 data pipe at 66 % of its
// wavefronts, six of which a sample's 24-byte record needs.  Four warps share
// a superpixel because one warp each (29 KB of shared memory per four) left
// the gathers 28 KB of L1: 49.5 and 17.7 ms.  12 CTAs per SM at 40 registers:
// 25.9 / 13.5 ms, 10 at 48: 26.3 / 13.6, 8 at 64: 26.2 / 13.8; two warps per
// CTA: 44.2 / 21.6, eight: 27.7 / 13.7.  BS_LANES 24, 48, 96: within 2 %.
constexpr int BS_LABELS = SWEEP_BOUNDED_LABELS;
constexpr int BS_LANES = 48;        // labels left at which the lanes turn to pixels
constexpr int BS_BATCH = 8;         // labels per round of that

// a label's projection into one neighbour view as it is kept in shared memory
struct LabelRec {
    float a, b, c;
    unsigned d;
    int e, f;
};

template <int FMT, int NW>
struct BoundedShared {
    static constexpr bool H16 = tex_fmt<FMT>() != LFD_RGBA_F32;
    // the chunk's pixels in the terms of one neighbour view:
    //   translation: {texture offset, (dv << 16 | du), colour as 16-bit rg, b}
    //   affine:      {x, y, rg, b}          general: {x, y, w, rg}
    // with (x, y, w) = P (du, dv, 0); F32 colours and the general form's blue are in `col`
    union {
        float4 rec[SWEEP_CHUNK];
        LabelRec lr[BS_BATCH * LFD_MAXN];
    };
    typename std::conditional<H16, unsigned, float4>::type col[SWEEP_CHUNK];
    float2 sum[BS_LABELS];             // {sum of the finished chunks, sum of this chunk} of each label
    double z[BS_LABELS];               // inverse depth of each label
    unsigned short list[BS_LABELS];    // labels not excluded
    float appr[BS_LANES];              // their costs in the lane order, negative when out
    unsigned km[BS_LABELS / 32];       // labels kept per pass
    unsigned long long low;            // {lowest partial sum, its label}
    unsigned bound;                    // bits of B
    float part[NW];
    int4 box[NW];
    unsigned long long best;           // {lowest exact cost, its label}
    int item;
    unsigned long long taken;
    SweepPair pair[LFD_MAXN];
};

// a label's projection into one neighbour view, and its samples there
template <int FMT, int PF>
struct LabelView {
    float cx, cy, cw;                  // general, affine: the label's column; affine: cw = 1 / w
    float fx, fy;                      // translation: bilinear fractions
    unsigned koff;                     //   texture entry of the anchor pixel (mod 2^32)
    int ox, oy;                        //   window offsets
    bool ok;                           // false: every sample is off the view (cost T)

    __device__ __forceinline__ void set(const SweepPair &sp, double z)
    {
        const double X = __dadd_rn(__dmul_rn(z, sp.q[0]), sp.pref[0]);
        const double Y = __dadd_rn(__dmul_rn(z, sp.q[1]), sp.pref[1]);
        if (PF == PF_SHIFT) {
            const double X0 = X * sp.icw, Y0 = Y * sp.icw;
            ok = sp.icw > 0.0 && fabs(X0) < 1e9 && fabs(Y0) < 1e9;
            const int ixk = ok ? __double2int_rd(X0) : 0, iyk = ok ? __double2int_rd(Y0) : 0;
            fx = ok ? (float)(X0 - (double)ixk) : 0.f;
            fy = ok ? (float)(Y0 - (double)iyk) : 0.f;
            ox = ixk + (fx >= 0.5f ? 1 : 0);
            oy = iyk + (fy >= 0.5f ? 1 : 0);
            koff = (unsigned)(iyk + 1) * (unsigned)(sp.Wi + 1) + (unsigned)(ixk + 1);
        } else {
            cx = (float)X;
            cy = (float)Y;
            const float w = (float)__dadd_rn(__dmul_rn(z, sp.q[2]), sp.pref[2]);
            ok = PF == PF_GENERAL || w > 0.f;
            cw = PF == PF_AFFINE ? rcp_approx(w) : w;
        }
    }

    __device__ __forceinline__ LabelRec pack() const
    {
        if (PF == PF_SHIFT) return LabelRec{fx, fy, 0.f, koff, ok ? ox : 0x40000000, oy};
        return LabelRec{cx, cy, cw, ok ? 1u : 0u, 0, 0};
    }

    __device__ __forceinline__ void unpack(const LabelRec &r)
    {
        if (PF == PF_SHIFT) {
            fx = r.a; fy = r.b; koff = r.d; ox = r.e; oy = r.f;
            ok = r.e != 0x40000000;
        } else {
            cx = r.a; cy = r.b; cw = r.c;
            ok = r.d != 0u;
        }
    }

    // every pixel of the box [x0, x1] x [y0, y1] of offsets samples inside the view
    __device__ __forceinline__ bool inside(const SweepPair &sp, int x0, int x1, int y0, int y1) const
    {
        if (!ok) return false;
        if (PF == PF_SHIFT)
            return ox + x0 >= 0 && ox + x1 <= sp.Wi - 1 && oy + y0 >= 0 && oy + y1 <= sp.Hi - 1;
        return box_inside(PF == PF_GENERAL, sp.a00, sp.a01, sp.a10, sp.a11, sp.a20, sp.a21, cx, cy, cw, sp.Wi, sp.Hi,
                          x0, x1, y0, y1);
    }

    template <typename C>
    __device__ __forceinline__ float at(const void *tex, unsigned npx, unsigned e, float fxx, float fyy, const C &c,
                                        float T) const
    {
        if constexpr (tex_fmt<FMT>() != LFD_RGBA_F32)
            return tssd_quad_href<FMT>(tex, (long long)e, (long long)npx, fxx, fyy, c.x, c.y, T);
        else
            return tssd_quad<FMT>(tex, (long long)e, (long long)npx, fxx, fyy, make_float3(c.x, c.y, c.z), T);
    }

    // one sample: {a, b, c} the pixel's view terms, `col` its colour
    template <bool INSIDE, typename C>
    __device__ __forceinline__ float sample(const SweepPair &sp, unsigned npx, float a, float b, float c, const C &col,
                                            float T) const
    {
        if (PF == PF_SHIFT) {
            const unsigned e = koff + __float_as_uint(a);
            if (INSIDE) return at(sp.tex, npx, e, fx, fy, col, T);
            const int dxy = __float_as_int(b);
            const bool in = ok && (unsigned)((int)(short)dxy + ox) <= (unsigned)(sp.Wi - 1) &&
                            (unsigned)((dxy >> 16) + oy) <= (unsigned)(sp.Hi - 1);
            const float t = at(sp.tex, npx, in ? e : 0u, fx, fy, col, T);
            return in ? t : T;
        }
        float r = cw, wz = 1.f;
        if (PF == PF_GENERAL) {
            wz = c + cw;
            r = rcp_approx(wz);
        }
        const float x = (a + cx) * r, y = (b + cy) * r;
        const bool in = INSIDE || (ok && wz > 0.f && x >= -0.5f && x < (float)sp.Wi - 0.5f && y >= -0.5f &&
                                   y < (float)sp.Hi - 0.5f);
        const float xs = in ? x : 0.f, ys = in ? y : 0.f;
        // floor by adding 1.5 * 2^23 towards -inf: exact for |x| < 2^22
        const float tx = __fadd_rd(xs, 12582912.f), ty = __fadd_rd(ys, 12582912.f);
        const int xi = __float_as_int(tx) - 0x4B400000, yi = __float_as_int(ty) - 0x4B400000;
        const unsigned e = (unsigned)(yi + 1) * (unsigned)(sp.Wi + 1) + (unsigned)(xi + 1);
        const float t = at(sp.tex, npx, e, xs - (tx - 12582912.f), ys - (ty - 12582912.f), col, T);
        return in ? t : T;
    }
};

// a pixel of the superpixel: its offset from the anchor (dv << 16 | du) and its
// colour (16-bit textures: {rg, b} in the texture's format)
template <int FMT>
struct SweepPixel {
    static constexpr bool H16 = tex_fmt<FMT>() != LFD_RGBA_F32;
    int dxy;
    typename std::conditional<H16, uint2, float3>::type col;

    __device__ __forceinline__ void load(const Workspace &w, const ViewDev &vd, int2 ref, int at)
    {
        const unsigned pk = __ldg(w.sp_pix + at);
        const int x = pk & 0xffff, y = pk >> 16;
        dxy = (int)(((unsigned)(y - ref.y) << 16) | ((unsigned)(x - ref.x) & 0xffffu));
        const float3 rc = texel_colour<FMT>(vd.quad, x, y, vd.W, vd.H);
        if constexpr (H16) col = make_uint2(pack2<tex_fmt<FMT>()>(rc.x, rc.y), pack2<tex_fmt<FMT>()>(rc.z, 0.f));
        else col = rc;
    }
    __device__ __forceinline__ int du() const { return (int)(short)dxy; }
    __device__ __forceinline__ int dv() const { return dxy >> 16; }

    // its terms in the view of `sp` (see BoundedShared::rec)
    template <int PF>
    __device__ __forceinline__ float3 terms(const SweepPair &sp) const
    {
        if (PF == PF_SHIFT)
            return make_float3(__int_as_float(dv() * (sp.Wi + 1) + du()), __int_as_float(dxy), 0.f);
        const float fu = (float)du(), fv = (float)dv();
        return make_float3(fmaf(sp.a00, fu, sp.a01 * fv), fmaf(sp.a10, fu, sp.a11 * fv),
                           PF == PF_GENERAL ? fmaf(sp.a20, fu, sp.a21 * fv) : 0.f);
    }
};

// cost += the chunk's samples of one label per lane, in pixel order
template <int FMT, int PF, int NW, bool INSIDE>
__device__ __forceinline__ float chunk_cost(const BoundedShared<FMT, NW> &sh, const SweepPair &sp, unsigned npx,
                                            const LabelView<FMT, PF> &lv, int cn, float cost, float T)
{
#pragma unroll 4
    for (int i = 0; i < cn; i++) {
        const float4 q = sh.rec[i];
        if constexpr (!BoundedShared<FMT, NW>::H16)
            cost += lv.template sample<INSIDE>(sp, npx, q.x, q.y, q.z, sh.col[i], T);
        else if constexpr (PF == PF_GENERAL)
            cost += lv.template sample<INSIDE>(sp, npx, q.x, q.y, q.z, make_uint2(__float_as_uint(q.w), sh.col[i]), T);
        else
            cost += lv.template sample<INSIDE>(sp, npx, q.x, q.y, 0.f,
                                               make_uint2(__float_as_uint(q.z), __float_as_uint(q.w)), T);
    }
    return cost;
}

// float keys ordered as integers (costs are not negative), ties to the lower label
__device__ __forceinline__ unsigned long long cost_key(float c, int k)
{
    return ((unsigned long long)__float_as_uint(c) << 32) | (unsigned)k;
}

// the sweep of superpixel gs by the CTA
template <int FMT, int PF, int NW>
__device__ __forceinline__ void bounded_sweep_sp(const Workspace &w, int gs, BoundedShared<FMT, NW> &sh,
                                                 float4 *planes, int *label_out)
{
    constexpr int THREADS = 32 * NW;
    constexpr int PASSES = (BS_LABELS / 32 + NW - 1) / NW;      // label passes per warp
    constexpr int PX = SWEEP_CHUNK / THREADS;                   // chunk pixels per thread
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int v = __ldg(w.sp_view + gs);
    const ViewDev &vd = w.views[v];
    if (vd.sweep_skip) return;               // warm-started view: its planes are given
    const int n = __ldg(w.sp_cnt + gs);
    if (n == 0) {
        if (tid == 0) {
            planes[gs] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (label_out) label_out[gs] = -1;
        }
        return;
    }
    const int2 ref = __ldg(w.sp_ref + gs);
    const int nnb = vd.nnb, L = vd.L, off = __ldg(w.sp_off + gs);
    const float T = vd.T;
    if (tid < nnb) {
        const PairDev &pd = w.pairs[v * LFD_MAXN + tid];
        SweepPair &sp = sh.pair[tid];
        sp.a00 = pd.Pf[0]; sp.a01 = pd.Pf[1];
        sp.a10 = pd.Pf[3]; sp.a11 = pd.Pf[4];
        sp.a20 = pd.Pf[6]; sp.a21 = pd.Pf[7];
        sp.Wi = pd.Wi; sp.Hi = pd.Hi;
        for (int r = 0; r < 3; r++) {
            sp.pref[r] = pd.P[3 * r] * ref.x + pd.P[3 * r + 1] * ref.y + pd.P[3 * r + 2];
            sp.q[r] = pd.q[r];
        }
        sp.icw = sp.pref[2] > 0.0 ? 1.0 / sp.pref[2] : 0.0;
        sp.tex = pd.quad_i;
    }
    for (int k = tid; k < L; k += THREADS) {
        sh.sum[k] = make_float2(0.f, 0.f);
        sh.list[k] = (unsigned short)k;
        const double u = vd.jitter ? jitter_u(vd.seed, vd.lf_index, vd.lv, gs - vd.sp_base, k) : 0.5;
        sh.z[k] = vd.inv_dmax + ((double)k + u) * vd.delta;
    }
    if (tid == 0) {
        sh.low = ~0ull;
        sh.best = ~0ull;
        sh.bound = __float_as_uint(INFINITY);
        sh.taken = 0;
    }

    const float eps = sweep_eps(n, nnb, SWEEP_CHUNK);
    int K = L, best_k = -1;
    unsigned long long taken = 0;            // per warp (lane 0's count is added up)
    bool bounded = false;                    // B is known
    // the remaining labels tie: carry them to their exact sums.  An infinite T
    // needs them too: a cost of infinity wins nowhere, not even as the last label
    bool exact_only = !(T < INFINITY);
    for (int pc = 0; pc < n && best_k < 0; pc += SWEEP_CHUNK) {
        const int cn = min(SWEEP_CHUNK, n - pc);
        SweepPixel<FMT> px[PX];
        int x0 = 0x7fff, x1 = -0x8000, y0 = 0x7fff, y1 = -0x8000;
#pragma unroll
        for (int r = 0; r < PX; r++)
            if (tid + r * THREADS < cn) {
                px[r].load(w, vd, ref, off + pc + tid + r * THREADS);
                x0 = min(x0, px[r].du()); x1 = max(x1, px[r].du());
                y0 = min(y0, px[r].dv()); y1 = max(y1, px[r].dv());
            }
        x0 = __reduce_min_sync(0xffffffffu, x0); x1 = __reduce_max_sync(0xffffffffu, x1);
        y0 = __reduce_min_sync(0xffffffffu, y0); y1 = __reduce_max_sync(0xffffffffu, y1);
        if (lane == 0) sh.box[wid] = make_int4(x0, x1, y0, y1);
        for (int j = 0; j < nnb; j++) {
            const SweepPair &sp = sh.pair[j];
            if (pc == 0 && j == 0) __syncthreads();              // the pairs and labels are set
            const unsigned npx = (unsigned)(sp.Wi + 1) * (unsigned)(sp.Hi + 1);
#pragma unroll
            for (int r = 0; r < PX; r++) {
                const int i = tid + r * THREADS;
                if (i < cn) {
                    const float3 q = px[r].template terms<PF>(sp);
                    float4 o = make_float4(q.x, q.y, q.z, 0.f);
                    if constexpr (BoundedShared<FMT, NW>::H16) {
                        if (PF == PF_GENERAL) {
                            o.w = __uint_as_float(px[r].col.x);
                            if (j == 0) sh.col[i] = px[r].col.y;
                        } else {
                            o.z = __uint_as_float(px[r].col.x);
                            o.w = __uint_as_float(px[r].col.y);
                        }
                    } else {
                        if (j == 0) sh.col[i] = make_float4(px[r].col.x, px[r].col.y, px[r].col.z, 0.f);
                    }
                    sh.rec[i] = o;
                }
            }
            __syncthreads();                 // records, box and label list
            int4 box = sh.box[0];
#pragma unroll
            for (int q = 1; q < NW; q++) {
                const int4 o = sh.box[q];
                box = make_int4(min(box.x, o.x), max(box.y, o.y), min(box.z, o.z), max(box.w, o.w));
            }
            const float B = __uint_as_float(sh.bound);
            const bool last = j == nnb - 1, end = last && pc + SWEEP_CHUNK >= n;
            unsigned long long low = ~0ull;  // the lane's lowest partial sum
            int kk[PASSES];
            unsigned keeps = 0;
#pragma unroll
            for (int h = 0; h < PASSES; h++) {
                const int p = wid + NW * h, base = 32 * p;
                kk[h] = 0;
                if (base < K) {
                    const int k = sh.list[min(base + lane, K - 1)];
                    float2 sm = sh.sum[k];
                    LabelView<FMT, PF> lv;
                    lv.set(sp, sh.z[k]);
                    const bool in = __all_sync(0xffffffffu, lv.inside(sp, box.x, box.y, box.z, box.w));
                    sm.y = in ? chunk_cost<FMT, PF, NW, true>(sh, sp, npx, lv, cn, sm.y, T)
                              : chunk_cost<FMT, PF, NW, false>(sh, sp, npx, lv, cn, sm.y, T);
                    taken += (unsigned)(min(32, K - base) * cn);
                    const float part = sm.x + sm.y;
                    if (last) sm = make_float2(part, 0.f);
                    const bool keep = base + lane < K && !(part > B);
                    const unsigned km = __ballot_sync(0xffffffffu, keep);
                    if (lane == 0) sh.km[p] = km;
                    if (keep) {
                        sh.sum[k] = sm;
                        low = min(low, cost_key(part, k));
                        keeps |= 1u << h;
                    }
                    kk[h] = k;
                }
            }
            if (end || !bounded) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) low = min(low, __shfl_xor_sync(0xffffffffu, low, o));
                if (lane == 0) atomicMin(end ? &sh.best : &sh.low, low);
            }
            __syncthreads();                 // list entries read, masks and sums written
            if (end) break;
            const int passes = (K + 31) / 32;
            int kept = 0;
            for (int p = 0; p < passes; p++) {
                const unsigned km = sh.km[p];
#pragma unroll
                for (int h = 0; h < PASSES; h++)
                    if (p == wid + NW * h && ((keeps >> h) & 1u))
                        sh.list[kept + __popc(km & ((1u << lane) - 1u))] = (unsigned short)kk[h];
                kept += __popc(km);
            }
            K = kept;
            if (!bounded) {
                // the incumbent: the lowest partial sum, summed in full (nothing is below it: its
                // low half is a label of the list, or, with infinite costs only, label 0)
                const int k = sh.low == ~0ull ? 0 : (int)(unsigned)sh.low;
                if (tid < nnb) {
                    LabelView<FMT, PF> lv;
                    lv.set(sh.pair[tid], sh.z[k]);
                    sh.lr[tid] = lv.pack();
                }
                __syncthreads();
                float c = 0.f;
                for (int i = tid; i < n; i += THREADS) {
                    SweepPixel<FMT> q;
                    q.load(w, vd, ref, off + i);
                    for (int j2 = 0; j2 < nnb; j2++) {
                        const SweepPair &s2 = sh.pair[j2];
                        LabelView<FMT, PF> lv;
                        lv.unpack(sh.lr[j2]);
                        const float3 t = q.template terms<PF>(s2);
                        c += lv.template sample<false>(s2, (unsigned)(s2.Wi + 1) * (unsigned)(s2.Hi + 1), t.x, t.y, t.z,
                                                       q.col, T);
                    }
                }
                c = warp_sum(c);
                if (lane == 0) sh.part[wid] = c;
                __syncthreads();
                if (tid == 0) {
                    float sum = 0.f;
                    for (int q = 0; q < NW; q++) sum += sh.part[q];
                    sh.bound = __float_as_uint(sum * (1.f + eps));
                    taken += (unsigned)(n * nnb);
                }
                bounded = true;
                continue;
            }
            if (K > BS_LANES || exact_only) continue;
            __syncthreads();                 // the list
            if (K == 1) {                    // every other label is out
                best_k = sh.list[0];
                break;
            }
            // lanes over pixels: the rest of every remaining label
            for (int t0 = 0; t0 < K; t0 += BS_BATCH) {
                const int tn = min(BS_BATCH, K - t0);
                for (int q = tid; q < tn * nnb; q += THREADS) {
                    LabelView<FMT, PF> lv;
                    lv.set(sh.pair[q % nnb], sh.z[sh.list[t0 + q / nnb]]);
                    sh.lr[q] = lv.pack();
                }
                __syncthreads();
                for (int t = wid; t < tn; t += NW) {
                    const float2 sl = sh.sum[sh.list[t0 + t]];
                    float c = sl.x + sl.y;
                    bool out = c > __uint_as_float(*(volatile unsigned *)&sh.bound);
                    for (int p2 = pc; p2 < n && !out; p2 += SWEEP_CHUNK) {
                        const int c2 = min(SWEEP_CHUNK, n - p2);
                        SweepPixel<FMT> q[SWEEP_CHUNK / 32];
#pragma unroll
                        for (int r = 0; r < SWEEP_CHUNK / 32; r++)
                            q[r].load(w, vd, ref, off + p2 + min(lane + 32 * r, c2 - 1));
                        for (int j2 = p2 == pc ? j + 1 : 0; j2 < nnb; j2++) {
                            const SweepPair &s2 = sh.pair[j2];
                            LabelView<FMT, PF> lv;
                            lv.unpack(sh.lr[t * nnb + j2]);
                            const unsigned np2 = (unsigned)(s2.Wi + 1) * (unsigned)(s2.Hi + 1);
                            float a = 0.f;
#pragma unroll
                            for (int r = 0; r < SWEEP_CHUNK / 32; r++) {
                                const float3 u = q[r].template terms<PF>(s2);
                                const float smp = lv.template sample<false>(s2, np2, u.x, u.y, u.z, q[r].col, T);
                                a += lane + 32 * r < c2 ? smp : 0.f;
                            }
                            c += warp_sum(a);
                            taken += (unsigned)c2;
                            if (c * (1.f - eps) > __uint_as_float(*(volatile unsigned *)&sh.bound)) {
                                out = true;
                                break;
                            }
                        }
                    }
                    if (lane == 0) {
                        sh.appr[t0 + t] = out ? -1.f : c;
                        if (!out) atomicMin(&sh.bound, __float_as_uint(c * (1.f + eps)));
                    }
                }
                __syncthreads();
            }
            // labels within the rounding of the best
            const float B2 = __uint_as_float(sh.bound);
            int ties = 0, mine[(BS_LANES + 31) / 32], rank[(BS_LANES + 31) / 32];
#pragma unroll
            for (int h = 0; h < (BS_LANES + 31) / 32; h++) {
                const int t = lane + 32 * h;
                const float a = t < K && t < BS_LANES ? sh.appr[t] : -1.f;
                const bool tie = a >= 0.f && !(a * (1.f - eps) > B2);
                const unsigned tm = __ballot_sync(0xffffffffu, tie);
                mine[h] = tie ? sh.list[t] : -1;
                rank[h] = ties + __popc(tm & ((1u << lane) - 1u));
                ties += __popc(tm);
            }
            __syncthreads();
            if (wid == 0)
#pragma unroll
                for (int h = 0; h < (BS_LANES + 31) / 32; h++)
                    if (mine[h] >= 0) sh.list[rank[h]] = (unsigned short)mine[h];
            K = ties;
            if (K == 1) {
                __syncthreads();
                best_k = sh.list[0];
                break;
            }
            exact_only = true;
        }
    }
    if (best_k < 0) best_k = sh.best == ~0ull || (unsigned)(sh.best >> 32) >= 0x7f800000u ? 0x7fffffff
                                                                                          : (int)(unsigned)sh.best;
    if (lane == 0) atomicAdd(&sh.taken, taken);
    __syncthreads();
    if (tid == 0) {
        const double u = vd.jitter ? jitter_u(vd.seed, vd.lf_index, vd.lv, gs - vd.sp_base, best_k) : 0.5;
        const double z = vd.inv_dmax + ((double)best_k + u) * vd.delta;
        planes[gs] = make_float4((float)(1.0 / z), 0.f, 0.f, -1.f);
        if (label_out) label_out[gs] = best_k;
        atomicAdd(&w.ctr->hyp, (unsigned long long)L);
        atomicAdd(&w.ctr->samples, (unsigned long long)L * n * nnb);
        atomicAdd(&w.ctr->taken_sweep, sh.taken);
    }
}

// persistent CTAs: superpixels of order_sweep[base .. base + count) in order
template <int FMT, int PF, int NW>
__global__ void __launch_bounds__(32 * NW, 48 / NW) k_sweep_bounded(const __grid_constant__ Workspace w, int base,
                                                                    int count, int qidx, float4 *planes, int *label_out)
{
    __shared__ BoundedShared<FMT, NW> sh;
    for (;;) {
        if (threadIdx.x == 0) sh.item = atomicAdd(&w.queue[qidx], 1);
        __syncthreads();
        const int item = sh.item;
        if (item >= count) break;
        bounded_sweep_sp<FMT, PF, NW>(w, __ldg(w.order_sweep + base + item), sh, planes, label_out);
        __syncthreads();
    }
}

template <int FMT, int PF>
static cudaError_t launch_bounded(const Workspace &w, const LaunchCfg &lc, int base, int count, int qidx,
                                  float4 *planes, int *label, cudaStream_t st)
{
    constexpr int NW = 4;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep_bounded<FMT, PF, NW>, 32 * NW, 0);
    if (e != cudaSuccess) return e;
    const int grid = max(1, min(count, per_sm * lc.num_sms));
    k_sweep_bounded<FMT, PF, NW><<<grid, 32 * NW, 0, st>>>(w, base, count, qidx, planes, label);
    return cudaGetLastError();
}

// camera-frame sweeps: 6 CTAs of 256 threads (12 of 128) per SM, at most 40
// registers; world-frame sweeps (more FP64 per label) 4, at most 64

// one CTA per superpixel of order_sweep[base .. base + count)
template <int FMT, bool WORLD, int THREADS, int PF>
__global__ void __launch_bounds__(THREADS, (WORLD ? 1024 : 1536) / THREADS) k_sweep(Workspace w, Consts c, int base,
                                                                                     float4 *planes, int *label_out,
                                                                                     float *cost_out)
{
    __shared__ SweepShared<THREADS, WORLD> sh;
    sweep_sp<FMT, WORLD, THREADS, PF>(w, c, __ldg(w.order_sweep + base + blockIdx.x), sh, planes, label_out,
                                       cost_out);
}

// persistent CTAs: superpixels of order_sweep[base .. base + count) taken in
// order (size classes, largest first), queue counter queue[qidx]
template <int FMT, bool WORLD, int THREADS, int PF>
__global__ void __launch_bounds__(THREADS, (WORLD ? 1024 : 1536) / THREADS) k_sweep_persistent(
    Workspace w, Consts c, int base, int count, int qidx, float4 *planes, int *label_out, float *cost_out)
{
    __shared__ SweepShared<THREADS, WORLD> sh;
    for (;;) {
        if (threadIdx.x == 0) sh.item = atomicAdd(&w.queue[qidx], 1);
        __syncthreads();
        const int item = sh.item;
        __syncthreads();
        if (item >= count) break;
        sweep_sp<FMT, WORLD, THREADS, PF>(w, c, __ldg(w.order_sweep + base + item), sh, planes, label_out, cost_out);
        __syncthreads();
    }
}

template <int FMT, bool WORLD, int THREADS, int PF>
static cudaError_t launch_sweep_a(const Workspace &w, const Consts &c, const LaunchCfg &lc, int base, int count,
                                  int qidx, float4 *planes, int *label, float *cost, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    if (lc.sweep_persistent) {
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, k_sweep_persistent<FMT, WORLD, THREADS, PF>, THREADS, 0);
        if (e != cudaSuccess) return e;
        const int grid = max(1, min(count, per_sm * lc.num_sms));
        k_sweep_persistent<FMT, WORLD, THREADS, PF><<<grid, THREADS, 0, st>>>(w, c, base, count, qidx, planes,
                                                                               label, cost);
    } else {
        k_sweep<FMT, WORLD, THREADS, PF><<<count, THREADS, 0, st>>>(w, c, base, planes, label, cost);
    }
    return cudaGetLastError();
}

template <int FMT, bool WORLD, int THREADS>
static cudaError_t launch_sweep_t(const Workspace &w, const Consts &c, const LaunchCfg &lc, int base, int count,
                                  int qidx, float4 *planes, int *label, float *cost, cudaStream_t st)
{
    if (!WORLD && c.affine && c.shift)
        return launch_sweep_a<FMT, false, THREADS, PF_SHIFT>(w, c, lc, base, count, qidx, planes, label, cost, st);
    if (!WORLD && c.affine)
        return launch_sweep_a<FMT, false, THREADS, PF_AFFINE>(w, c, lc, base, count, qidx, planes, label, cost, st);
    return launch_sweep_a<FMT, WORLD, THREADS, PF_GENERAL>(w, c, lc, base, count, qidx, planes, label, cost, st);
}

template <int FMT>
static cudaError_t launch_sweep_f(const Workspace &w, const Consts &c, const LaunchCfg &lc, int threads, int base,
                                  int count, int qidx, float4 *planes, int *label, float *cost, cudaStream_t st)
{
    // arg-min only (no cost_out), camera frame, up to BS_LABELS labels (its
    // shared-memory lists): the bounded sweep, where the class's sizes suit it
    // (sweep_bounded).  Costs need every label's full sum, world-frame sweeps
    // and larger label counts keep the full sweep as well.
    if (c.sweep_bounded && !cost && !c.sweep_frame) {
        if (c.affine && c.shift) return launch_bounded<FMT, PF_SHIFT>(w, lc, base, count, qidx, planes, label, st);
        if (c.affine) return launch_bounded<FMT, PF_AFFINE>(w, lc, base, count, qidx, planes, label, st);
        return launch_bounded<FMT, PF_GENERAL>(w, lc, base, count, qidx, planes, label, st);
    }
    if (c.sweep_frame)   // world-frame sweeps: 128 or 256 threads
        return threads <= 128 ? launch_sweep_t<FMT, true, 128>(w, c, lc, base, count, qidx, planes, label, cost, st)
                              : launch_sweep_t<FMT, true, 256>(w, c, lc, base, count, qidx, planes, label, cost, st);
    switch (threads) {
    case 64: return launch_sweep_t<FMT, false, 64>(w, c, lc, base, count, qidx, planes, label, cost, st);
    case 128: return launch_sweep_t<FMT, false, 128>(w, c, lc, base, count, qidx, planes, label, cost, st);
    case 160: return launch_sweep_t<FMT, false, 160>(w, c, lc, base, count, qidx, planes, label, cost, st);
    case 192: return launch_sweep_t<FMT, false, 192>(w, c, lc, base, count, qidx, planes, label, cost, st);
    case 224: return launch_sweep_t<FMT, false, 224>(w, c, lc, base, count, qidx, planes, label, cost, st);
    default: return launch_sweep_t<FMT, false, 256>(w, c, lc, base, count, qidx, planes, label, cost, st);
    }
}

cudaError_t launch_sweep(const Workspace &w, const Consts &c, const LaunchCfg &lc, int threads, int base, int count,
                         int qidx, float4 *planes, int *label, float *cost, cudaStream_t st)
{
    switch (c.fmt) {
    case LFD_RGBA8: return launch_sweep_f<LFD_RGBA8>(w, c, lc, threads, base, count, qidx, planes, label, cost, st);
    case LFD_RGBA_F16:
        return launch_sweep_f<LFD_RGBA_F16>(w, c, lc, threads, base, count, qidx, planes, label, cost, st);
    case LFD_RGBA_BF16:
        return launch_sweep_f<LFD_RGBA_BF16>(w, c, lc, threads, base, count, qidx, planes, label, cost, st);
    case LFD_RGBA_F32:
        return launch_sweep_f<LFD_RGBA_F32>(w, c, lc, threads, base, count, qidx, planes, label, cost, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lfd
