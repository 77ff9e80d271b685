// track.cu -- the frame-to-model tracking loss (Eq. 2 with the alpha^3 and
// inlier masks of Supp. A) for the tracking keyframes of a plan:
//   k_track_median  one cluster per tracking keyframe: the lower median of
//                   the FP32 depth errors of the pixels with input depth, by
//                   a three-pass radix select over the float's bits (11 + 10
//                   + 10; non-negative floats order as their bit patterns);
//   k_track_loss    one CTA per tile: inlier test e <= 50 * median (FP32),
//                   weight M_in * alpha^3, the tile's loss summed in a fixed
//                   order, and for the standalone entry the cotangents and
//                   the inlier mask.
// The inlier decisions use the FP32 values the oracle's mirror uses, so they
// are reproduced exactly; the weights and the loss are values.
#include "gs_internal.cuh"

namespace {

using namespace gsk;

constexpr uint32_t kInfBits = 0x7f800000u;  // +inf marks a pixel without input depth
constexpr int kMedThreads = 1024;
constexpr int kMedBins = 2048;
constexpr int kMedCluster = 8;  // CTAs per keyframe (the portable cluster size)
constexpr int kMedUnroll = 8;   // pixel loads in flight per thread beyond the kept ones
// pixels per thread held in registers over the passes: of the 64 that 1024
// threads leave each, eight for those loads and 16 to work with (with 48 kept:
// 18.7 us for 640x480, 17.9 with 40, and 20.2 against 20.4 for 768x512, where
// 48 hold the whole slice)
constexpr int kMedKeep = 65536 / kMedThreads - kMedUnroll - 16;
constexpr int kMedGroup = 4;    // of those, taken or left out together
static_assert(kMedKeep % kMedGroup == 0, "the kept pixels are whole groups");
// the three digits, high to low, of a non-negative float's 31 bits
__device__ __forceinline__ constexpr int med_shift(int pass) { return pass == 0 ? 20 : (pass == 1 ? 10 : 0); }
__device__ __forceinline__ constexpr uint32_t med_mask(int pass) { return pass == 0 ? 0x7ffu : 0x3ffu; }

// One cluster of kMedCluster CTAs per tracking keyframe: each CTA counts the
// digits of its eighth of the pixels in its own shared histogram (one per
// pass, cleared together up front), and after one cluster barrier every CTA
// adds the eight histograms through distributed shared memory and finds the
// digit that holds the median's rank -- the same on all of them, so nothing
// is sent back.  The first kMedKeep pixels per thread of its slice
// are read once and kept in registers over the three passes; what lies beyond
// (frames of more than 327,680 pixels) is read by each.  Bound by latency (one
// 640x480 frame is 1.2 MB): 14.1, 17.9, 17.8 and 34.0 us for 320x240, 640x480,
// 660x480 and 1200x680 by ncu; with one limit for a whole slice, 38 pixels, and
// none left out, 16.7, 18.1, 22.8 and 38.6.  One CTA per keyframe took 346 us on a
// 640x480 frame, by ncu: each pass one dependent load and one match_any per
// 1024 pixels; the tracking iteration spent two thirds of its time there (40
// iterations of a 640x480 frame on 150k Gaussians: 18.97 -> 7.06 ms with
// this kernel).
__global__ void __cluster_dims__(kMedCluster, 1, 1) __launch_bounds__(kMedThreads) k_track_median(const gsl::TrackArgs a)
{
    __shared__ __align__(8) uint32_t hist[3][kMedBins];
    __shared__ uint32_t s_scan[kMedThreads / 32 + 1];
    __shared__ uint32_t s_sel[2];
    const uint32_t rank = blockIdx.x % kMedCluster;
    const int vp = a.track_vps[blockIdx.x / kMedCluster];
    const VpDesc &d = a.vps[vp];
    // (a keyframe has at most 2^30 pixels)
    const uint32_t n = (uint32_t)d.W * (uint32_t)d.H, per = (n + kMedCluster - 1) / kMedCluster;
    const uint32_t i0 = min(rank * per, n), len = min(i0 + per, n) - i0;
    const uint32_t *v = reinterpret_cast<const uint32_t *>(a.err) + d.pix_base + i0;
    for (int b = threadIdx.x; b < 3 * kMedBins; b += kMedThreads)
        (&hist[0][0])[b] = 0;
    pdl_wait();
    // (a group that lies past the slice is left out)
    uint32_t kept[kMedKeep];
#pragma unroll
    for (int g = 0; g < kMedKeep; g += kMedGroup)
        if ((uint32_t)g * kMedThreads < len) {
#pragma unroll
            for (int u = g; u < g + kMedGroup; ++u) {
                const uint32_t i = u * kMedThreads + threadIdx.x;
                kept[u] = i < len ? v[i] : kInfBits;
            }
        }
    __syncthreads();
    uint32_t prefix = 0, mask = 0, k = 0, m = 0;
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
        uint32_t *h = hist[pass];
        auto count = [&](uint32_t x) {
            if (x < kInfBits && (x & mask) == prefix)
                atomicAdd(&h[(x >> med_shift(pass)) & med_mask(pass)], 1u);
        };
#pragma unroll
        for (int g = 0; g < kMedKeep; g += kMedGroup)
            if ((uint32_t)g * kMedThreads < len) {
#pragma unroll
                for (int u = g; u < g + kMedGroup; ++u)
                    count(kept[u]);
            }
        for (uint32_t base = kMedKeep * kMedThreads + threadIdx.x; base < len; base += kMedUnroll * kMedThreads) {
            uint32_t x[kMedUnroll];
#pragma unroll
            for (int u = 0; u < kMedUnroll; ++u)
                x[u] = base + u * kMedThreads < len ? v[base + u * kMedThreads] : kInfBits;
#pragma unroll
            for (int u = 0; u < kMedUnroll; ++u)
                count(x[u]);
        }
        cluster_sync();
        // the cluster's counts of bins 2t and 2t + 1, their exclusive scan,
        // and the bin holding rank k
        uint32_t h0 = 0, h1 = 0;
#pragma unroll
        for (int c = 0; c < kMedCluster; ++c) {
            const uint2 q = cluster_load2(&h[2 * threadIdx.x], (uint32_t)c);
            h0 += q.x;
            h1 += q.y;
        }
        uint32_t tot;
        const uint32_t ex = block_excl_scan<kMedThreads>(h0 + h1, s_scan, tot);
        if (pass == 0) {
            m = tot;  // (no pixel has input depth: every pass selects nothing)
            k = m > 0 ? (m - 1) / 2 : 0;
            if (threadIdx.x == 0)
                s_sel[0] = s_sel[1] = 0;
            __syncthreads();
        }
        if (k >= ex && k < ex + h0) {
            s_sel[0] = 2 * threadIdx.x;
            s_sel[1] = k - ex;
        } else if (k >= ex + h0 && k < ex + h0 + h1) {
            s_sel[0] = 2 * threadIdx.x + 1;
            s_sel[1] = k - ex - h0;
        }
        __syncthreads();
        prefix |= s_sel[0] << med_shift(pass);
        mask |= med_mask(pass) << med_shift(pass);
        k = s_sel[1];
        __syncthreads();
    }
    cluster_sync();  // every CTA has read this one's histograms
    if (rank == 0 && threadIdx.x == 0) {
        a.med[vp] = m > 0 ? __uint_as_float(prefix) : 0.0f;
        a.n_valid[vp] = (int)m;
    }
}

__global__ void __launch_bounds__(256) k_track_loss(const gsl::TrackArgs a)
{
    __shared__ float s_red[8];
    const uint32_t t = a.first_tile + blockIdx.x;
    const int vp = (int)a.tile_vp[t];
    const VpDesc &d = a.vps[vp];
    pdl_wait();
    if (d.loss_kind != 1)
        return;
    const uint32_t lt = t - d.tile_base;
    const int px = (int)(lt % (uint32_t)d.TX) * kTile + (threadIdx.x & 15);
    const int py = (int)(lt / (uint32_t)d.TX) * kTile + (threadIdx.x >> 4);
    float l = 0.0f;
    if (px < d.W && py < d.H) {
        const int64_t HW = (int64_t)d.W * d.H, off = (int64_t)py * d.W + px, pix = d.pix_base + off;
        const float e = a.err[pix];
        const float thr = 50.0f * a.med[vp];
        const bool in = a.n_valid[vp] > 0 && __float_as_uint(e) < kInfBits && e <= thr;
        const float al = 1.0f - a.t_final[pix];
        const float w = in ? al * al * al : 0.0f;
        if (in)
            l = w * (d.lambda_c * a.col[pix] + (1.0f - d.lambda_c) * e);
        if (a.w)
            a.w[pix] = w;
        if (a.inlier)
            a.inlier[pix] = in ? 1 : 0;
        auto sg = [](float x) -> float { return x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f); };
        if (a.d_rgb)
            for (int ch = 0; ch < 3; ++ch) {
                const int64_t q = 3 * d.pix_base + ch * HW + off;
                a.d_rgb[q] = w * d.lambda_c * sg(a.rgb[q] - d.t_rgb[ch * HW + off]);
            }
        if (a.d_depth)
            a.d_depth[pix] = w * (1.0f - d.lambda_c) * sg(a.depth[pix] - d.t_depth[off]);
    }
    l = warp_sum(l);
    if ((threadIdx.x & 31) == 0)
        s_red[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int w = 0; w < 8; ++w)
            s += s_red[w];
        a.tile_loss[t] = s;
    }
}

// depth error and colour L1 of rendered images (tracking keyframes)
__global__ void k_track_prep(const gsl::TrackArgs a, const float *rgb, const float *depth, float *err, float *col)
{
    const uint32_t t = blockIdx.x;
    const VpDesc &d = a.vps[a.tile_vp[t]];
    if (d.loss_kind != 1)
        return;
    const uint32_t lt = t - d.tile_base;
    const int px = (int)(lt % (uint32_t)d.TX) * kTile + (threadIdx.x & 15);
    const int py = (int)(lt / (uint32_t)d.TX) * kTile + (threadIdx.x >> 4);
    if (px >= d.W || py >= d.H)
        return;
    const int64_t HW = (int64_t)d.W * d.H, off = (int64_t)py * d.W + px, pix = d.pix_base + off;
    const float ed = depth[pix] - d.t_depth[off];
    err[pix] = d.t_depth[off] > 0.0f ? fabsf(ed) : __uint_as_float(kInfBits);
    float c = 0.0f;
    for (int ch = 0; ch < 3; ++ch)
        c += fabsf(rgb[3 * d.pix_base + ch * HW + off] - d.t_rgb[ch * HW + off]);
    col[pix] = c;
}

}  // namespace

namespace gsl {

void track_loss(const TrackArgs &a, cudaStream_t s)
{
    if (a.n_track <= 0 || a.n_tiles == 0)
        return;
    track_median(a, s);
    track_tiles(a, s);
}

void track_median(const TrackArgs &a, cudaStream_t s)
{
    launch_pdl(k_track_median, a.n_track * kMedCluster, kMedThreads, 0, s, a);
}

void track_tiles(const TrackArgs &a, cudaStream_t s) { launch_pdl(k_track_loss, a.n_tiles, 256, 0, s, a); }

void track_prep(const TrackArgs &a, const float *rgb, const float *depth, float *err, float *col, cudaStream_t s)
{
    if (a.n_tiles == 0)
        return;
    k_track_prep<<<a.n_tiles, 256, 0, s>>>(a, rgb, depth, err, col);
    ++g_launches;
}

}  // namespace gsl
