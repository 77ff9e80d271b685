// params.cu -- the adjoint to every Gaussian parameter (the optional output
// of gs_render_backward): the adjoint kernel leaves each (tile, record)
// pair's screen gradients in the record's own slots, and one thread per
// Gaussian chains its records' sums, over the cameras in camera order,
// through the projection, the rigid transform (Eq. 8/9) and the scale /
// rotation / opacity parameterisation.  Fixed summation order, no atomics
// on the gradients.
#include <algorithm>

#include "gs_internal.cuh"

namespace {

using namespace gsk;

constexpr int kParamThreads = 128, kParamWarps = kParamThreads / 32;
constexpr uint32_t kShortSlots = 32;  // a record of more slots is summed by a warp of k_long_sums
constexpr int kStage = 64;            // slots staged at a time there (two per lane)

// First slot of every record's (tile, record) gradients: the record of tile
// rectangle [x0, x1) x [y0, y1) owns (x1 - x0)(y1 - y0) consecutive slots,
// one per tile in row-major order, so that the adjoint's tile CTA knows its
// slot from the record alone and nothing has to be sorted by record.  A
// block's records are consecutive; where the block's slots start follows
// the order in which the blocks ask (no result depends on it).
// Records of more than kShortSlots tiles are also listed (totals[1] of them).
__global__ void __launch_bounds__(kScanThreads) k_rec_slots(const int32_t *counts, uint32_t n, uint32_t *totals,
                                                           uint32_t *first, uint32_t *longs)
{
    __shared__ uint32_t s_warp[kScanThreads / 32 + 1];
    __shared__ uint32_t s_base;
    constexpr int K = kScanTile / kScanThreads;
    const uint32_t base = blockIdx.x * kScanTile + threadIdx.x * K;
    uint32_t c[K], sum = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        c[k] = base + k < n ? (uint32_t)counts[base + k] : 0u;
        sum += c[k];
    }
    uint32_t tot;
    uint32_t ex = block_excl_scan<kScanThreads>(sum, s_warp, tot);
    if (threadIdx.x == 0)
        s_base = tot ? atomicAdd(totals, tot) : 0u;
    __syncthreads();
    ex += s_base;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (c[k])
            first[base + k] = ex;
        if (c[k] > kShortSlots)
            longs[atomicAdd(totals + 1, 1u)] = base + k;
        ex += c[k];
    }
}

// The sum over a record's tiles runs in tile order (an FP32 sum of a splat
// over thousands of tiles cancels by 1e4, so another order shows at 1e-4 of
// the gradient), one lane per component.  A long record's is taken by a warp
// here, which stages 64 slots in shared memory while the next 64 are
// loading, and left in its first slot: a splat over a whole 1200x680 frame
// (3,225 slots) is a chain of 3,225 additions per component, and several of
// them in one block of k_param_grads, camera after camera, were its tail
// (300k Gaussians, 4 x 1200x680: 95 us in one kernel, 29 + 50 in two).
__global__ void __launch_bounds__(kParamThreads) k_long_sums(const uint32_t *totals, const uint32_t *longs,
                                                            const int32_t *counts, const uint32_t *first, float *dup)
{
    __shared__ __align__(16) float s_stage[kParamWarps][kStage * 12];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t n_long = totals[1];
    for (uint32_t l = blockIdx.x * kParamWarps + warp; l < n_long; l += gridDim.x * kParamWarps) {
        const uint32_t r = longs[l], n = (uint32_t)counts[r];
        float4 *p = reinterpret_cast<float4 *>(dup) + 3 * (size_t)first[r];
        float4 *st = reinterpret_cast<float4 *>(s_stage[warp]);
        // batch b: float4s [192 b, 192 b + 192) of the record's 3 n
        float4 v[6];
        const uint32_t n4 = 3 * n;
#pragma unroll
        for (int u = 0; u < 6; ++u)
            if (32u * u + lane < n4)
                v[u] = p[32 * u + lane];
        float G = 0.0f;
        for (uint32_t b = 0; b < n; b += kStage) {
#pragma unroll
            for (int u = 0; u < 6; ++u)
                st[32 * u + lane] = v[u];
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                const uint32_t q = 3 * (b + kStage) + 32 * u + lane;
                if (q < n4)
                    v[u] = p[q];
            }
            const int cntb = (int)min((uint32_t)kStage, n - b);
            if (lane < 10) {
#pragma unroll 8
                for (int k = 0; k < cntb; ++k)
                    G += s_stage[warp][12 * k + lane];
            }
            __syncwarp();
        }
        if (lane < 10)
            reinterpret_cast<float *>(p)[lane] = G;
    }
}

// One thread per Gaussian chains its records' gradients; a short record's
// sum over its tiles before that is taken by one lane per component, three
// records per warp, straight from its slots with several loads in flight.
// Most visible records cover a handful of tiles.  One thread summing its own
// records, each slot's load waiting for the last, took 646 us on the
// 300k-Gaussian, 4 x 1200x680 step (ncu), 33 MB or 5 us of HBM traffic, and
// grouping the slots by record took 14 launches of radix sort: the step's
// 1.86 ms became 1.21 with the slots alone.
__global__ void __launch_bounds__(kParamThreads) k_param_grads(const gsl::ParamArgs a)
{
    __shared__ float s_G[kParamThreads][10];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kParamThreads + threadIdx.x;
    const int comp = lane % 10, sub = lane / 10;  // lanes 30 and 31 sum nothing
    // object-frame accumulators over cameras
    float gmu[3] = {0, 0, 0}, GS[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}}, dop = 0.0f, drgb[3] = {0, 0, 0};
    for (int c = 0; c < a.n_vps; ++c) {
        const VpDesc &d = a.vps[c];
        const uint32_t r = d.rec_base + (uint32_t)i;
        uint32_t cnt = i < a.n ? (uint32_t)a.counts[r] : 0u;
        const uint32_t off = cnt ? a.rec_slot[r] : 0u;
        if (cnt > kShortSlots)
            cnt = 1;  // summed by k_long_sums
        unsigned m = __ballot_sync(0xffffffffu, cnt > 0);
        while (m) {
            int src = -1;
#pragma unroll
            for (int o = 0; o < 3; ++o) {
                const int f = __ffs(m) - 1;
                m &= m - 1;
                if (sub == o)
                    src = f;
            }
            const uint32_t n = __shfl_sync(0xffffffffu, cnt, src & 31), b = __shfl_sync(0xffffffffu, off, src & 31);
            if (src >= 0) {
                const float *p = a.dup_grads + 12 * (size_t)b + comp;
                float G = 0.0f;
#pragma unroll 8
                for (uint32_t k = 0; k < n; ++k)
                    G += p[12 * k];
                s_G[32 * warp + src][comp] = G;
            }
        }
        __syncwarp();
        float G[10];
#pragma unroll
        for (int k = 0; k < 10; ++k)
            G[k] = s_G[threadIdx.x][k];
        __syncwarp();  // (the next camera's sums take their place)
        if (cnt == 0)
            continue;
        const float4 q1 = a.rec[3 * (size_t)r + 1];
        const float4 x0 = a.aux[2 * (size_t)r], x1 = a.aux[2 * (size_t)r + 1];
        const float fx = d.fx, fy = d.fy;
        const float mx = x0.x, my = x0.y, mz = q1.z;
        const float S00 = x0.z, S01 = x0.w, S02 = x1.x, S11 = x1.y, S12 = x1.z, S22 = x1.w;
        // screen -> camera frame (the same chain as the pose adjoint)
        const float gp = 0.5f * G[2], gq = 0.5f * G[3], gs = 0.5f * G[4];
        const float iz = 1.0f / mz, iz2 = iz * iz;
        const float j00 = fx * iz, j11 = fy * iz, j02 = -fx * mx * iz2, j12 = -fy * my * iz2;
        const float r00 = gp * j00, r01 = gq * j11, r02 = gp * j02 + gq * j12;
        const float r10 = gq * j00, r11 = gs * j11, r12 = gq * j02 + gs * j12;
        const float Gc[3][3] = {{j00 * r00, j00 * r01, j00 * r02},
                                {j00 * r01, j11 * r11, j11 * r12},
                                {j00 * r02, j11 * r12, j02 * r02 + j12 * r12}};
        const float dJ00 = 2.0f * (r00 * S00 + r01 * S01 + r02 * S02);
        const float dJ02 = 2.0f * (r00 * S02 + r01 * S12 + r02 * S22);
        const float dJ11 = 2.0f * (r10 * S01 + r11 * S11 + r12 * S12);
        const float dJ12 = 2.0f * (r10 * S02 + r11 * S12 + r12 * S22);
        const float du = G[0], dv = G[1], dz = G[5];
        const float gm[3] = {du * fx * iz - dJ02 * fx * iz2, dv * fy * iz - dJ12 * fy * iz2,
                             -du * fx * mx * iz2 - dv * fy * my * iz2 + dz - dJ00 * fx * iz2 - dJ11 * fy * iz2 +
                                 2.0f * iz2 * iz * (dJ02 * fx * mx + dJ12 * fy * my)};
        // camera-from-object rotation M = V_R T_R of this camera and pose
        float M[3][3];
        const float *P = a.pose32 + 12 * c;
#pragma unroll
        for (int u = 0; u < 3; ++u)
#pragma unroll
            for (int v = 0; v < 3; ++v)
                M[u][v] = d.w2c[4 * u] * P[v] + d.w2c[4 * u + 1] * P[4 + v] + d.w2c[4 * u + 2] * P[8 + v];
        // object frame: g_mu = M^T g_m, G_Sigma = M^T Gc M
        float T1[3][3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            gmu[u] += M[0][u] * gm[0] + M[1][u] * gm[1] + M[2][u] * gm[2];
#pragma unroll
            for (int v = 0; v < 3; ++v)
                T1[u][v] = Gc[u][0] * M[0][v] + Gc[u][1] * M[1][v] + Gc[u][2] * M[2][v];
        }
#pragma unroll
        for (int u = 0; u < 3; ++u)
#pragma unroll
            for (int v = 0; v < 3; ++v)
                GS[u][v] += M[0][u] * T1[0][v] + M[1][u] * T1[1][v] + M[2][u] * T1[2][v];
        dop += G[6];
        drgb[0] += G[7];
        drgb[1] += G[8];
        drgb[2] += G[9];
    }
    if (i >= a.n)
        return;
    // Sigma = R(q) S^2 R(q)^T with S = diag(e^s); o = sigmoid(logit)
    const float4 q = a.quats[i], sc = a.scales[i];
    const float n2 = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
    const float ql = sqrtf(n2), iq = 1.0f / ql;
    const float w = q.x * iq, x = q.y * iq, y = q.z * iq, z = q.w * iq;
    const float R[3][3] = {{1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)},
                           {2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)},
                           {2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)}};
    const float sg2[3] = {expf(2.0f * sc.x), expf(2.0f * sc.y), expf(2.0f * sc.z)};
    // dL/ds_k = 2 sigma_k^2 (R^T G R)_kk ;  dL/dR = 2 G R S^2
    float GR[3][3];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v)
            GR[u][v] = GS[u][0] * R[0][v] + GS[u][1] * R[1][v] + GS[u][2] * R[2][v];
    float ds[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        ds[k] = 2.0f * sg2[k] * (R[0][k] * GR[0][k] + R[1][k] * GR[1][k] + R[2][k] * GR[2][k]);
    float dR[3][3];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v)
            dR[u][v] = 2.0f * GR[u][v] * sg2[v];
    // partial derivatives of R(q_hat) w.r.t. (w, x, y, z)
    const float gw = 2 * (-z * dR[0][1] + y * dR[0][2] + z * dR[1][0] - x * dR[1][2] - y * dR[2][0] + x * dR[2][1]);
    const float gx = 2 * (y * dR[0][1] + z * dR[0][2] + y * dR[1][0] - 2 * x * dR[1][1] - w * dR[1][2] + z * dR[2][0] +
                          w * dR[2][1] - 2 * x * dR[2][2]);
    const float gy = 2 * (-2 * y * dR[0][0] + x * dR[0][1] + w * dR[0][2] + x * dR[1][0] + z * dR[1][2] - w * dR[2][0] +
                          z * dR[2][1] - 2 * y * dR[2][2]);
    const float gz = 2 * (-2 * z * dR[0][0] - w * dR[0][1] + x * dR[0][2] + w * dR[1][0] - 2 * z * dR[1][1] +
                          y * dR[1][2] + x * dR[2][0] + y * dR[2][1]);
    // through q_hat = q / |q|
    const float dot = w * gw + x * gx + y * gy + z * gz;
    const float4 dq = make_float4((gw - w * dot) * iq, (gx - x * dot) * iq, (gy - y * dot) * iq, (gz - z * dot) * iq);
    const float o = 1.0f / (1.0f + expf(-a.logits[i]));
    if (a.g_means)
        reinterpret_cast<float4 *>(a.g_means)[i] = make_float4(gmu[0], gmu[1], gmu[2], 0.0f);
    if (a.g_scales)
        reinterpret_cast<float4 *>(a.g_scales)[i] = make_float4(ds[0], ds[1], ds[2], 0.0f);
    if (a.g_quats)
        reinterpret_cast<float4 *>(a.g_quats)[i] = dq;
    if (a.g_logits)
        a.g_logits[i] = dop * o * (1.0f - o);
    if (a.g_rgb)
        reinterpret_cast<float4 *>(a.g_rgb)[i] = make_float4(drgb[0], drgb[1], drgb[2], 0.0f);
}

inline uint32_t div_up(size_t a, size_t b) { return (uint32_t)((a + b - 1) / b); }

}  // namespace

namespace gsl {

size_t long_records(uint32_t cap) { return cap / (kShortSlots + 1) + 1; }

void rec_slots(const int32_t *counts, uint32_t n_records, uint32_t *totals, uint32_t *first, uint32_t *longs,
               cudaStream_t s)
{
    cudaMemsetAsync(totals, 0, 2 * sizeof(uint32_t), s);
    if (n_records == 0)
        return;
    k_rec_slots<<<div_up(n_records, kScanTile), kScanThreads, 0, s>>>(counts, n_records, totals, first, longs);
    ++g_launches;
}

void long_sums(const uint32_t *totals, const uint32_t *longs, uint32_t cap, const int32_t *counts, const uint32_t *first,
               float *dup_grads, cudaStream_t s)
{
    const uint32_t blocks = std::min<uint32_t>(div_up(long_records(cap), kParamWarps), 152 * 8);
    k_long_sums<<<blocks, kParamThreads, 0, s>>>(totals, longs, counts, first, dup_grads);
    ++g_launches;
}

void param_grads(const ParamArgs &a, cudaStream_t s)
{
    if (a.n <= 0)
        return;
    k_param_grads<<<div_up((size_t)a.n, kParamThreads), kParamThreads, 0, s>>>(a);
    ++g_launches;
}

}  // namespace gsl
