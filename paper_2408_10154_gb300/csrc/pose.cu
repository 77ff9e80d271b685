// pose.cu -- per-keyframe reductions and the on-device registration step:
// tile twists -> 6-vector per keyframe (FP32 TwoSum pairs in a fixed
// order, one FP64 value per component),
// Adam on the twist with a cosine-decayed learning rate, exponential-map
// pose update about the moving submap's centroid (Sec. 3.2; learning rates
// Supp. B), the standalone L1 loss, the Eq. 7 fusion and the Eq. 8/9 rigid
// transform of a submap.  Latency-bound tiny kernels, FP64 state.
#include <algorithm>
#include <cmath>

#include "gs_internal.cuh"

namespace {

using namespace gsk;

// exp([w]x) = I + a [w]x + b [w]x^2
__device__ __forceinline__ void so3_coef(const double *w, double &a, double &b)
{
    const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    const double th = sqrt(th2);
    if (th < 1e-8) {
        a = 1.0 - th2 / 6.0;
        b = 0.5 - th2 / 24.0;
    } else {
        double sn, cs;
        sincos(th, &sn, &cs);
        a = sn / th;
        b = (1.0 - cs) / th2;
    }
}

// entry (i, j) of [w]x
__device__ __forceinline__ double skew(const double *w, int i, int j)
{
    if (i == j)
        return 0.0;
    const double x = w[3 - i - j];
    return (j - i + 3) % 3 == 1 ? -x : x;
}

__device__ __forceinline__ double so3_entry(const double *w, double a, double b, int i, int j)
{
    const double k2 = skew(w, i, 0) * skew(w, 0, j) + skew(w, i, 1) * skew(w, 1, j) + skew(w, i, 2) * skew(w, 2, j);
    return (i == j ? 1.0 : 0.0) + a * skew(w, i, j) + b * k2;
}

// b^n for a step count n >= 1 (binary powering: a few multiplies instead of
// a general pow, whose FP64 log/exp chain is long on this part)
__device__ __forceinline__ double pow_count(double b, double n)
{
    unsigned long long m = (unsigned long long)n;
    double r = 1.0, x = b;
    while (m) {
        if (m & 1ull)
            r *= x;
        x *= x;
        m >>= 1;
    }
    return r;
}

// Learning-rate schedule of iteration k in [0, iters).
__device__ __forceinline__ double cosine_schedule(int k, int iters, float lr_final)
{
    const double kPi = 3.14159265358979323846;
    const double f = lr_final;
    return f + (1.0 - f) * 0.5 * (1.0 + cos(kPi * (double)k / (double)iters));
}

// Adam step with gradient gi, learning rate lr and the bias corrections
// bc = 1 - b^t: updates the moments m, v and returns the step.
__device__ __forceinline__ double adam_step(double &m, double &v, double gi, double lr, double bc1, double bc2, float b1f,
                                            float b2f, float epsf)
{
    const double b1 = b1f, b2 = b2f, eps = epsf;
    m = b1 * m + (1.0 - b1) * gi;
    v = b2 * v + (1.0 - b2) * gi * gi;
    const double mh = m / bc1;
    const double vh = v / bc2;
    return -lr * mh / (sqrt(vh) + eps);
}

// Pose update by the step xi about pivot c:
// R <- exp(-s_w) R, t <- exp(-s_w)(t - c) + c - s_v (xi carries the signs).
__device__ void exp_update(double *pose, const double *xi, const double *c)
{
    double dR[3][3], ca, cb;
    so3_coef(xi, ca, cb);
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            dR[i][j] = so3_entry(xi, ca, cb, i, j);
    double R[3][3], tt[3];
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j)
            R[i][j] = pose[4 * i + j];
        tt[i] = pose[4 * i + 3];
    }
    const double rel[3] = {tt[0] - c[0], tt[1] - c[1], tt[2] - c[2]};
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j)
            pose[4 * i + j] = dR[i][0] * R[0][j] + dR[i][1] * R[1][j] + dR[i][2] * R[2][j];
        pose[4 * i + 3] = dR[i][0] * rel[0] + dR[i][1] * rel[1] + dR[i][2] * rel[2] + c[i] + xi[3 + i];
    }
}

// Adam step on the twist g (about pivot c) and the pose update, serially;
// st[12] counts the steps taken
__device__ void adam_exp_update(double *pose, double *st, const double *g, const double *c, int k, int iters,
                                float lr_rot, float lr_trans, float b1f, float b2f, float epsf, float lr_final)
{
    const double t = st[12] + 1.0;
    const double sched = cosine_schedule(k, iters, lr_final);
    const double bc1 = 1.0 - pow_count(b1f, t), bc2 = 1.0 - pow_count(b2f, t);
    double xi[6];
    for (int i = 0; i < 6; ++i)
        xi[i] = adam_step(st[i], st[6 + i], g[i], (i < 3 ? (double)lr_rot : (double)lr_trans) * sched, bc1, bc2, b1f,
                          b2f, epsf);
    st[12] = t;
    exp_update(pose, xi, c);
}

// pivot = R mu_bar + t (world) and its camera-frame image for keyframe d
__device__ void pivots_of(const VpDesc &d, const double *pose, const double *mbar, double *piv, double *ccam)
{
    for (int i = 0; i < 3; ++i)
        piv[i] = pose[4 * i] * mbar[0] + pose[4 * i + 1] * mbar[1] + pose[4 * i + 2] * mbar[2] + pose[4 * i + 3];
    for (int i = 0; i < 3; ++i)
        ccam[i] = (double)d.w2c[4 * i] * piv[0] + (double)d.w2c[4 * i + 1] * piv[1] + (double)d.w2c[4 * i + 2] * piv[2] +
                  (double)d.w2c[4 * i + 3];
}

// Mean of each Gaussian set's means: 1024 running sums of two interleaved
// FP32 TwoSum chains each, TwoSum butterflies over warps of 32 and a
// fixed-order TwoSum of the 32 warps (in k_pose_init), one FP64 division
// (FP64 sums over 10^5 means were latency-bound on the slow FP64 pipe).
// One CTA per warp of the set, kCentUnroll pairs of loads in flight: the 32
// warps on one SM took 75 us for 150k means (ncu), two loads in flight each.
constexpr int kCentWarps = gsl::kCentroidWarps, kCentSums = 32 * kCentWarps, kCentUnroll = 8;

__global__ void __launch_bounds__(32) k_centroid(const VpDesc *vps, const int *set_vp, float2 *part)
{
    const VpDesc &d = vps[set_vp[blockIdx.y]];
    const int n = d.n;
    const float4 *means = d.means;
    float hs[2][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}}, ls[2][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
    auto add = [&](int c, const float4 &m) {
        two_sum_add(hs[c][0], ls[c][0], m.x, 0.0f);
        two_sum_add(hs[c][1], ls[c][1], m.y, 0.0f);
        two_sum_add(hs[c][2], ls[c][2], m.z, 0.0f);
    };
    int64_t i = 32 * blockIdx.x + threadIdx.x;
    for (; i + (2 * kCentUnroll - 1) * kCentSums < n; i += 2 * kCentUnroll * kCentSums) {
        float4 m[2 * kCentUnroll];
#pragma unroll
        for (int u = 0; u < 2 * kCentUnroll; ++u)
            m[u] = means[i + u * kCentSums];
#pragma unroll
        for (int u = 0; u < 2 * kCentUnroll; ++u)
            add(u & 1, m[u]);
    }
    for (; i + kCentSums < n; i += 2 * kCentSums) {
        const float4 m0 = means[i], m1 = means[i + kCentSums];
        add(0, m0);
        add(1, m1);
    }
    if (i < n)
        add(0, means[i]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float h = hs[0][k], l = ls[0][k];
        two_sum_add(h, l, hs[1][k], ls[1][k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float bh = __shfl_xor_sync(0xffffffffu, h, o), bl = __shfl_xor_sync(0xffffffffu, l, o);
            two_sum_add(h, l, bh, bl);
        }
        if (threadIdx.x == 0)
            part[(blockIdx.y * kCentWarps + blockIdx.x) * 3 + k] = make_float2(h, l);
    }
}

__global__ void k_pose_init(const gsl::PoseArgs a)
{
    const int vp = blockIdx.x * blockDim.x + threadIdx.x;
    if (vp >= a.n_vps)
        return;
    {
        // the set's centroid, joined by every keyframe that needs it and
        // kept by the set's first (a set's keyframes are consecutive)
        const VpDesc &d = a.vps[vp];
        const float2 *part = a.cent_part + (size_t)d.set * kCentWarps * 3;
        float h[3], l[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            h[k] = part[k].x;
            l[k] = part[k].y;
        }
#pragma unroll 8
        for (int w = 1; w < kCentWarps; ++w)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float2 v = part[3 * w + k];
                two_sum_add(h[k], l[k], v.x, v.y);
            }
        double mbar[3];
        for (int k = 0; k < 3; ++k)
            mbar[k] = d.n > 0 ? ((double)h[k] + (double)l[k]) / d.n : 0.0;
        if (vp == 0 || a.vps[vp - 1].set != d.set)
            for (int k = 0; k < 3; ++k)
                a.centroid[3 * d.set + k] = mbar[k];
        double I[12];
        for (int k = 0; k < 12; ++k)
            I[k] = (k % 5 == 0) ? 1.0 : 0.0;
        pivots_of(d, I, mbar, a.pivot + 3 * vp, a.c_cam + 3 * vp);
    }
    double *P = a.pose64 + 12 * vp;
    for (int k = 0; k < 12; ++k) {
        P[k] = (k % 5 == 0) ? 1.0 : 0.0;
        a.pose32[12 * vp + k] = (float)P[k];
    }
    for (int k = 0; k < 13; ++k)
        a.adam[13 * vp + k] = 0.0;
    if (a.expo) {
        for (int k = 0; k < 7; ++k)
            a.expo[7 * vp + k] = 0.0;
        a.expo32[2 * vp] = 1.0f;
        a.expo32[2 * vp + 1] = 0.0f;
    }
}

// 1024 threads per block: a keyframe's 3,225 tile pairs (1200x680) are
// about three loads deep per thread (256 threads waited on thirteen).
constexpr int kPoseThreads = 1024, kPoseWarps = kPoseThreads / 32;

// One block per keyframe: reduce the tile twists and losses in a fixed
// order, rotate the twist to the world frame, then (update) take the step.
// Bound by the latency of the step's FP64 chain (this part issues an FP64
// instruction of a warp every 16 clocks): so what needs no gradient -- the
// schedule's cosine and the bias corrections -- is found by other warps
// while the tiles are summed, and the 3x3 products of the exponential map
// run one entry per lane instead of all on one.  Each entry's operations
// and their order are those of exp_update.
__global__ void __launch_bounds__(kPoseThreads) k_pose_update(const gsl::PoseArgs a)
{
    __shared__ float s[kPoseWarps][9][2];
    __shared__ double s_tot[9], s_g[6], s_xi[6], s_pre[5], s_dR[9], s_P[12];
    const int vp = blockIdx.x;
    const VpDesc &d = a.vps[vp];
    const uint32_t nt = (uint32_t)d.TX * d.TY;
    const bool expo = d.exposure && a.tile_expo && a.expo;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // (a gradient-only caller has neither pose nor optimiser state)
    const bool update = a.update && a.tile_twist;
    const int iters = d.iters > 0 ? d.iters : a.iters;
    double *st = update ? a.adam + 13 * vp : nullptr;
    // warp 0's operands of the step, loaded ahead of the sums
    double m = 0.0, v = 0.0, P0 = 0.0, taken = 0.0;
    if (update && (warp == 0 || warp >= kPoseWarps - 5)) {
        taken = st[12];
        if (warp == 0 && lane < 6) {
            m = st[lane];
            v = st[6 + lane];
        }
        if (warp == 0 && lane < 12)
            P0 = a.pose64[12 * vp + lane];
    }
    if (update && (int)taken < iters) {
        // s_pre: schedule, 1 - b1^t, 1 - b2^t of the pose and of the exposure
        if (warp == kPoseWarps - 1 && lane == 0)
            s_pre[0] = cosine_schedule((int)taken, iters, a.lr_final);
        if (warp == kPoseWarps - 2 && lane == 0)
            s_pre[1] = 1.0 - pow_count(a.beta1, taken + 1.0);
        if (warp == kPoseWarps - 3 && lane == 0)
            s_pre[2] = 1.0 - pow_count(a.beta2, taken + 1.0);
        if (expo && warp == kPoseWarps - 4 && lane == 0)
            s_pre[3] = 1.0 - pow((double)a.beta1, a.expo[7 * vp + 6] + 1.0);
        if (expo && warp == kPoseWarps - 5 && lane == 0)
            s_pre[4] = 1.0 - pow((double)a.beta2, a.expo[7 * vp + 6] + 1.0);
    }
    pdl_wait();  // (what is above reads only the state of the update before)
    // (hi, lo) FP32 pairs summed by TwoSum in a fixed order (per thread,
    // then butterflies, then the warps); one FP64 value per component.  A
    // warp without tiles holds zeros, which leave a TwoSum as it is.
    const int nw = (int)min((nt + 31) / 32, (uint32_t)kPoseWarps);
    if (warp < nw) {
        float hs[9], ls[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            hs[i] = ls[i] = 0.0f;
#pragma unroll 4
        for (uint32_t k = threadIdx.x; k < nt; k += blockDim.x) {
            const size_t t = d.tile_base + k;
            if (a.tile_twist)
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const float2 w = a.tile_twist[t * 6 + i];
                    two_sum_add(hs[i], ls[i], w.x, w.y);
                }
            two_sum_add(hs[6], ls[6], a.tile_loss[t], 0.0f);
            if (expo) {
                two_sum_add(hs[7], ls[7], a.tile_expo[2 * t], 0.0f);
                two_sum_add(hs[8], ls[8], a.tile_expo[2 * t + 1], 0.0f);
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if ((i < 6 && !a.tile_twist) || (i > 6 && !expo))
                continue;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float bh = __shfl_xor_sync(0xffffffffu, hs[i], o), bl = __shfl_xor_sync(0xffffffffu, ls[i], o);
                two_sum_add(hs[i], ls[i], bh, bl);
            }
            if (lane == 0) {
                s[warp][i][0] = hs[i];
                s[warp][i][1] = ls[i];
            }
        }
    }
    __syncthreads();
    if (warp != 0)
        return;
    if (lane < 9 && (lane >= 6 || a.tile_twist) && (lane <= 6 || expo)) {
        float h = s[0][lane][0], l = s[0][lane][1];
#pragma unroll 8
        for (int w = 1; w < nw; ++w)
            two_sum_add(h, l, s[w][lane][0], s[w][lane][1]);
        s_tot[lane] = (double)h + (double)l;
        if (lane == 6)
            a.loss[vp] = s_tot[6];
    }
    if (!a.tile_twist)
        return;
    __syncwarp();
    // camera frame -> world frame: w = Rv^T w_c, v = Rv^T v_c
    double gi = 0.0;
    if (lane < 6) {
        const int r = lane % 3, o = lane < 3 ? 0 : 3;
        gi = (double)d.w2c[r] * s_tot[o] + (double)d.w2c[4 + r] * s_tot[o + 1] + (double)d.w2c[8 + r] * s_tot[o + 2];
        if (a.grad)
            a.grad[6 * vp + lane] = gi;
    }
    if (!update)
        return;
    const int k = (int)taken;
    if (k >= iters)
        return;
    if (lane < 6) {
        s_xi[lane] = adam_step(m, v, gi, (lane < 3 ? (double)d.lr_rot : (double)d.lr_trans) * s_pre[0], s_pre[1],
                               s_pre[2], a.beta1, a.beta2, a.eps);
        st[lane] = m;
        st[6 + lane] = v;
    }
    if (lane < 12)
        s_P[lane] = P0;
    if (lane == 6)
        st[12] = taken + 1.0;
    __syncwarp();
    // R <- exp(xi_w) R, t <- exp(xi_w)(t - c) + c + xi_v (exp_update), entry
    // (i, j) on lane 3 i + j, then on lane 4 i + j
    double ca, cb;
    so3_coef(s_xi, ca, cb);
    if (lane < 9)
        s_dR[lane] = so3_entry(s_xi, ca, cb, lane / 3, lane % 3);
    __syncwarp();
    const double *c = a.pivot + 3 * vp;
    double Pn = 0.0;
    if (lane < 12) {
        const int i = lane >> 2, j = lane & 3;
        double q[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            q[r] = s_P[4 * r + j];
            if (j == 3)
                q[r] = q[r] - c[r];
        }
        Pn = s_dR[3 * i] * q[0] + s_dR[3 * i + 1] * q[1] + s_dR[3 * i + 2] * q[2];
        if (j == 3)
            Pn = Pn + c[i] + s_xi[3 + i];
    }
    __syncwarp();
    if (lane < 12) {
        s_P[lane] = Pn;
        a.pose64[12 * vp + lane] = Pn;
        a.pose32[12 * vp + lane] = (float)Pn;
    }
    if (expo && (lane == 16 || lane == 17)) {
        // Adam on the exposure (a, b) with the pose's schedule; e = a, b,
        // m_a, m_b, v_a, v_b, steps taken
        const int i = lane - 16;
        double *e = a.expo + 7 * vp;
        const double t = e[6] + 1.0;
        double em = e[2 + i], ev = e[4 + i];
        const double b1 = a.beta1, b2 = a.beta2, eps = a.eps, g = s_tot[7 + i];
        em = b1 * em + (1.0 - b1) * g;
        ev = b2 * ev + (1.0 - b2) * g * g;
        const double mh = em / s_pre[3], vh = ev / s_pre[4];
        double x = e[i];
        x -= (double)d.lr_exposure * s_pre[0] * mh / (sqrt(vh) + eps);
        e[i] = x;
        e[2 + i] = em;
        e[4 + i] = ev;
        a.expo32[2 * vp + i] = i == 0 ? (float)exp(x) : (float)x;
        __syncwarp(0x30000u);  // both lanes have read the count
        if (i == 0)
            e[6] = t;
    }
    __syncwarp();
    // the pivot R mu_bar + t and its camera-frame image (pivots_of)
    if (lane < 3) {
        const double *mb = a.centroid + 3 * d.set;
        s_g[lane] = s_P[4 * lane] * mb[0] + s_P[4 * lane + 1] * mb[1] + s_P[4 * lane + 2] * mb[2] + s_P[4 * lane + 3];
        a.pivot[3 * vp + lane] = s_g[lane];
    }
    __syncwarp();
    if (lane < 3)
        a.c_cam[3 * vp + lane] = (double)d.w2c[4 * lane] * s_g[0] + (double)d.w2c[4 * lane + 1] * s_g[1] +
                                 (double)d.w2c[4 * lane + 2] * s_g[2] + (double)d.w2c[4 * lane + 3];
}

__global__ void k_expo32(const double *expo, float *expo32, int n)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) {
        expo32[2 * v] = (float)exp(expo[7 * v]);
        expo32[2 * v + 1] = (float)expo[7 * v + 1];
    }
}

__global__ void k_pose_step(int n, double *pose, double *state, const double *grad, const double *pivot, int k,
                            int iters, float lr_rot, float lr_trans, float b1, float b2, float eps, float lr_final)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    adam_exp_update(pose + 12 * i, state + 13 * i, grad + 6 * i, pivot + 3 * i, k, iters, lr_rot, lr_trans, b1, b2,
                    eps, lr_final);
}

// ---------------------------------------------------------------- fusion
__device__ void jacobi4(double A[4][4], double V[4][4])
{
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j)
            V[i][j] = i == j ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 30; ++sweep) {
        double off = 0.0;
        for (int p = 0; p < 4; ++p)
            for (int q = p + 1; q < 4; ++q)
                off += A[p][q] * A[p][q];
        if (off < 1e-60)
            break;
        for (int p = 0; p < 4; ++p)
            for (int q = p + 1; q < 4; ++q) {
                if (fabs(A[p][q]) < 1e-300)
                    continue;
                const double theta = (A[q][q] - A[p][p]) / (2.0 * A[p][q]);
                const double tt = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                const double c = 1.0 / sqrt(tt * tt + 1.0), s = tt * c;
                for (int k = 0; k < 4; ++k) {  // A <- J^T A J
                    const double akp = A[k][p], akq = A[k][q];
                    A[k][p] = c * akp - s * akq;
                    A[k][q] = s * akp + c * akq;
                }
                for (int k = 0; k < 4; ++k) {
                    const double apk = A[p][k], aqk = A[q][k];
                    A[p][k] = c * apk - s * aqk;
                    A[q][k] = s * apk + c * aqk;
                }
                for (int k = 0; k < 4; ++k) {
                    const double vkp = V[k][p], vkq = V[k][q];
                    V[k][p] = c * vkp - s * vkq;
                    V[k][q] = s * vkp + c * vkq;
                }
            }
    }
}

// Eigenvectors (columns of V) and eigenvalues (diagonal of A) of a symmetric
// 4x4 in FP32: cyclic Jacobi, unrolled so that everything stays in registers.
__device__ __forceinline__ void jacobi4_f32(float (&A)[4][4], float (&V)[4][4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            V[i][j] = i == j ? 1.0f : 0.0f;
    for (int sweep = 0; sweep < 6; ++sweep) {
        float off = 0.0f;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = p + 1; q < 4; ++q) {
                off += fabsf(A[p][q]);
                if (fabsf(A[p][q]) < 1e-30f)
                    continue;
                const float theta = (A[q][q] - A[p][p]) / (2.0f * A[p][q]);
                const float t = copysignf(1.0f, theta) / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.0f)));
                const float c = rsqrtf(fmaf(t, t, 1.0f)), s = t * c;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float x = A[k][p], y = A[k][q];
                    A[k][p] = c * x - s * y;
                    A[k][q] = s * x + c * y;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float x = A[p][k], y = A[q][k];
                    A[p][k] = c * x - s * y;
                    A[q][k] = s * x + c * y;
                    const float u = V[k][p], v = V[k][q];
                    V[k][p] = c * u - s * v;
                    V[k][q] = s * u + c * v;
                }
            }
        if (off < 1e-6f)
            break;
    }
}

// Top eigenvector of a symmetric 4x4: the FP32 eigenvectors, then FP64
// residuals corrected along the other three eigenvectors in FP32 (each step
// gains the FP32 factors' accuracy over the relative gap), until the
// residual is FP64's own.  Returns false (x unspecified) where that is not
// reached: a gap below 1e-3 of the largest entry, or values not finite.
__device__ __forceinline__ bool top_eigenvector4(const double (&K)[4][4], double (&x)[4])
{
    double scale = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            scale = fmax(scale, fabs(K[i][j]));
    if (!(scale > 0.0) || !(scale < 1e300))
        return false;
    const double inv = 1.0 / scale;
    float A[4][4], V[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            A[i][j] = (float)(K[i][j] * inv);
    jacobi4_f32(A, V);
    // the largest eigenvalue into column 0
#pragma unroll
    for (int i = 1; i < 4; ++i)
        if (A[i][i] > A[0][0]) {
            const float e = A[0][0];
            A[0][0] = A[i][i];
            A[i][i] = e;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float v = V[k][0];
                V[k][0] = V[k][i];
                V[k][i] = v;
            }
        }
    float g[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (!(A[0][0] - A[i + 1][i + 1] > 1e-3f))
            return false;
        g[i] = 1.0f / (A[0][0] - A[i + 1][i + 1]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        x[k] = V[k][0];
    for (int it = 0; it < 8; ++it) {
        double y[4], rho = 0.0, xx = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            y[i] = (K[i][0] * x[0] + K[i][1] * x[1] + K[i][2] * x[2] + K[i][3] * x[3]) * inv;
            rho += x[i] * y[i];
            xx += x[i] * x[i];
        }
        rho /= xx;
        float r[4], rmax = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            r[i] = (float)(y[i] - rho * x[i]);
            rmax = fmaxf(rmax, fabsf(r[i]));
        }
        if (rmax < 1e-15f)
            return true;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float w = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                w = fmaf(V[k][i + 1], r[k], w);
            w *= g[i];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                x[k] += (double)(w * V[k][i + 1]);
        }
    }
    return false;
}

// One warp per problem: weighted chordal L2 mean of the rotations (the
// quaternion maximising tr(R^T sum w_i R_i), i.e. the top eigenvector of
// Horn's symmetric 4x4 matrix) and weighted mean of the translations.  Lane
// 4 i + j sums entry (i, j) of the weighted estimates, in their order.
// Latency only: the FP64 Jacobi sweeps of one thread, whose arrays were
// indexed in local memory, took 92 to 385 us per call (ncu; most of it
// sweeps after convergence, their threshold being absolute); they remain
// for eigenvalues too close for the FP32 start.
__global__ void __launch_bounds__(32) k_fuse(const gsl::FuseArgs a)
{
    __shared__ double s_m[12];
    const int p = blockIdx.x, lane = threadIdx.x;
    const int first = a.prob_first[p], count = a.prob_count[p];
    const int i = lane >> 2, j = lane & 3;
    double sum = 0.0, wsum = 0.0;
    for (int e0 = first; e0 < first + count; e0 += 32) {
        const int n = min(32, first + count - e0);
        const double wl = lane < n ? 1.0 / fmax(a.eps[e0 + lane], 1e-12) : 0.0;
        for (int q = 0; q < n; ++q) {
            const int e = e0 + q;
            const double w = __shfl_sync(0xffffffffu, wl, q);
            if (lane < 12) {
                const double *src = a.pose64 + 12 * (size_t)e;
                double t;
                if (!a.reverse[e])
                    t = src[lane];
                else if (j < 3)
                    t = src[4 * j + i];
                else
                    t = -(src[i] * src[3] + src[4 + i] * src[7] + src[8 + i] * src[11]);
                if (a.est_out)
                    a.est_out[12 * (size_t)e + lane] = t;
                sum += w * t;
            }
            wsum += w;
        }
    }
    if (lane < 12)
        s_m[lane] = sum;
    __syncwarp();
    if (lane != 0)
        return;
    const double M[3][3] = {{s_m[0], s_m[1], s_m[2]}, {s_m[4], s_m[5], s_m[6]}, {s_m[8], s_m[9], s_m[10]}};
    double K[4][4] = {
        {M[0][0] + M[1][1] + M[2][2], M[2][1] - M[1][2], M[0][2] - M[2][0], M[1][0] - M[0][1]},
        {M[2][1] - M[1][2], M[0][0] - M[1][1] - M[2][2], M[0][1] + M[1][0], M[0][2] + M[2][0]},
        {M[0][2] - M[2][0], M[0][1] + M[1][0], -M[0][0] + M[1][1] - M[2][2], M[1][2] + M[2][1]},
        {M[1][0] - M[0][1], M[0][2] + M[2][0], M[1][2] + M[2][1], -M[0][0] - M[1][1] + M[2][2]}};
    double v[4];
    if (!top_eigenvector4(K, v)) {
        double V[4][4];
        jacobi4(K, V);
        int best = 0;
        for (int k = 1; k < 4; ++k)
            if (K[k][k] > K[best][best])
                best = k;
        for (int k = 0; k < 4; ++k)
            v[k] = V[k][best];
    }
    double w = v[0], x = v[1], y = v[2], z = v[3];
    const double nq = sqrt(w * w + x * x + y * y + z * z);
    w /= nq; x /= nq; y /= nq; z /= nq;
    double *T = a.T_out + 12 * (size_t)p;
    T[0] = 1 - 2 * (y * y + z * z); T[1] = 2 * (x * y - w * z); T[2] = 2 * (x * z + w * y);
    T[4] = 2 * (x * y + w * z); T[5] = 1 - 2 * (x * x + z * z); T[6] = 2 * (y * z - w * x);
    T[8] = 2 * (x * z - w * y); T[9] = 2 * (y * z + w * x); T[10] = 1 - 2 * (x * x + y * y);
    for (int r = 0; r < 3; ++r)
        T[4 * r + 3] = wsum > 0 ? s_m[4 * r + 3] / wsum : 0.0;
    a.conf[p] = count > 0 ? wsum / count : 0.0;
}

// ---------------------------------------------------------------- loss
constexpr int kLossTiles = 4;  // tiles per block: 32 loads of a thread in flight together

// L1 loss, its signs and the tiles' sums (each in one order: rows of the
// tile by warps of two, then the warps).  Bound by HBM once enough loads are
// in flight: one tile per block (8 loads a thread, a barrier behind them)
// took 48 us for four 1200x680 views, 48 B per pixel (23 us at the copy
// rate); four tiles take 32 us.
__global__ void __launch_bounds__(256) k_loss_tiles(const VpDesc *vps, const uint32_t *tile_vp, uint32_t n_tiles,
                                                    const float *rgb, const float *depth, float *d_rgb,
                                                    float *d_depth, float *tile_loss)
{
    __shared__ float s_red[kLossTiles][8];
    float x[kLossTiles][4], y[kLossTiles][4];
    bool in[kLossTiles];
    auto place = [&](int u, const VpDesc *&d, int64_t &HW, int64_t &off) {
        const uint32_t t = blockIdx.x * kLossTiles + u;
        if (t >= n_tiles)
            return false;
        d = &vps[tile_vp[t]];
        const uint32_t lt = t - d->tile_base;
        const int px = (int)(lt % (uint32_t)d->TX) * kTile + (threadIdx.x & 15);
        const int py = (int)(lt / (uint32_t)d->TX) * kTile + (threadIdx.x >> 4);
        HW = (int64_t)d->W * d->H;
        off = (int64_t)py * d->W + px;
        return px < d->W && py < d->H;
    };
#pragma unroll
    for (int u = 0; u < kLossTiles; ++u) {
        const VpDesc *d = nullptr;
        int64_t HW = 0, off = 0;
        in[u] = place(u, d, HW, off);
        if (!in[u])
            continue;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            x[u][ch] = rgb[3 * d->pix_base + ch * HW + off];
            y[u][ch] = d->t_rgb[ch * HW + off];
        }
        x[u][3] = depth[d->pix_base + off];
        y[u][3] = d->t_depth[off];
    }
    auto sg = [](float e) -> float { return e > 0.0f ? 1.0f : (e < 0.0f ? -1.0f : 0.0f); };
#pragma unroll
    for (int u = 0; u < kLossTiles; ++u) {
        float l = 0.0f;
        if (in[u]) {
            const VpDesc *d = nullptr;
            int64_t HW = 0, off = 0;
            place(u, d, HW, off);
            const float inv3 = d->inv3hw, inv1 = d->invhw;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                const float e = x[u][ch] - y[u][ch];
                l += fabsf(e) * inv3;
                if (d_rgb)
                    d_rgb[3 * d->pix_base + ch * HW + off] = sg(e) * inv3;
            }
            const float e = x[u][3] - y[u][3];
            l += fabsf(e) * inv1;
            if (d_depth)
                d_depth[d->pix_base + off] = sg(e) * inv1;
        }
        l = warp_sum(l);
        if ((threadIdx.x & 31) == 0)
            s_red[u][threadIdx.x >> 5] = l;
    }
    __syncthreads();
    if (threadIdx.x < kLossTiles && blockIdx.x * kLossTiles + threadIdx.x < n_tiles) {
        float s = 0.0f;
        for (int w = 0; w < 8; ++w)
            s += s_red[threadIdx.x][w];
        tile_loss[blockIdx.x * kLossTiles + threadIdx.x] = s;
    }
}

// ---------------------------------------------------------------- Eq. 8/9
// quaternion of R (largest-pivot branch), w >= 0
__host__ __device__ __forceinline__ void rigid_quat(const double *T, double &qw, double &qx, double &qy, double &qz)
{
    const double tr = T[0] + T[5] + T[10];
    if (tr > 0) {
        const double s = sqrt(tr + 1.0) * 2;
        qw = 0.25 * s; qx = (T[9] - T[6]) / s; qy = (T[2] - T[8]) / s; qz = (T[4] - T[1]) / s;
    } else if (T[0] > T[5] && T[0] > T[10]) {
        const double s = sqrt(1.0 + T[0] - T[5] - T[10]) * 2;
        qw = (T[9] - T[6]) / s; qx = 0.25 * s; qy = (T[1] + T[4]) / s; qz = (T[2] + T[8]) / s;
    } else if (T[5] > T[10]) {
        const double s = sqrt(1.0 + T[5] - T[0] - T[10]) * 2;
        qw = (T[2] - T[8]) / s; qx = (T[1] + T[4]) / s; qy = 0.25 * s; qz = (T[6] + T[9]) / s;
    } else {
        const double s = sqrt(1.0 + T[10] - T[0] - T[5]) * 2;
        qw = (T[4] - T[1]) / s; qx = (T[2] + T[8]) / s; qy = (T[6] + T[9]) / s; qz = 0.25 * s;
    }
}

// mu <- R mu + t and q <- q_R (x) q of one Gaussian in FP64, each result
// rounded once to FP32
__device__ __noinline__ void rigid_apply64(const double *T, const float4 m, const float4 q, float4 &om, float4 &oq)
{
    double qw, qx, qy, qz;
    rigid_quat(T, qw, qx, qy, qz);
    om.x = (float)(T[0] * m.x + T[1] * m.y + T[2] * m.z + T[3]);
    om.y = (float)(T[4] * m.x + T[5] * m.y + T[6] * m.z + T[7]);
    om.z = (float)(T[8] * m.x + T[9] * m.y + T[10] * m.z + T[11]);
    om.w = 0.0f;
    oq.x = (float)(qw * q.x - qx * q.y - qy * q.z - qz * q.w);
    oq.y = (float)(qw * q.y + qx * q.x + qy * q.w - qz * q.z);
    oq.z = (float)(qw * q.z - qx * q.w + qy * q.x + qz * q.y);
    oq.w = (float)(qw * q.w + qx * q.z - qy * q.y + qz * q.x);
}

// s + e = a + b exactly (Knuth), both lanes
__device__ __forceinline__ f32x2 two_sum2(f32x2 a, f32x2 b, f32x2 &e)
{
    const f32x2 s = add2(a, b), bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}

__device__ __forceinline__ f32x2 abs2(f32x2 v) { return v & 0x7fffffff7fffffffull; }

// c0 m0 + c1 m1 + c2 m2 + c3 m3 of two Gaussians (the lanes), c = ch + cl:
// products by fma, sums by TwoSum, their errors in L.  The value S + L is
// within 33 u^2 of the terms' magnitudes `mag` (u = 2^-24; the split of c,
// the products' and the sums' second-order roundings) plus underflows of
// 2^-149, so where S + L - e and S + L + e round alike with e = 2^-42 mag
// and mag >= 2^-100, that is the nearest FP32 value, and `sure` (per lane)
// stays set; so it does where every product is 0.
__device__ __forceinline__ f32x2 dot4_x2(const float *ch, const float *cl, const f32x2 (&m)[4], bool &sure0, bool &sure1)
{
    f32x2 S = 0, L = 0, mag = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const f32x2 c = bc2(ch[k]), p = mul2(c, m[k]);
        const f32x2 e = fma2(bc2(cl[k]), m[k], fma2(c, m[k], p ^ 0x8000000080000000ull));
        if (k == 0) {
            S = p;
            L = e;
            mag = abs2(p);
        } else {
            f32x2 r;
            S = two_sum2(S, p, r);
            L = add2(L, add2(e, r));
            mag = add2(mag, abs2(p));
        }
    }
    const f32x2 err = mul2(mag, bc2(2.2737368e-13f));  // 2^-42
    const f32x2 hi = add2(S, add2(L, err)), lo = add2(S, sub2(L, err));
    float h0, h1, l0, l1, g0, g1;
    x2_split(hi, h0, h1);
    x2_split(lo, l0, l1);
    x2_split(mag, g0, g1);
    constexpr float kTiny = 7.8886091e-31f;                  // 2^-100
    sure0 = sure0 && h0 == l0 && (g0 >= kTiny || g0 == 0.0f);  // (a NaN is not equal to itself)
    sure1 = sure1 && h1 == l1 && (g1 >= kTiny || g1 == 0.0f);
    return hi;
}

constexpr int kRigidThreads = 128, kRigidPairs = 2;  // two Gaussians per pair
constexpr int kRigidPerBlock = kRigidThreads * 2 * kRigidPairs;

// Eq. 8/9 of kRigidPerBlock Gaussians per block.  64 B of traffic per
// Gaussian against 25 FP64 operations in the plain form, which this part's
// FP64 pipe (two lanes per SM and clock) runs at a fifth of HBM's rate: with
// R's quaternion found per Gaussian as well, 4.4 M Gaussians took 661 us
// (ncu).  So the sums are taken in FP32 pairs (dot4_x2), packed two
// Gaussians at a time, and the few whose rounding that leaves open (about
// one in 10^4) in FP64: every result is FP64's rounded to FP32.  A call on 24
// maps of 4.4 M Gaussians in all: 665 -> 189 us, most of that the host's.
// Bound by the FP32 pipe (about 300 lane operations per Gaussian, 37 us) and
// HBM (42 us) in turn, so eight CTAs of 64 registers per SM for one to
// compute while another loads: 86 -> 70 us by ncu (five CTAs of 92 registers;
// one pair per thread 73-76, three or four 98-102).
__device__ __forceinline__ void rigid_block(const gsl::MapDesc &m, unsigned blk)
{
    const int64_t base = (int64_t)blk * kRigidPerBlock + threadIdx.x;
    float4 a[2 * kRigidPairs], q[2 * kRigidPairs];
#pragma unroll
    for (int u = 0; u < 2 * kRigidPairs; ++u) {
        const int64_t i = base + u * kRigidThreads;
        const bool in = i < m.n;
        a[u] = in ? m.means[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        q[u] = in ? m.quats[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    const float *qh = m.r.qh, *ql = m.r.ql;
    // rows of the quaternion product q_R (x) q
    const float ch[4][4] = {{qh[0], -qh[1], -qh[2], -qh[3]},
                            {qh[1], qh[0], -qh[3], qh[2]},
                            {qh[2], qh[3], qh[0], -qh[1]},
                            {qh[3], -qh[2], qh[1], qh[0]}};
    const float cl[4][4] = {{ql[0], -ql[1], -ql[2], -ql[3]},
                            {ql[1], ql[0], -ql[3], ql[2]},
                            {ql[2], ql[3], ql[0], -ql[1]},
                            {ql[3], -ql[2], ql[1], ql[0]}};
#pragma unroll
    for (int u = 0; u < kRigidPairs; ++u) {
        const float4 a0 = a[2 * u], a1 = a[2 * u + 1], q0 = q[2 * u], q1 = q[2 * u + 1];
        const f32x2 am[4] = {x2(a0.x, a1.x), x2(a0.y, a1.y), x2(a0.z, a1.z), bc2(1.0f)};
        const f32x2 qm[4] = {x2(q0.x, q1.x), x2(q0.y, q1.y), x2(q0.z, q1.z), x2(q0.w, q1.w)};
        bool sure[2] = {true, true};
        float rm[3][2], rq[4][2];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            x2_split(dot4_x2(m.r.Th + 4 * k, m.r.Tl + 4 * k, am, sure[0], sure[1]), rm[k][0], rm[k][1]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            x2_split(dot4_x2(ch[k], cl[k], qm, sure[0], sure[1]), rq[k][0], rq[k][1]);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int64_t i = base + (2 * u + v) * kRigidThreads;
            if (i >= m.n)
                continue;
            float4 om = make_float4(rm[0][v], rm[1][v], rm[2][v], 0.0f);
            float4 oq = make_float4(rq[0][v], rq[1][v], rq[2][v], rq[3][v]);
            if (!sure[v])
                rigid_apply64(m.r.T, a[2 * u + v], q[2 * u + v], om, oq);
            m.out_means[i] = om;
            m.out_quats[i] = oq;
        }
    }
}

__global__ void __launch_bounds__(kRigidThreads, 8) k_transform(const __grid_constant__ gsl::MapDesc m)
{
    rigid_block(m, blockIdx.x);
}

// many submaps, each with its own T: blocks [blk_base, next blk_base) of map k
__global__ void __launch_bounds__(kRigidThreads, 8) k_transform_batch(const gsl::MapDesc *maps, int n_maps)
{
    int lo = 0, hi = n_maps - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (maps[mid].blk_base <= blockIdx.x) lo = mid; else hi = mid - 1;
    }
    rigid_block(maps[lo], blockIdx.x - maps[lo].blk_base);
}

}  // namespace

namespace gsl {

void centroids(const VpDesc *vps, const int *set_vp, int n_sets, float2 *part, cudaStream_t s)
{
    // (grids are at most 65,535 high)
    for (int f = 0; f < n_sets; f += 32768) {
        k_centroid<<<dim3(kCentWarps, std::min(n_sets - f, 32768)), 32, 0, s>>>(vps, set_vp + f,
                                                                              part + (size_t)f * kCentWarps * 3);
        ++g_launches;
    }
}

void pose_init(const PoseArgs &a, cudaStream_t s)
{
    if (a.n_vps > 0) {
        k_pose_init<<<(a.n_vps + 127) / 128, 128, 0, s>>>(a);
        ++g_launches;
    }
}

void pose_update(const PoseArgs &a, cudaStream_t s)
{
    if (a.n_vps > 0)
        launch_pdl(k_pose_update, a.n_vps, kPoseThreads, 0, s, a);
}

void pose_step_raw(int n, double *pose, double *state, const double *grad, const double *pivot, int k, int iters,
                   float lr_rot, float lr_trans, float b1, float b2, float eps, float lr_final, cudaStream_t s)
{
    if (n > 0) {
        k_pose_step<<<(n + 127) / 128, 128, 0, s>>>(n, pose, state, grad, pivot, k, iters, lr_rot, lr_trans, b1, b2,
                                                    eps, lr_final);
        ++g_launches;
    }
}

void fuse(const FuseArgs &a, cudaStream_t s)
{
    if (a.n_problems > 0) {
        k_fuse<<<a.n_problems, 32, 0, s>>>(a);
        ++g_launches;
    }
}

void loss(const VpDesc *vps, int n_vps, uint32_t n_tiles, const uint32_t *tile_vp, const float *rgb,
          const float *depth, double *loss_out, float *d_rgb, float *d_depth, float *tile_loss, cudaStream_t s)
{
    if (n_tiles == 0)
        return;
    k_loss_tiles<<<(n_tiles + kLossTiles - 1) / kLossTiles, 256, 0, s>>>(vps, tile_vp, n_tiles, rgb, depth, d_rgb, d_depth,
                                                                        tile_loss);
    PoseArgs a{};
    a.vps = vps;
    a.n_vps = n_vps;
    a.tile_loss = tile_loss;
    a.loss = loss_out;
    k_pose_update<<<n_vps, kPoseThreads, 0, s>>>(a);
    g_launches += 2;
}

void exposure_floats(const double *expo, float *expo32, int n_vps, cudaStream_t s)
{
    if (n_vps <= 0)
        return;
    k_expo32<<<(n_vps + 127) / 128, 128, 0, s>>>(expo, expo32, n_vps);
    ++g_launches;
}

void loss_reduce(const VpDesc *vps, int n_vps, const float *tile_loss, double *loss_out, cudaStream_t s)
{
    if (n_vps <= 0)
        return;
    PoseArgs a{};
    a.vps = vps;
    a.n_vps = n_vps;
    a.tile_loss = tile_loss;
    a.loss = loss_out;
    k_pose_update<<<n_vps, kPoseThreads, 0, s>>>(a);
    ++g_launches;
}

Rigid make_rigid(const double *T)
{
    Rigid r;
    double q[4];
    rigid_quat(T, q[0], q[1], q[2], q[3]);
    for (int k = 0; k < 12; ++k) {
        r.T[k] = T[k];
        r.Th[k] = (float)T[k];
        r.Tl[k] = (float)(T[k] - (double)r.Th[k]);
    }
    for (int k = 0; k < 4; ++k) {
        r.qh[k] = (float)q[k];
        r.ql[k] = (float)(q[k] - (double)r.qh[k]);
    }
    // a coefficient whose low part would underflow sends every Gaussian to
    // FP64 (NaN sums are never sure)
    auto splits = [](double c) { return c == 0.0 || fabs(c) >= 7.8886090522101181e-31; };
    bool ok = true;
    for (int k = 0; k < 12; ++k)
        ok = ok && splits(T[k]);
    for (int k = 0; k < 4; ++k)
        ok = ok && splits(q[k]);
    if (!ok)
        r.Th[0] = NAN;
    return r;
}

unsigned transform_blocks(int64_t n) { return (unsigned)((n + kRigidPerBlock - 1) / kRigidPerBlock); }

void transform(const MapDesc &m, cudaStream_t s)
{
    if (m.n <= 0)
        return;
    k_transform<<<transform_blocks(m.n), kRigidThreads, 0, s>>>(m);
    ++g_launches;
}

void transform_batch(const MapDesc *maps, int n_maps, unsigned blocks, cudaStream_t s)
{
    if (n_maps <= 0 || blocks == 0)
        return;
    k_transform_batch<<<blocks, kRigidThreads, 0, s>>>(maps, n_maps);
    ++g_launches;
}

}  // namespace gsl
