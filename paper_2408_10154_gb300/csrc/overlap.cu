// overlap.cu -- the overlap ratio of two submaps under an estimated
// T_{P->Q} (the supplement's loop filter): P's means are moved by T, each
// moved mean finds its closest mean of Q and each mean of Q its closest
// moved mean of P (exact nearest neighbours: FP32 squared distances
// dx = b - a per axis, fma(dz, dz, fma(dy, dy, dx * dx)), ties to the
// smaller index), the reciprocal pairs form the putative correspondences K,
// and OR = |{(p, q) in K : |T p - q|^2 < tau^2}| / |K|.
//
// k_nn is a brute-force sweep: targets staged through shared memory 2048 at
// a time (one broadcast load per target per warp), four queries per thread;
// FP32-ALU bound at ~9 operations per (query, target) pair.
//
// k_nn_grid searches a uniform grid over the targets instead: each query
// scans the 3x3x3 cells around its own, then the shells of cells at
// Chebyshev distance r = 2, 3, ..., and stops after shell r once its best
// squared distance is below (r s - margin)^2 (1 - 1e-6): a target outside
// the searched block lies at least r s - margin away (cell boundaries are
// computed in FP32 within the box), and its FP32 squared distance exceeds
// the best, so the result is the brute-force argmin whatever the grid.
// Queries that would need more than kNNMaxRing shells go to the brute-force
// sweep.  Both sets have a grid of the same cells, built by the same
// launches, and both directions are searched in one; the grid is chosen on
// the device, so nothing is read back before the end.
#include <cfloat>

#include <algorithm>

#include "gs_internal.cuh"

namespace {

constexpr int kNNMaxRing = 6;

constexpr int kNNThreads = 256;
constexpr int kNNQ = 4;        // queries per thread
constexpr int kNNChunk = 2048; // targets per shared-memory stage (32 KB)

struct Rigid32 {
    float T[12];
};

__device__ __forceinline__ float4 rigid32(const Rigid32 &T, const float4 &v)
{
    float r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        r[k] = __fmaf_rn(T.T[4 * k + 2], v.z,
                         __fmaf_rn(T.T[4 * k + 1], v.y, __fmaf_rn(T.T[4 * k], v.x, T.T[4 * k + 3])));
    return make_float4(r[0], r[1], r[2], 0.0f);
}

__global__ void k_rigid32(const float4 *p, int n, const __grid_constant__ Rigid32 T, float4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        out[i] = rigid32(T, p[i]);
}

__global__ void __launch_bounds__(kNNThreads) k_nn(const float4 *A, int na, const float4 *B, int nb, int32_t *nn,
                                                   float *d2)
{
    __shared__ float4 sb[kNNChunk];
    const int base = blockIdx.x * kNNThreads * kNNQ + threadIdx.x;
    float ax[kNNQ], ay[kNNQ], az[kNNQ], best[kNNQ];
    int bi[kNNQ];
#pragma unroll
    for (int q = 0; q < kNNQ; ++q) {
        const int i = base + q * kNNThreads;
        const float4 a = i < na ? A[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        ax[q] = a.x;
        ay[q] = a.y;
        az[q] = a.z;
        best[q] = __int_as_float(0x7f800000);
        bi[q] = -1;
    }
    for (int c0 = 0; c0 < nb; c0 += kNNChunk) {
        const int cnt = min(kNNChunk, nb - c0);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += kNNThreads)
            sb[k] = B[c0 + k];
        __syncthreads();
        for (int j = 0; j < cnt; ++j) {
            const float4 b = sb[j];
#pragma unroll
            for (int q = 0; q < kNNQ; ++q) {
                const float dx = __fsub_rn(b.x, ax[q]), dy = __fsub_rn(b.y, ay[q]), dz = __fsub_rn(b.z, az[q]);
                const float d = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
                if (d < best[q]) {  // strict: the first (smallest) index keeps a tie
                    best[q] = d;
                    bi[q] = c0 + j;
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kNNQ; ++q) {
        const int i = base + q * kNNThreads;
        if (i < na) {
            nn[i] = bi[q];
            if (d2)
                d2[i] = best[q];
        }
    }
}

// brute-force nearest neighbours of the queries listed in list[0 .. n_list)
// of each direction: blocks [0, blocks0) take direction 0
__global__ void __launch_bounds__(kNNThreads) k_nn_list(const gsl::OverlapArgs o, unsigned blocks0)
{
    const int dir = blockIdx.x >= blocks0 ? 1 : 0;
    const float4 *A = dir ? o.q : o.pt, *B = dir ? o.pt : o.q;
    const int nb = dir ? o.np : o.nq;
    const int32_t *list = o.list + (dir ? o.np : 0);
    int32_t *nn = dir ? o.nn_qp : o.nn_pq;
    float *d2 = dir ? nullptr : o.d2;
    const uint32_t nl = o.hdr->n_list[dir];
    const uint32_t base = (blockIdx.x - (dir ? blocks0 : 0)) * kNNThreads * kNNQ;
    if (base >= nl)
        return;
    __shared__ float4 sb[kNNChunk];
    float ax[kNNQ], ay[kNNQ], az[kNNQ], best[kNNQ];
    int bi[kNNQ];
#pragma unroll
    for (int q = 0; q < kNNQ; ++q) {
        const uint32_t i = base + q * kNNThreads + threadIdx.x;
        const float4 a = i < nl ? A[list[i]] : make_float4(0.f, 0.f, 0.f, 0.f);
        ax[q] = a.x;
        ay[q] = a.y;
        az[q] = a.z;
        best[q] = __int_as_float(0x7f800000);
        bi[q] = -1;
    }
    for (int c0 = 0; c0 < nb; c0 += kNNChunk) {
        const int cnt = min(kNNChunk, nb - c0);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += kNNThreads)
            sb[k] = B[c0 + k];
        __syncthreads();
        for (int j = 0; j < cnt; ++j) {
            const float4 b = sb[j];
#pragma unroll
            for (int q = 0; q < kNNQ; ++q) {
                const float dx = __fsub_rn(b.x, ax[q]), dy = __fsub_rn(b.y, ay[q]), dz = __fsub_rn(b.z, az[q]);
                const float d = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
                if (d < best[q]) {
                    best[q] = d;
                    bi[q] = c0 + j;
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kNNQ; ++q) {
        const uint32_t i = base + q * kNNThreads + threadIdx.x;
        if (i < nl) {
            nn[list[i]] = bi[q];
            if (d2)
                d2[list[i]] = best[q];
        }
    }
}

// float <-> order-preserving uint (for atomic min / max of floats)
__device__ __forceinline__ uint32_t f2o(float f)
{
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The grid over the box of both sets: about 1.8 cells per point of the
// larger one, at most max_cells and 2048 per axis.  F: float, or double
// where extents or their products leave float's range.
template <typename F>
__device__ bool choose_grid(const gsl::OverlapArgs &o, const float (&mn)[3], const float (&mx)[3], gsl::NNGrid &g)
{
    F lo[3], ext[3], emax = 0, amax = 0;
    for (int k = 0; k < 3; ++k) {
        lo[k] = (F)mn[k];
        ext[k] = (F)mx[k] - lo[k];
        emax = max(emax, ext[k]);
        amax = max(amax, max((F)fabsf(mn[k]), (F)fabsf(mx[k])));
    }
    const F pad = (F)1e-3 * emax + (F)1e-6;
    F lvol = 0;
    for (int k = 0; k < 3; ++k) {
        lo[k] -= pad;
        ext[k] = max(ext[k] + 2 * pad, pad);
        lvol += log2(ext[k]);
    }
    F cell = exp2((lvol - log2((F)1.8 * (F)max(o.np, o.nq))) / 3);
    cell = max(cell, (emax + 2 * pad) / 2048);
    int dims[3];
    for (int it = 0;; ++it) {
        double cells = 1.0;
        for (int k = 0; k < 3; ++k) {
            dims[k] = max(1, (int)min(ceil(ext[k] / cell), (F)4096));
            cells *= dims[k];
        }
        if (cells <= (double)o.max_cells)
            break;
        if (it > 200)
            return false;  // (not reached: the cells' number falls by 1.2 to 1.7 each time)
        cell *= (F)1.2;
    }
    g.ox = (float)lo[0];
    g.oy = (float)lo[1];
    g.oz = (float)lo[2];
    g.s = (float)cell;
    g.inv_s = 1.0f / g.s;
    g.nx = dims[0];
    g.ny = dims[1];
    g.nz = dims[2];
    g.margin = (float)((F)4e-6 * (emax + 2 * pad + amax) + (F)1e-7);
    return true;
}

__device__ void choose_grid(const gsl::OverlapArgs &o)
{
    float mn[3], mx[3], amax = 0.0f;
    bool ok = __ldcg(&o.hdr->bad) == 0;
    auto o2f = [](uint32_t u) { return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u); };
    for (int k = 0; k < 3; ++k) {
        mn[k] = o2f(~__ldcg(&o.hdr->box[k]));
        mx[k] = o2f(__ldcg(&o.hdr->box[3 + k]));
        amax = fmaxf(amax, fmaxf(fabsf(mn[k]), fabsf(mx[k])));
    }
    gsl::NNGrid g{};
    if (ok)
        ok = amax < 1e30f ? choose_grid<float>(o, mn, mx, g) : choose_grid<double>(o, mn, mx, g);
    o.hdr->grid = g;
    o.hdr->ok = ok ? 1 : 0;
}

// Moves P by T, finds the bounding box of the moved P and Q (as
// order-preserving integers; the minima complemented, so that the header
// starts at zero), and in the last block to finish chooses the grid.
__global__ void __launch_bounds__(256) k_moved_bbox(const gsl::OverlapArgs o, const __grid_constant__ Rigid32 T)
{
    uint32_t m[6] = {0, 0, 0, 0, 0, 0};
    bool bad = false;  // an infinity or NaN (whose bits the sign operations of f2o need not keep)
    const uint32_t n = (uint32_t)o.np + (uint32_t)o.nq;
    for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float4 v;
        if (i < (uint32_t)o.np) {
            v = rigid32(T, o.p[i]);
            o.pt[i] = v;
        } else {
            v = o.q[i - o.np];
        }
        const uint32_t c[3] = {f2o(v.x), f2o(v.y), f2o(v.z)};
        bad |= !(fabsf(v.x) <= FLT_MAX) || !(fabsf(v.y) <= FLT_MAX) || !(fabsf(v.z) <= FLT_MAX);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            m[k] = max(m[k], ~c[k]);
            m[3 + k] = max(m[3 + k], c[k]);
        }
    }
    // warp, then block (shared memory), then one atomic per block and bound
    // (an atomic per warp serialised ~10^4 of them on six addresses)
    __shared__ uint32_t s_m[6][8];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const uint32_t w = __reduce_max_sync(0xffffffffu, m[k]);
        if ((threadIdx.x & 31) == 0)
            s_m[k][threadIdx.x >> 5] = w;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(&o.hdr->bad, 1u);
    if (threadIdx.x < 6) {
        uint32_t w = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            w = max(w, s_m[threadIdx.x][j]);
        atomicMax(&o.hdr->box[threadIdx.x], w);
        __threadfence();
    }
    if (threadIdx.x >= 32)
        return;
    __syncwarp();
    if (threadIdx.x == 0 && atomicAdd(&o.hdr->blocks_done, 1u) == gridDim.x - 1) {
        __threadfence();
        choose_grid(o);
    }
}

__device__ __forceinline__ int cell_axis(float x, float o, float inv_s, int n)
{
    const float t = floorf(__fmul_rn(__fsub_rn(x, o), inv_s));
    return (int)fminf(fmaxf(t, 0.0f), (float)(n - 1));
}

__device__ __forceinline__ uint32_t cell_of(const gsl::NNGrid &g, const float4 &p)
{
    return (uint32_t)cell_axis(p.x, g.ox, g.inv_s, g.nx) +
           (uint32_t)g.nx * ((uint32_t)cell_axis(p.y, g.oy, g.inv_s, g.ny) +
                             (uint32_t)g.ny * (uint32_t)cell_axis(p.z, g.oz, g.inv_s, g.nz));
}

// counts of the cells of both sets (Q's after P's)
__global__ void __launch_bounds__(256) k_cell_count(const gsl::OverlapArgs o)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, np = (uint32_t)o.np;
    if (i >= np + (uint32_t)o.nq || !o.hdr->ok)
        return;
    const uint32_t c = cell_of(o.hdr->grid, i < np ? o.pt[i] : o.q[i - np]) + (i < np ? 0u : o.max_cells);
    o.cell[i] = c;
    atomicAdd(&o.count[c], 1u);
}

// Exclusive scan of the cell counts, two launches: sums of blocks of 2048
// cells, then every block adds the sums before its own (at most a few
// thousand) and scans.  Cells past the grid hold zeros.
constexpr int kCellTile = gsk::kScanTile, kCellThreads = gsk::kScanThreads, kCellPer = kCellTile / kCellThreads;

__global__ void __launch_bounds__(kCellThreads) k_cell_sums(const uint32_t *count, uint32_t n, uint32_t *sums)
{
    __shared__ uint32_t s[kCellThreads / 32];
    const uint32_t base = blockIdx.x * kCellTile + threadIdx.x;
    uint32_t acc = 0;
#pragma unroll
    for (int k = 0; k < kCellPer; ++k)
        acc += base + k * kCellThreads < n ? count[base + k * kCellThreads] : 0u;
    acc = __reduce_add_sync(0xffffffffu, acc);
    if ((threadIdx.x & 31) == 0)
        s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
#pragma unroll
        for (int w = 0; w < kCellThreads / 32; ++w)
            t += s[w];
        sums[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kCellThreads) k_cell_starts(uint32_t *count, uint32_t n, const uint32_t *sums,
                                                              uint32_t *start)
{
    __shared__ uint32_t s_warp[kCellThreads / 32 + 1], s_before[kCellThreads / 32];
    uint32_t before = 0;
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += kCellThreads)
        before += sums[b];
    before = __reduce_add_sync(0xffffffffu, before);
    if ((threadIdx.x & 31) == 0)
        s_before[threadIdx.x >> 5] = before;
    const uint32_t base = blockIdx.x * kCellTile + threadIdx.x * kCellPer;
    uint32_t v[kCellPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kCellPer; ++k) {
        v[k] = base + k < n ? count[base + k] : 0u;
        sum += v[k];
    }
    uint32_t tot;
    uint32_t ex = gsk::block_excl_scan<kCellThreads>(sum, s_warp, tot);
#pragma unroll
    for (int w = 0; w < kCellThreads / 32; ++w)
        ex += s_before[w];
#pragma unroll
    for (int k = 0; k < kCellPer; ++k) {
        if (base + k < n) {
            start[base + k] = ex;
            count[base + k] = ex;  // the scatter's cursor
        }
        ex += v[k];
    }
    if (base + kCellPer >= n && base < n)
        start[n] = ex;
}

// both sets bucketed by cell, the index in w (order within a cell
// arbitrary: ties are broken by index)
__global__ void __launch_bounds__(256) k_cell_scatter(const gsl::OverlapArgs o)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, np = (uint32_t)o.np;
    if (i >= np + (uint32_t)o.nq || !o.hdr->ok)
        return;
    float4 v = i < np ? o.pt[i] : o.q[i - np];
    v.w = __uint_as_float(i < np ? i : i - np);
    o.spts[atomicAdd(&o.count[o.cell[i]], 1u)] = v;
}

// One thread per query of either set, in cell order (neighbouring lanes
// search the same cells).  The cells x - r .. x + r of a row are one run of
// the sorted targets, so a row costs its two ends and then one 16 B load
// per target; the ends of the nine rows around the query are loaded
// together.  Bound by the latency of those loads.  Cell by cell, each with
// its own two ends and the targets' indices in a second array, the two
// directions took 152 and 138 us for 150k against 131k room points (ncu).
__global__ void __launch_bounds__(256) k_nn_grid(const gsl::OverlapArgs o)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (uint32_t)o.np + (uint32_t)o.nq || !o.hdr->ok)
        return;
    const gsl::NNGrid g = o.hdr->grid;
    const int dir = t >= (uint32_t)o.np ? 1 : 0;
    const float4 a = o.spts[t];
    const int i = __float_as_int(a.w);
    const uint32_t *start = o.start + (dir ? 0u : o.max_cells);  // the other set's cells
    const int cx = cell_axis(a.x, g.ox, g.inv_s, g.nx), cy = cell_axis(a.y, g.oy, g.inv_s, g.ny),
              cz = cell_axis(a.z, g.oz, g.inv_s, g.nz);
    float best = __int_as_float(0x7f800000);
    int bi = -1;
    auto scan_run = [&](uint32_t j0, uint32_t j1) {
#pragma unroll 2
        for (uint32_t j = j0; j < j1; ++j) {
            const float4 b = o.spts[j];
            const float dx = __fsub_rn(b.x, a.x), dy = __fsub_rn(b.y, a.y), dz = __fsub_rn(b.z, a.z);
            const float d = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
            const int idx = __float_as_int(b.w);
            if (d < best || (d == best && idx < bi)) {
                best = d;
                bi = idx;
            }
        }
    };
    // A row's targets are at least this far (squared): the gaps between the
    // query and the row's cells in y and z, less the margin of their
    // boundaries.  A row beyond the best so far is left out (a tie is not
    // beyond: it may hold the smaller index).
    const float fy = a.y - (g.oy + (float)cy * g.s), fz = a.z - (g.oz + (float)cz * g.s);
    auto gap = [&](int d, float f) {
        const float x = d > 0 ? (float)d * g.s - f : (d < 0 ? f - (float)(d + 1) * g.s : 0.0f);
        return fmaxf(x - g.margin, 0.0f);
    };
    auto row_dist2 = [&](int dy, int dz) {
        const float gy = gap(dy, fy), gz = gap(dz, fz);
        return (gy * gy + gz * gz) * (1.0f - 1e-6f);
    };
    auto row_of = [&](int y, int z) { return (uint32_t)g.nx * ((uint32_t)y + (uint32_t)g.ny * (uint32_t)z); };
    {
        const int x0 = max(cx - 1, 0), x1 = min(cx + 1, g.nx - 1);
        uint32_t j0[9], j1[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int y = cy + k % 3 - 1, z = cz + k / 3 - 1;
            const bool in = y >= 0 && y < g.ny && z >= 0 && z < g.nz;
            j0[k] = in ? start[row_of(y, z) + x0] : 0u;
            j1[k] = in ? start[row_of(y, z) + x1 + 1] : 0u;
        }
        // the query's own row first, then the others nearest first
        constexpr int kOrder[9] = {4, 1, 3, 5, 7, 0, 2, 6, 8};
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int k = kOrder[q];
            if (k == 4 || row_dist2(k % 3 - 1, k / 3 - 1) <= best)
                scan_run(j0[k], j1[k]);
        }
    }
    for (int r = 1;;) {
        const bool covered = cx - r <= 0 && cx + r >= g.nx - 1 && cy - r <= 0 && cy + r >= g.ny - 1 &&
                             cz - r <= 0 && cz + r >= g.nz - 1;
        const float lb = (float)r * g.s - g.margin;
        if (covered || (lb > 0.0f && best < lb * lb * (1.0f - 1e-6f)))
            break;
        if (r >= kNNMaxRing) {
            // far from every target: the brute-force sweep
            o.list[(dir ? (size_t)o.np : 0) + atomicAdd(&o.hdr->n_list[dir], 1u)] = i;
            return;
        }
        ++r;
        // the shell of cells at Chebyshev distance r (clipped to the grid)
        const int x0 = max(cx - r, 0), x1 = min(cx + r, g.nx - 1);
        for (int z = max(cz - r, 0); z <= min(cz + r, g.nz - 1); ++z)
            for (int y = max(cy - r, 0); y <= min(cy + r, g.ny - 1); ++y) {
                if (row_dist2(y - cy, z - cz) > best)
                    continue;
                const uint32_t row = row_of(y, z);
                if (z == cz - r || z == cz + r || y == cy - r || y == cy + r) {
                    scan_run(start[row + x0], start[row + x1 + 1]);
                } else {
                    if (cx - r >= 0)
                        scan_run(start[row + cx - r], start[row + cx - r + 1]);
                    if (cx + r < g.nx)
                        scan_run(start[row + cx + r], start[row + cx + r + 1]);
                }
            }
    }
    if (dir) {
        o.nn_qp[i] = bi;
    } else {
        o.nn_pq[i] = bi;
        o.d2[i] = best;
    }
}

// |K| and the pairs of K within tau (counts[0], counts[1])
__global__ void k_reciprocal(const int32_t *nn_pq, const float *d2, int np, const int32_t *nn_qp, float tau2,
                             unsigned long long *counts, const int *ok)
{
    if (ok && !*ok)
        return;  // (no neighbours were found)
    __shared__ unsigned s_k[8], s_in[8];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned k = 0, in = 0;
    if (i < np) {
        const int32_t j = nn_pq[i];
        if (j >= 0 && nn_qp[j] == i) {
            k = 1;
            in = d2[i] < tau2 ? 1u : 0u;
        }
    }
    k = __reduce_add_sync(0xffffffffu, k);
    in = __reduce_add_sync(0xffffffffu, in);
    if ((threadIdx.x & 31) == 0) {
        s_k[threadIdx.x >> 5] = k;
        s_in[threadIdx.x >> 5] = in;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long a = 0, b = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a += s_k[w];
            b += s_in[w];
        }
        if (a)
            atomicAdd(&counts[0], a);
        if (b)
            atomicAdd(&counts[1], b);
    }
}

inline unsigned div_up(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

}  // namespace

namespace gsl {

size_t overlap_sum_blocks(uint32_t max_cells) { return div_up(2 * (long long)max_cells, kCellTile); }

namespace {
Rigid32 rigid_arg(const OverlapArgs &a)
{
    Rigid32 T;
    for (int k = 0; k < 12; ++k)
        T.T[k] = a.T32[k];
    return T;
}
}  // namespace

void overlap_grid(const OverlapArgs &a, cudaStream_t s)
{
    const unsigned nb = div_up((long long)a.np + a.nq, 256);
    const uint32_t n_cells = 2 * a.max_cells;
    const unsigned sb = (unsigned)overlap_sum_blocks(a.max_cells);
    cudaMemsetAsync(a.hdr, 0, sizeof(NNHeader), s);
    cudaMemsetAsync(a.count, 0, sizeof(uint32_t) * (size_t)n_cells, s);
    k_moved_bbox<<<std::min<unsigned>(nb, 4 * 152), 256, 0, s>>>(a, rigid_arg(a));
    k_cell_count<<<nb, 256, 0, s>>>(a);
    k_cell_sums<<<sb, kCellThreads, 0, s>>>(a.count, n_cells, a.sums);
    k_cell_starts<<<sb, kCellThreads, 0, s>>>(a.count, n_cells, a.sums, a.start);
    k_cell_scatter<<<nb, 256, 0, s>>>(a);
    k_nn_grid<<<nb, 256, 0, s>>>(a);
    const unsigned b0 = div_up(a.np, kNNThreads * kNNQ), b1 = div_up(a.nq, kNNThreads * kNNQ);
    k_nn_list<<<b0 + b1, kNNThreads, 0, s>>>(a, b0);
    k_reciprocal<<<div_up(a.np, 256), 256, 0, s>>>(a.nn_pq, a.d2, a.np, a.nn_qp, a.tau2, a.hdr->counts,
                                                  &a.hdr->ok);
    g_launches += 8;
}

void overlap(const OverlapArgs &a, cudaStream_t s)
{
    cudaMemsetAsync(a.hdr, 0, sizeof(NNHeader), s);
    if (a.np > 0) {
        k_rigid32<<<div_up(a.np, 256), 256, 0, s>>>(a.p, a.np, rigid_arg(a), a.pt);
        k_nn<<<div_up(a.np, kNNThreads * kNNQ), kNNThreads, 0, s>>>(a.pt, a.np, a.q, a.nq, a.nn_pq, a.d2);
        g_launches += 2;
    }
    if (a.nq > 0) {
        k_nn<<<div_up(a.nq, kNNThreads * kNNQ), kNNThreads, 0, s>>>(a.q, a.nq, a.pt, a.np, a.nn_qp, nullptr);
        ++g_launches;
    }
    if (a.np > 0) {
        k_reciprocal<<<div_up(a.np, 256), 256, 0, s>>>(a.nn_pq, a.d2, a.np, a.nn_qp, a.tau2, a.hdr->counts,
                                                      nullptr);
        ++g_launches;
    }
}

}  // namespace gsl
