// probe.cuh -- a look at a problem before it is searched: what a walk per query
// would visit, and what the block search's tiles would have to settle exactly.
//
// A CTA per sampled query scores up to 1024 leaves, spread over the tree,
// and evaluates the points of a few of them; counts go out (the same in every
// call).  No chain of loads is longer than a few, so that the whole look costs
// little more than its read-back; a sample of walks would take as long as its
// longest walk.
#pragma once

#include "knn_tc.cuh"

namespace dt {

constexpr int kProbeThreads = 128, kProbeTop = 8, kProbeRangeTop = 16, kProbeRows = 64;

// The i-th of S strata of [0, n), at a place of its own in each (the first point or leaf
// of a subtree is in a corner of it).
__device__ __forceinline__ int64_t probe_pick(int i, int64_t n, int S) {
    const uint32_t width = (uint32_t)(n / S);
    return i * n / S + (width > 1 ? ((uint32_t)(i + 1) * 0x9e3779b1u >> 8) % width : 0u);
}

template <int DP>
__device__ __forceinline__ float probe_load(float (&q)[DP], const float* qp, const float* rbox) {
    // the query, and its distance from the reference root's centre
    float a2 = 0.f;
#pragma unroll
    for (int j = 0; j < DP / 4; ++j) {
        const float4 v = reinterpret_cast<const float4*>(qp)[j];
        q[4 * j] = v.x;
        q[4 * j + 1] = v.y;
        q[4 * j + 2] = v.z;
        q[4 * j + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < DP; ++j) {
        const float t = q[j] - 0.5f * (rbox[j] + rbox[DP + j]);
        a2 = fmaf(t, t, a2);
    }
    return sqrtf(a2);
}

// The CTA's counts (kept and near summed over its threads, pts the same in all);
// true for the first warp of the last CTA, which gets the totals.
__device__ __forceinline__ bool probe_total(const ProbeArgs& a, int kept, int near, int pts, int& all_kept,
                                            int& all_near, int& all_pts) {
    __shared__ int part[2][kProbeThreads / 32];
    __shared__ bool s_last;
    const int tid = threadIdx.x, lane = tid & 31;
    kept = __reduce_add_sync(0xffffffffu, kept);
    near = __reduce_add_sync(0xffffffffu, near);
    if (lane == 0) {
        part[0][tid >> 5] = kept;
        part[1][tid >> 5] = near;
    }
    __syncthreads();
    if (tid == 0) {
        kept = near = 0;
        for (int w = 0; w < kProbeThreads / 32; ++w) {
            kept += part[0][w];
            near += part[1][w];
        }
        a.out->kept[blockIdx.x] = kept;
        a.out->near[blockIdx.x] = near;
        a.out->pts[blockIdx.x] = pts;
        __threadfence();
        s_last = atomicAdd(&a.out->done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || tid >= 32) return false;
    __threadfence();
    int k = 0, n = 0, m = 0;  // (at most 1024 x 1024 per CTA, of 128)
    for (int q = lane; q < (int)gridDim.x; q += 32) {
        k += __ldcg(&a.out->kept[q]);
        n += __ldcg(&a.out->near[q]);
        m += __ldcg(&a.out->pts[q]);
    }
    all_kept = __reduce_add_sync(0xffffffffu, k);
    all_near = __reduce_add_sync(0xffffffffu, n);
    all_pts = __reduce_add_sync(0xffffffffu, m);
    return true;
}

// Whether the extents (the reference points' radius about their box centre, the
// queries' largest distance from it) keep squared distances, and the
// tensor-core keys' bounds relative to them, inside float32's range; radius is
// the larger of the two.  One warp.
template <int DP>
__device__ __forceinline__ bool probe_extents(const ProbeArgs& a, float& radius) {
    float c2 = 0.f;
    for (int j = threadIdx.x & 31; j < DP; j += 32) {
        const float t = 0.5f * (a.qbox[j] + a.qbox[DP + j]) - 0.5f * (a.rbox[j] + a.rbox[DP + j]);
        c2 += t * t;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, off);
    const float rl = a.rlam[0], qr = sqrtf(c2) + a.qlam[0];
    radius = fmaxf(qr, rl);
    return rl >= 1e-12f && rl <= 1e15f && qr <= 1e15f;
}

// The rule, from what a walk would visit of the reference tree per query (share
// of the leaves) and how many of the evaluated points the tile's band would hold
// (near).
//
// A walk per query visits few leaves where the points' intrinsic dimension is
// low, whatever the space they lie in, and then beats the tiles, whose blocks
// must visit what any of 128 queries needs.  Walks and tiles, by the share
// of the leaves: 300k x 50k points of d = 16 with three latent dimensions 0.1%, 0.77
// and 1.52 ms; with six 0.6%, 6.2 and 6.3; with ten 4.6%, 33 and 7.7; 1M x 20k of d =
// 32, four latent dimensions 0.1%, 1.4 and 6.8 ms; seven 0.7%, 11 and 16; eight 1.3%,
// 19 and 16; the mixture, d = 10, 1M x 100k 4%, 69 and 18 ms, d = 16, 1M x 200k 11%, 312
// and 41.  Few points in all: 20k x 100k, four latent dimensions 1.5%, 300 points,
// 1.5 and 1.8 ms; five 3.5%, 700, 2.7 and 2.1; 30k x 40k of d = 10 with three in 32
// leaves, of which a walk visits two, 1.1 and 1.5.  Lists of 64 (k > 18) cost the tiles
// half as much again, and few queries leave the GPU to the latency of either:
// mixture, d = 10, k = 30, 250k x 8,200, 20,000 points, 3.5 and 4.0 ms; 1M x 4,100,
// 51,000 points, 6.7 and 5.3; 250k x 16,400, 6.2 and 5.2.
// Where the band holds more than a list (equal or nearly equal distances), the
// tiles' work is done twice: queries at the centre of a sphere 16.8 against 14.2
// ms.  A healthy band holds about k points of all, or about one of those sampled.
template <int DP>
__device__ __forceinline__ bool far_by_tiles(const ProbeArgs& a, float share, float near) {
    const float leaves = share * (float)a.nleaves, points = share * (float)a.nr;
    const float scale = (float)a.nleaves / (float)a.leaves;  // leaves behind each scored one
    return share >= (DP <= 16 ? 0.011f : 0.016f) && leaves >= 8.f && points >= 480.f &&
           (a.k <= 18 || a.nq >= 16384 || points >= 24000.f) && near * scale <= fmaxf(a.k + 14.f, 2.f * (a.k + scale));
}

// The furthest neighbours: the query's k-th furthest distance is estimated from
// the points of the eight sampled leaves that reach farthest (as the
// (k x share)-th furthest, the sampled leaves being that share of all);
// kept counts the sampled leaves that reach beyond it, near the evaluated points
// within the tile's error band of it.
template <int DP>
__global__ void __launch_bounds__(kProbeThreads) k_probe_far(const ProbeArgs a) {
    using Bd = TcBound<3, DP, OP_FAR>;
    __shared__ float dm[kProbeLeaves], pv[kProbeTop * kProbeRows];
    __shared__ unsigned long long wkey[2][kProbeThreads / 32];
    __shared__ int tbeg[kProbeTop], tcnt[kProbeTop];
    __shared__ uint32_t s_kth;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float q[DP];
    const float qa = probe_load<DP>(q, a.qpts + probe_pick(blockIdx.x, a.nq, gridDim.x) * DP, a.rbox);
    const int S = a.leaves;
    for (int i = tid; i < S; i += kProbeThreads) {
        const float4* lo4 = reinterpret_cast<const float4*>(a.rbox + (a.rleaf0 + probe_pick(i, a.nleaves, S)) * 2 * DP);
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < DP / 4; ++j) {
            const float4 lo = lo4[j], hi = lo4[DP / 4 + j];
            const float g0 = fmaxf(q[4 * j] - lo.x, hi.x - q[4 * j]);
            const float g1 = fmaxf(q[4 * j + 1] - lo.y, hi.y - q[4 * j + 1]);
            const float g2 = fmaxf(q[4 * j + 2] - lo.z, hi.z - q[4 * j + 2]);
            const float g3 = fmaxf(q[4 * j + 3] - lo.w, hi.w - q[4 * j + 3]);
            s = fmaf(g0, g0, fmaf(g1, g1, fmaf(g2, g2, fmaf(g3, g3, s))));
        }
        dm[i] = s;
    }
    if (tid == 0) s_kth = 0x7f800000u;
    __syncthreads();
    // the leaves that reach farthest ...
    unsigned long long last = ~0ull;
    int nt = 0;
    for (; nt < kProbeTop; ++nt) {
        unsigned long long best = 0;  // (reach, leaf + 1)
        for (int i = tid; i < S; i += kProbeThreads) {
            const unsigned long long key = ((unsigned long long)__float_as_uint(dm[i]) << 32) | (unsigned)(i + 1);
            if (key < last && key > best) best = key;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
        if (lane == 0) wkey[nt & 1][warp] = best;
        __syncthreads();
        for (int w = 0; w < kProbeThreads / 32; ++w) best = max(best, wkey[nt & 1][w]);
        if (best == 0) break;  // (fewer than eight leaves)
        last = best;
        if (tid == 0) {
            const int64_t nd = a.rleaf0 + probe_pick((int)(uint32_t)best - 1, a.nleaves, S);
            tbeg[nt] = a.rbeg[nd];
            tcnt[nt] = a.rcnt[nd];
        }
    }
    __syncthreads();
    // ... and their points, a warp per leaf in turn
    int np = 0;
    int64_t all = 0;  // the points of those leaves, evaluated or not
    for (int t = 0; t < nt; ++t) {
        const int rows = min(tcnt[t], kProbeRows);
        if (t % (kProbeThreads / 32) == warp)
            for (int r = lane; r < rows; r += 32)
                pv[np + r] = approx_d2<DP>(q, a.rpts + (tbeg[t] + probe_pick(r, tcnt[t], rows)) * DP);
        np += rows;
        all += tcnt[t];
    }
    __syncthreads();
    const float share = (float)S / (float)a.nleaves * (float)np / (float)max(all, (int64_t)1);
    const int want = min(np, max(1, (int)ceilf(a.k * share)));
    for (int v = tid; v < np; v += kProbeThreads) {
        int g = 0;
        for (int j = 0; j < np; ++j) g += pv[j] > pv[v];
        if (g < want) atomicMin(&s_kth, __float_as_uint(pv[v]));
    }
    __syncthreads();
    const float kth = __uint_as_float(s_kth);
    const float band = -Bd::band(Bd::ub(-kth, qa, a.rlam[0]), qa, a.rlam[0]);
    int kept = 0, near = 0;
    for (int i = tid; i < S; i += kProbeThreads) kept += dm[i] >= kth;
    for (int v = tid; v < np; v += kProbeThreads) near += pv[v] >= band;
    int all_kept, all_near, all_pts;
    if (!probe_total(a, kept, near, np, all_kept, all_near, all_pts)) return;
    float radius;
    const bool extents = probe_extents<DP>(a, radius);
    if (lane == 0) {
        a.out->gate = extents && far_by_tiles<DP>(a, (float)all_kept / ((float)gridDim.x * (float)S),
                                                  (float)all_near / (float)gridDim.x);
    }
}

// Range searches, from a walk's share of the leaves, the points in them, and the
// share of those that lie within the upper end (which the tiles evaluate one by
// one, and in float64 when they write them).
//
// The tiles win where many leaves are visited for few results (the mixture, d = 16,
// 1M x 50k points: radius 2.0 1.3% of the leaves, 22.9 -> 2.8 ms; 2.5 2.0% and 0.03%
// of the points, 32.9 -> 5.2; 3.0 2.6% and 0.3%, 42.6 -> 20.4; 10k x 150k at 2.0, 260
// points, 2.1 -> 1.0; eight latent dimensions, 300k x 50k, 1.1% and 0.4%, 15.5 -> 7.9;
// d = 32 at 5.5 3.2% and 0.5%, 50 -> 16) and lose where the results are many or the
// leaves few, most of all at low intrinsic dimension (the mixture at 3.5 2.9% and
// 1.4%, 77 -> 103; d = 10 at 1.9 1.2% and 0.6%, 12.2 -> 14.1; 300k x 50k points of
// three latent dimensions at 0.4 1.1% and 45%, 40 -> 243; 1M x 20k of six in d = 32 at
// 0.6 0.2% and 0.5%, 6.5 -> 8.6; at 1.0 0.8% and 2.2%, 24 -> 72; distances of 9 to 20
// among Gaussian points, where nearly all points lie within the upper end, 64 -> 207).
// Leaves of more than 64 points halve what a walk pays per point (leaves of 390, the
// mixture at 3.2 0.4%, 2.5 -> 2.9; d = 10 at 1.9, of 490, 0.3%, 10.9 -> 15.1).
template <int DP>
__device__ __forceinline__ bool range_by_tiles_pays(const ProbeArgs& a, float share, float within) {
    const float few = (DP <= 16 ? 0.0045f : 0.008f) * (a.nr > 64 * a.nleaves ? 0.5f : 1.f);
    return share >= 0.0025f && share * (float)a.nr >= 150.f && within <= few;
}

// Range searches: kept counts the sampled leaves that meet the range, near the
// points within its upper end of up to sixteen of them, evenly chosen.
template <int DP>
__global__ void __launch_bounds__(kProbeThreads) k_probe_range(const ProbeArgs a) {
    __shared__ int list[kProbeLeaves], wcnt[kProbeThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float q[DP];
    probe_load<DP>(q, a.qpts + probe_pick(blockIdx.x, a.nq, gridDim.x) * DP, a.rbox);
    const int S = a.leaves;
    const float dn = 1.f - 2.f * rel_eps<DP>(), up = 1.f + 2.f * rel_eps<DP>();
    int kept = 0, found = 0;  // this thread's, the CTA's so far
    for (int i0 = 0; i0 < S; i0 += kProbeThreads) {
        const int i = i0 + tid;
        bool keep = false;
        if (i < S) {
            const float4* lo4 = reinterpret_cast<const float4*>(a.rbox + (a.rleaf0 + probe_pick(i, a.nleaves, S)) * 2 * DP);
            float mn = 0.f, mx = 0.f;
#pragma unroll
            for (int j = 0; j < DP / 4; ++j) {
                const float4 lo = lo4[j], hi = lo4[DP / 4 + j];
                const float l[4] = {lo.x, lo.y, lo.z, lo.w}, h[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float below = l[t] - q[4 * j + t], above = q[4 * j + t] - h[t];
                    const float g = fmaxf(fmaxf(below, above), 0.f), f = fmaxf(-below, -above);
                    mn = fmaf(g, g, mn);
                    mx = fmaf(f, f, mx);
                }
            }
            keep = !(mn * dn > a.hi2_up) && !(mx * up < a.lo2_dn);
        }
        kept += keep;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wcnt[warp] = __popc(m);
        __syncthreads();
        int at = found + __popc(m & ((1u << lane) - 1u));
        for (int w = 0; w < kProbeThreads / 32; ++w) {
            if (w < warp) at += wcnt[w];
            found += wcnt[w];
        }
        if (keep) list[at] = i;
        __syncthreads();
    }
    int near = 0, pts = 0;
    const int nt = min(found, kProbeRangeTop);
    for (int t = 0; t < nt; ++t) {
        const int64_t nd = a.rleaf0 + probe_pick(list[probe_pick(t, found, nt)], a.nleaves, S);
        const int rc = a.rcnt[nd], rows = min(rc, kProbeRows);
        pts += rows;
        if (t % (kProbeThreads / 32) != warp) continue;
        for (int r = lane; r < rows; r += 32)
            near += approx_d2<DP>(q, a.rpts + (a.rbeg[nd] + probe_pick(r, rc, rows)) * DP) <= a.hi2_up;
    }
    // (each query by the leaves it stands for: sixteen times found / nt)
    const int weight = nt == kProbeRangeTop ? found : kProbeRangeTop;
    int all_kept, all_near, all_pts;
    if (!probe_total(a, kept, near * weight, pts * weight, all_kept, all_near, all_pts)) return;
    float radius;
    const bool extents = probe_extents<DP>(a, radius);
    if (lane == 0) {
        const float share = (float)all_kept / ((float)gridDim.x * (float)S);
        // (a range far below the extents: the tensor-core keys' error, about 1e-4
        // of their square, would add too many candidates)
        a.out->gate = extents && a.hi_up * a.hi_up >= 4e-4f * radius * radius &&
                      range_by_tiles_pays<DP>(a, share, (float)all_near / fmaxf((float)all_pts, 1.f));
    }
}

template <int DP>
int launch_probe_range(const ProbeArgs& a, cudaStream_t s) {
    DT_LAUNCH(k_probe_range<DP>, (int)(a.nq < kProbeQueries ? a.nq : kProbeQueries), kProbeThreads, 0, s, a);
    return DTREE_OK;
}

template <int DP>
int launch_probe_far(const ProbeArgs& a, cudaStream_t s) {
    DT_LAUNCH(k_probe_far<DP>, (int)(a.nq < kProbeQueries ? a.nq : kProbeQueries), kProbeThreads, 0, s, a);
    return DTREE_OK;
}

}  // namespace dt
