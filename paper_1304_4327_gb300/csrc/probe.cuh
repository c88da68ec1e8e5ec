// probe.cuh -- a look at a problem before it is searched: what a walk per query
// would visit, and what the block search's tiles would have to settle exactly.
//
// A CTA per sampled query scores up to 1024 leaves, evenly spaced in the tree,
// and evaluates the points of a few of them; counts go out (the same in every
// call).  No chain of loads is longer than a few, so that the whole look costs
// little more than its read-back; a sample of walks would take as long as its
// longest walk.
#pragma once

#include "knn_tc.cuh"

namespace dt {

constexpr int kProbeThreads = 128, kProbeTop = 8, kProbeRows = 64;

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

// The CTA's two counts; true for the first warp of the last CTA, which gets the
// totals.
__device__ __forceinline__ bool probe_total(const ProbeArgs& a, int kept, int near, int& all_kept, int& all_near) {
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
        __threadfence();
        s_last = atomicAdd(&a.out->done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || tid >= 32) return false;
    __threadfence();
    int k = 0, n = 0;  // (at most 1024 per CTA, of 64)
    for (int q = lane; q < (int)gridDim.x; q += 32) {
        k += __ldcg(&a.out->kept[q]);
        n += __ldcg(&a.out->near[q]);
    }
    all_kept = __reduce_add_sync(0xffffffffu, k);
    all_near = __reduce_add_sync(0xffffffffu, n);
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
// of the leaves, number of them) and how many points the tile's band would hold
// (near, where scale leaves stand behind each scored one).
//
// A walk per query visits few leaves where the points' intrinsic dimension is
// low, whatever the space they lie in, and then beats the tiles, whose blocks
// must visit what any of 128 queries needs.  Walks and tiles, by the share
// estimated: 300k x 50k points of d = 16 with three latent dimensions 0.1%, 0.77
// and 1.52 ms; with seven 1.1%, 8.7 and 6.9; with ten 3.6%, 33 and 7.7; 1M x 20k
// of d = 32, four latent dimensions 0.2%, 1.4 and 6.8 ms; six 1.1%, 9.2 and 15.8;
// eight 2.1%, 19 and 16; the mixture, d = 10, 1M x 100k 3%, 69 and 18 ms, d = 16, 1M x
// 200k 8%, 312 and 41.  Few leaves in all: 20k x 100k, four latent dimensions 1%,
// 11 of 1024 leaves, 1.5 and 1.8 ms.  Lists of 64 (k > 18) cost the tiles half
// as much again, and few queries leave the GPU to the latency of either:
// mixture, d = 10, 250k x 8,200, k = 30, 570 leaves, 3.5 and 4.0 ms; 1M x 4,100, 1,090
// leaves, 6.7 and 5.3; 250k x 16,400, 6.2 and 5.2.
// Where the band holds more than a list (equal or nearly equal distances), the
// tiles' work is done twice: queries at the centre of a sphere 16.8 against 14.2
// ms.  A healthy band holds about k points of all, or about one of those sampled.
__device__ __forceinline__ bool far_by_tiles(int k, int64_t nq, float share, float visits, float near, float scale) {
    return share >= 0.018f && visits >= 24.f && (k <= 18 || nq >= 16384 || visits >= 800.f) &&
           near <= fmaxf(k + 14.f, 2.f * (k + scale));
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
    const float qa = probe_load<DP>(q, a.qpts + (blockIdx.x * a.nq / gridDim.x) * DP, a.rbox);
    const int S = a.leaves;
    for (int i = tid; i < S; i += kProbeThreads) {
        const float4* lo4 = reinterpret_cast<const float4*>(a.rbox + (a.rleaf0 + i * a.nleaves / S) * 2 * DP);
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
            const int64_t nd = a.rleaf0 + ((int64_t)(uint32_t)best - 1) * a.nleaves / S;
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
                pv[np + r] = approx_d2<DP>(q, a.rpts + ((int64_t)tbeg[t] + r) * DP);
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
    int all_kept, all_near;
    if (!probe_total(a, kept, near, all_kept, all_near)) return;
    float radius;
    const bool extents = probe_extents<DP>(a, radius);
    if (lane == 0) {
        const float scale = (float)a.nleaves / (float)S;
        const float kept_q = (float)all_kept / (float)gridDim.x, near_q = (float)all_near / (float)gridDim.x;
        a.out->gate = extents && far_by_tiles(a.k, a.nq, kept_q / (float)S, kept_q * scale, near_q * scale, scale);
    }
}

template <int DP>
int launch_probe_far(const ProbeArgs& a, cudaStream_t s) {
    DT_LAUNCH(k_probe_far<DP>, (int)(a.nq < kProbeQueries ? a.nq : kProbeQueries), kProbeThreads, 0, s, a);
    return DTREE_OK;
}

}  // namespace dt
