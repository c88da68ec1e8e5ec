// emst.cuh -- the Euclidean minimum spanning tree by Boruvka rounds (dtree_emst).
//
// Section 7 ("Boruvka's Algorithm"): every component finds the shortest edge
// from one of its points to a point outside it, the components joined by
// those edges merge, and the rounds repeat until one component is left.
// Edges are ranked by (float64 squared length, lower original index, higher
// original index): every edge has its own rank, so the tree is unique and
// the components' chosen edges can only form trees and two-cycles (a pair of
// components choosing the same edge).
//
// One round on the GPU, all in kernels:
//   1. node labels: a node's component when all its points share one, else -1;
//   2. a length no longer than which every component's shortest edge must be:
//      from the edges of earlier rounds that still leave the component and
//      from the pairs inside a packet (k_emst_prep, not in the first round);
//   3. for every point that can still hold its component's shortest edge, its
//      nearest point outside the component (k_emst_nn);
//   4. every component's shortest edge: an atomicMin over the squared lengths
//      (at the end of step 3), then over the endpoint pairs among the points
//      that reach it;
//   5. hooks: each component points to the component across its edge (a
//      two-cycle keeps the lower id as the root), and each edge is written
//      once, in component-id order; then the roots are found and the points
//      relabelled.
#pragma once

#include "packet.cuh"

namespace dt {

struct EmstArgs {
    const float* pts;       // tree order, DP floats each
    const int32_t* idx;     // tree position -> original index
    const int32_t* nbeg;
    const int32_t* ncnt;
    const float* box;
    int64_t n;
    int hr;
    Packets pk, pk1;        // the points as packets, and as packets of up to 32
    int first;              // the first round: no earlier results, no bounds
    const int32_t* comp;    // per point: its component (a root point's tree position)
    const int32_t* nlab;    // per node: its component if all its points share one, else -1
    // per point, kept from round to round
    double* bd;             // the squared length of its edge br
    int32_t* br;            // the other end of its best edge out (tree position), or -1
    float* lb;              // no point outside its component is nearer than this (squared)
    unsigned char* done;    // br is its nearest point outside the component
    // per component, of this round
    uint32_t* cub;          // bits of a float no smaller than its shortest edge's squared length
    unsigned long long* ck1;    // the key of its shortest edge
    unsigned long long* stats;  // [0] point distances, [1] leaves visited
};

// Order-preserving key of a non-negative double (inf included).
__device__ __forceinline__ unsigned long long dkey(double v) {
    return (unsigned long long)__double_as_longlong(v);
}

// Lowers a component's bound to v (bits of a non-negative float order like it).
__device__ __forceinline__ void emst_publish(uint32_t* cub, float v) {
    if (__float_as_uint(v) < *reinterpret_cast<volatile uint32_t*>(cub)) atomicMin(cub, __float_as_uint(v));
}

// Edges from the point with original index o: is the one of squared length d
// to r before the one of squared length e to t?
__device__ __forceinline__ bool emst_before(double d, uint32_t o, uint32_t r, double e, uint32_t t) {
    const uint32_t l1 = min(o, r), l2 = min(o, t);
    return d < e || (d == e && (l1 < l2 || (l1 == l2 && max(o, r) < max(o, t))));
}

// Upper bounds of the components' shortest edges before the search: each
// point's edge of an earlier round, where it still leaves the component, and
// the pairs of points in its packet.  They let the search skip every point
// whose lower bound exceeds its component's (on 1M uniform points in d = 3 all
// but a few per cent from the third round on).
template <int DP>
__global__ void __launch_bounds__(128) k_emst_prep(const EmstArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= a.pk1.count) return;
    const int2 pr = packet_range(a.pk1, a.nbeg, a.ncnt, w);
    if (pr.y == 0) return;
    const bool in = lane < pr.y;
    const int64_t pos = pr.x + (in ? lane : 0);
    const int32_t mine = in ? a.comp[pos] : -1;
    float best = INFINITY;
    if (in) {
        const int32_t r = a.br[pos];
        if (r >= 0 && a.comp[r] != mine) {
            best = __double2float_ru(a.bd[pos]);
        } else if (r >= 0) {
            a.br[pos] = -1;
            a.done[pos] = 0;
        }
    }
    if (!__all_sync(0xffffffffu, mine == __shfl_sync(0xffffffffu, mine, 0) || !in)) {
        float q[DP];
        load_row<DP>(q, a.pts + pos * DP);
        float key = INFINITY;
        for (int e = 0; e < pr.y; ++e)
            if (__shfl_sync(0xffffffffu, mine, e) != mine)
                key = fminf(key, approx_d2<DP>(q, a.pts + (int64_t)(pr.x + e) * DP));
        best = fminf(best, key_up<DP>(key));
    }
    // one update per component of the packet, by its first lane
    const unsigned peers = __match_any_sync(0xffffffffu, mine);
    best = __uint_as_float(__reduce_min_sync(peers, __float_as_uint(best)));
    if (in && lane == __ffs(peers) - 1 && best < INFINITY) emst_publish(a.cub + mine, best);
}

// The smallest of a value over a point's G lanes (a power of two).
__device__ __forceinline__ float emst_lanes_min(float v, int G) {
    for (int off = G >> 1; off > 0; off >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

// The nearest point outside its component of every point that can still hold
// its component's shortest edge, by packets (packet.cuh) that walk the tree
// nearer child first.  The G lanes of a point share its bound and keep a best
// edge each, the best of which is taken at the end.  Other warps lower a
// component's bound meanwhile, so that the lanes may read different values:
// each takes the smallest, or what one lane pruned by a smaller bound would be
// missing from what the point's first lane then records (done, lb).
//
// Score: a lane prunes a node when all the node's points lie in its own
// component, or when the squared d_min, rounded down, exceeds the smaller of
// its own best and its component's (strictly: an equal length may still have
// a lower rank; the holder of the component's shortest edge never prunes that
// edge's other end).
// BaseCase: float32 keys decide wherever their error cannot matter: a key
// clearly below the best's replaces it, one clearly above is dropped, and
// only between them (ties, near-ties) are both recomputed in float64 and
// ranked by (length, endpoints).  Each point's final edge gets its float64
// length at the end.
// Points are skipped without a walk when an earlier round's answer still
// leaves the component and was the nearest (the points outside a component
// only become fewer), or when no outside point can be as near as the
// component's bound.
//
// Tree and edges of 1M uniform points, d = 3: 240 -> 8.4 ms; of 60k points of the
// 16-dimensional mixture: 198 -> 9.9 ms (against a float64 walk per point).
template <int DP>
__global__ void __launch_bounds__(128) k_emst_nn(const EmstArgs a) {
    __shared__ PacketStack stacks[4];
    PacketStack& st = stacks[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= a.pk.count) return;
    const int2 pr = packet_range(a.pk, a.nbeg, a.ncnt, w);
    if (pr.y == 0) return;
    const int gs = a.pk.gs, G = 1 << gs;
    const int qi = lane >> gs, sub = lane & (G - 1);
    const bool in = qi < pr.y;
    const int64_t pos = pr.x + (in ? qi : 0);
    const int32_t mine = a.comp[pos];
    double bd = INFINITY;   // float64 length of the best edge (valid only where have64)
    int32_t br = -1;
    bool have64 = false, need = in, done = false;
    float cub = INFINITY;
    if (!a.first && in) cub = __uint_as_float(*reinterpret_cast<volatile uint32_t*>(a.cub + mine));
    cub = emst_lanes_min(cub, G);
    if (!a.first && in) {
        br = a.br[pos];
        bd = a.bd[pos];
        have64 = br >= 0;
        done = br >= 0 && a.done[pos];
        need = !done && !(a.lb[pos] > cub);
        if (!done && !need) br = -1;  // no outside point is near enough: not the holder
    }
    unsigned long long n_pts = 0, n_leaves = 0;
    if (__any_sync(0xffffffffu, need) && a.nlab[0] == -1) {
        float q[DP];
        load_row<DP>(q, a.pts + pos * DP);
        float bk = need && br >= 0 ? approx_d2<DP>(q, a.pts + (int64_t)br * DP) : INFINITY;  // br's key
        float bound = fminf(key_up<DP>(bk), cub);
        const uint32_t op = (uint32_t)a.idx[pos];
        int sp = 0;
        st.push(sp, 0, 0.f, lane);
        while (sp > 0) {
            --sp;
            const int32_t n = st.node[sp];
            const float dm = st.d[sp][lane];
            const bool want = need && !(dm > bound);
            const unsigned wants = __ballot_sync(0xffffffffu, want);
            if (!wants) continue;
            if (level_of_node(n) == a.hr) {
                const int rb = a.nbeg[n], rc = a.ncnt[n];
                ++n_leaves;
                n_pts += (unsigned long long)rc * (__popc(wants) >> gs);
                for (int r0 = 0; r0 < rc; r0 += 32) {
                    // the points whose key may beat the best before them (few:
                    // a running minimum), gathered without branches
                    const int rn = min(32, rc - r0);
                    float hi = key_hi<DP>(bk);  // a larger key cannot be as near as br
                    unsigned m = 0;
#pragma unroll 4
                    for (int e = sub; e < rn; e += G) {
                        const int r = rb + r0 + e;
                        const float d = approx_d2<DP>(q, a.pts + (int64_t)r * DP);
                        const float key = a.comp[r] == mine ? INFINITY : d;
                        m |= (key <= hi ? 1u : 0u) << e;
                        hi = fminf(hi, key_hi<DP>(key));
                    }
                    if (!want) m = 0;
                    while (m) {
                        const int r = rb + r0 + __ffs(m) - 1;
                        m &= m - 1;
                        if (a.comp[r] == mine) continue;  // (an overflowing key)
                        const float key = approx_d2<DP>(q, a.pts + (int64_t)r * DP);
                        if (key > key_hi<DP>(bk)) continue;
                        if (br < 0 || key < key_lo<DP>(bk)) {
                            br = r;
                            bk = key;
                            have64 = false;
                            continue;
                        }
                        // too close to call in float32: float64 lengths, then endpoints
                        if (!have64) bd = exact_d2<DP>(q, a.pts + (int64_t)br * DP);
                        have64 = true;
                        const double d = exact_d2<DP>(q, a.pts + (int64_t)r * DP);
                        if (emst_before(d, op, (uint32_t)a.idx[r], bd, (uint32_t)a.idx[br])) {
                            bd = d;
                            br = r;
                            bk = key;
                        }
                    }
                }
                const float up = key_up<DP>(emst_lanes_min(bk, G));
                if (want) {
                    if (up < cub) emst_publish(a.cub + mine, up);
                    cub = fminf(cub, __uint_as_float(*reinterpret_cast<volatile uint32_t*>(a.cub + mine)));
                }
                cub = emst_lanes_min(cub, G);
                bound = fminf(up, cub);
                continue;
            }
            const int64_t l = 2 * (int64_t)n + 1;
            float d0, d1;
            packet_child_dmin<DP>(q, a.box + l * 2 * DP, d0, d1);
            const bool w0 = want && a.nlab[l] != mine && !(d0 > bound);
            const bool w1 = want && a.nlab[l + 1] != mine && !(d1 > bound);
            packet_push_near_first(st, sp, (int32_t)l, w0 ? d0 : INFINITY, w1 ? d1 : INFINITY, w0, w1, lane);
        }
        // the best of the point's G lanes, in float64 and by endpoints
        if (need && br >= 0 && !have64) bd = exact_d2<DP>(q, a.pts + (int64_t)br * DP);
        if (br < 0) bd = INFINITY;
        float best = bk;
        for (int off = G >> 1; off > 0; off >>= 1) {
            best = fminf(best, __shfl_xor_sync(0xffffffffu, best, off));
            const double d = __shfl_xor_sync(0xffffffffu, bd, off);
            const int32_t r = __shfl_xor_sync(0xffffffffu, br, off);
            if (r >= 0 && (br < 0 || emst_before(d, op, (uint32_t)a.idx[r], bd, (uint32_t)a.idx[br]))) {
                bd = d;
                br = r;
            }
        }
        if (need) {
            done = br >= 0 && key_up<DP>(best) <= cub;
            // (an overflowing key stands for the largest float at least, as in packet.cuh)
            const float least = fminf(fminf(best, cub), kKeyMax);
            if (sub == 0) a.lb[pos] = fmaxf(__fmul_rd(least, 1.f - 8.f * rel_eps<DP>()) - kKeyTiny, 0.f);
        }
    }
    if (in && sub == 0) {
        a.bd[pos] = bd;
        a.br[pos] = br;
        a.done[pos] = done;
        if (br >= 0) {
            const unsigned long long k = dkey(bd);
            if (k < *reinterpret_cast<volatile unsigned long long*>(a.ck1 + mine)) atomicMin(a.ck1 + mine, k);
        }
    }
    if (lane == 0 && n_leaves) {
        atomicAdd(&a.stats[0], n_pts);
        atomicAdd(&a.stats[1], n_leaves);
    }
}

template <int DP>
int launch_emst_nn(const EmstArgs& a, cudaStream_t s) {
    if (!a.first) DT_LAUNCH(k_emst_prep<DP>, (int)((a.pk1.count + 3) / 4), 128, 0, s, a);
    DT_LAUNCH(k_emst_nn<DP>, (int)((a.pk.count + 3) / 4), 128, 0, s, a);
    return DTREE_OK;
}

}  // namespace dt
