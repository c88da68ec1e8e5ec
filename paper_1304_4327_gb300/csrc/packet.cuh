// packet.cuh -- walks of a tree by packets of points (the spanning tree's
// nearest-edge search).
//
// A packet is up to 32 / G points of one query-tree node, G lanes of a warp
// for each (G a power of two).  Neighbours in the tree want almost the same
// reference nodes, so the warp walks the reference tree once for all of them:
// every box is read at one address for the whole warp, each lane computes its
// point's bound from registers with no shuffles, and a node is entered while
// any lane wants it; a leaf's points are dealt out to the G lanes of a point.
// What this costs is the distances of points that would have pruned the node;
// what it saves is all but one of 32 / G node visits.  G = 1 does the least
// work; few points take a larger G, so that their packets fill the GPU.
#pragma once

#include "knn_tile.cuh"

namespace dt {

// The points of a tree as packets of up to `size` = 32 >> gs points: the nodes
// [first, first + 2^level) in chunks (cpn of them per node; more than one only
// where leaves hold more than a packet).
struct Packets {
    int64_t first, count;
    int cpn, gs;
};

inline Packets make_packets(const dtree_t* t, int gs) {
    const int size = 32 >> gs;
    const int level = t->height < level_of_count(t->n, size) ? t->height : level_of_count(t->n, size);
    const int64_t nodes = (int64_t)1 << level;
    Packets p;
    p.gs = gs;
    p.first = nodes - 1;
    p.cpn = (int)(((t->n + nodes - 1) / nodes + size - 1) / size);
    p.count = nodes * p.cpn;
    return p;
}

// log2 of the lanes per point for n points: G = 1 once their packets give every
// SM sixteen warps, else the G (up to 8) that does.
inline int packet_lanes(int64_t n, int sms) {
    int gs = 0;
    while (gs < 3 && (n << gs) < (int64_t)sms * 16 * 32) ++gs;
    return gs;
}

// First tree position and number of points of packet w.
__device__ __forceinline__ int2 packet_range(const Packets& p, const int32_t* nbeg, const int32_t* ncnt, int64_t w) {
    const int64_t node = p.first + w / p.cpn;
    const int size = 32 >> p.gs, c = (int)(w % p.cpn) * size;
    return make_int2(nbeg[node] + c, max(0, min(size, ncnt[node] - c)));
}

// The depth-first walk's stack, one per warp: per entry the node and each
// lane's bound of it.  A walk holds at most one more entry than the tree has
// levels (the callers check height <= 30).
struct PacketStack {
    int32_t node[32];
    float d[32][32];
    __device__ __forceinline__ void push(int& sp, int32_t n, float dist, int lane) {
        if (lane == 0) node[sp] = n;
        d[sp][lane] = dist;
        __syncwarp();
        ++sp;
    }
};

template <int DP>
__device__ __forceinline__ void load_row(float (&q)[DP], const float* p) {
#pragma unroll
    for (int j = 0; j < DP / 4; ++j) {
        const float4 v = reinterpret_cast<const float4*>(p)[j];
        q[4 * j] = v.x;
        q[4 * j + 1] = v.y;
        q[4 * j + 2] = v.z;
        q[4 * j + 3] = v.w;
    }
}

// float32 squared distances (approx_d2) and the exact ones.  A key k of a
// squared distance D satisfies |k - D| <= rel_eps D + 2^-140 (the second term
// covers squares that underflow); kKeyTiny is far above that.
//   key_up(k)  no smaller than D
//   key_lo(k)  a key below it belongs to a strictly smaller distance than k's
//   key_hi(k)  a key above it belongs to a strictly larger distance than k's
constexpr float kKeyTiny = 1e-37f;
constexpr float kKeyMax = 3.4028234e38f;  // what an overflowing key stands for at least (but for its error)

template <int DP>
__device__ __forceinline__ float key_up(float k) {
    return __fadd_ru(__fmul_ru(k, 1.f + 2.f * rel_eps<DP>()), kKeyTiny);
}
template <int DP>
__device__ __forceinline__ float key_lo(float k) {
    return __fsub_rd(__fmul_rd(k, 1.f - 4.f * rel_eps<DP>()), kKeyTiny);
}
template <int DP>
__device__ __forceinline__ float key_hi(float k) {
    return __fadd_ru(__fmul_ru(k, 1.f + 4.f * rel_eps<DP>()), kKeyTiny);
}

// Squared d_min of a lane's point to each of two sibling boxes (bx: lo, hi of
// the left one, then of the right one), rounded down.  An overflow counts as
// the largest float.
template <int DP>
__device__ __forceinline__ void packet_child_dmin(const float (&q)[DP], const float* __restrict__ bx, float& d0,
                                                  float& d1) {
    float s[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float4* lo4 = reinterpret_cast<const float4*>(bx + c * 2 * DP);
        const float4* hi4 = reinterpret_cast<const float4*>(bx + c * 2 * DP + DP);
#pragma unroll
        for (int j = 0; j < DP / 4; ++j) {
            const float4 lo = lo4[j], hi = hi4[j];
            const float g0 = fmaxf(fmaxf(lo.x - q[4 * j], q[4 * j] - hi.x), 0.f);
            const float g1 = fmaxf(fmaxf(lo.y - q[4 * j + 1], q[4 * j + 1] - hi.y), 0.f);
            const float g2 = fmaxf(fmaxf(lo.z - q[4 * j + 2], q[4 * j + 2] - hi.z), 0.f);
            const float g3 = fmaxf(fmaxf(lo.w - q[4 * j + 3], q[4 * j + 3] - hi.w), 0.f);
            s[c] = fmaf(g0, g0, s[c]);
            s[c] = fmaf(g1, g1, s[c]);
            s[c] = fmaf(g2, g2, s[c]);
            s[c] = fmaf(g3, g3, s[c]);
        }
    }
    const float f = 1.f - 2.f * rel_eps<DP>();
    d0 = fmaxf(__fsub_rd(__fmul_rd(fminf(s[0], kKeyMax), f), kKeyTiny), 0.f);
    d1 = fmaxf(__fsub_rd(__fmul_rd(fminf(s[1], kKeyMax), f), kKeyTiny), 0.f);
}

// Push the wanted ones of two siblings (l, l + 1) so that the one nearer to
// the packet (the smallest d_min of a lane that wants it) is taken first.
// An unwanted lane's bound is +inf.
__device__ __forceinline__ void packet_push_near_first(PacketStack& st, int& sp, int32_t l, float d0, float d1,
                                                       bool w0, bool w1, int lane) {
    const bool any0 = __any_sync(0xffffffffu, w0), any1 = __any_sync(0xffffffffu, w1);
    if (any0 && any1) {
        const uint32_t m0 = __reduce_min_sync(0xffffffffu, __float_as_uint(d0));
        const uint32_t m1 = __reduce_min_sync(0xffffffffu, __float_as_uint(d1));
        const bool right = m1 < m0;
        st.push(sp, right ? l : l + 1, right ? d0 : d1, lane);
        st.push(sp, right ? l + 1 : l, right ? d1 : d0, lane);
    } else if (any0) {
        st.push(sp, l, d0, lane);
    } else if (any1) {
        st.push(sp, l + 1, d1, lane);
    }
}

}  // namespace dt
