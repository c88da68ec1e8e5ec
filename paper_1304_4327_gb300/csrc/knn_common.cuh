// knn_common.cuh -- shared declarations of the kNN kernels (dtree_knn).
#pragma once

#include "dtree_internal.cuh"

namespace dt {

// Counters gathered on the device (dtree_stats order).
enum StatSlot {
    ST_SCORED = 0,
    ST_PRUNED,
    ST_EMITTED,
    ST_SKIPPED,
    ST_EVALUATED,
    ST_POINT_PAIRS,
    ST_RERANK,
    ST_FALLBACK,
    ST_SEED_PAIRS,
    ST_NSTAT
};

// What a BaseCase tile pass starts from and what it leaves behind.
enum TileMode {
    MODE_SEED = 0,  // seed leaves only, empty lists in, approximate lists out
    MODE_MAIN = 1   // traversal candidates, lists in, exact re-rank + output out
};

// Which neighbours a search finds.  The furthest ones are found by the same
// passes with every distance negated: keys are -d^2, node bounds -d_max (a
// lower bound on the negated distances), B's terms negated k-th distances, so
// that "smaller is better" holds throughout and B_1, A + 2 lambda and Score keep
// their form (Section 5's paragraph on k-furthest neighbours inverts the rules;
// this inverts the distances).
// A range search visits the leaf pairs within its range and keeps no lists.
enum SearchOp { OP_NEAR = 0, OP_FAR = 1, OP_RANGE = 2 };

constexpr int kQB = 128;           // queries of one work item (one thread each)
constexpr int kEmptyIdx = 0x7fffffff;

// One kNN problem of a batch, as the kernels see it.  Blocks (query-tree
// nodes at the block level) are numbered across the batch: the problem's
// blocks are [block0, block0 + nblocks).  Its queries occupy rows
// [q0, q0 + n_query) of the per-query arrays (candidate lists, bounds), in
// query-tree order, and its query nodes of levels 0..Lb occupy entries
// [node0, node0 + 2^(Lb+1) - 1) of the per-node bound arrays.
struct ProbDev {
    // query tree
    const float* qpts;
    const int32_t* qidx;
    const int32_t* qbeg;
    const int32_t* qcnt;
    const float* qlam;
    const float* qbox;  // nodes x 2 x DP
    // reference tree
    const float* rpts;
    const int32_t* ridx;
    const int32_t* rbeg;
    const int32_t* rcnt;
    const float* rbox;  // nodes x 2 x DP; the root box's centre is the tensor-core centring point
    const float* rlam;  // nodes: lambda (largest distance from the box centre to a point)
    const void* rops;   // tensor-core operand rows of the reference points (or null)
    int64_t rls8;       // 8-row groups per leaf in rops
    // outputs, rows in the caller's query order
    int64_t* out_idx;
    float* out_dist;
    int64_t qblock0;  // heap id of the first query block in the query tree
    int64_t rleaf0;   // heap id of reference leaf 0
    int64_t q0;       // first row of the problem in the per-query arrays
    int64_t node0;    // first entry of the problem in the per-node arrays
    int32_t block0;   // first block of the problem
    int32_t nblocks;
    int32_t cpb;      // work items (chunks of <= 128 queries) per block
    int32_t k;
    int32_t mono;
    int32_t Lb;       // level of the query blocks
    int32_t hr;       // height of the reference tree
    int32_t Ls;       // level of the greedy seed subtree in the reference tree
    int32_t Lp;       // level of the learned proposal's cells (the proposed seed subtrees)
    int32_t item0;    // first work item of the problem
    int32_t bound;    // dtree_bound of the node and point lower bounds
    float lo_dn;      // range search: a float below d_lo (0: no lower end)
};

// ---- lower bounds on distances to a node (Section 3: d_min), rounded down
// so that float32 rounding can only keep what the exact rule would prune.
// A node's centre is its box centre 0.5 (lo + hi) (in float32 exactly as the
// build computed lambda around it: halving is exact); lambda bounds the
// distance from it to every point of the node.

// The box-centre distance |C_a - C_b| of two nodes, rounded down.
template <int DP>
__device__ __forceinline__ float centre_dist_down(const float* a, const float* b) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < DP; ++j) {
        const float t = 0.5f * (a[j] + a[DP + j]) - 0.5f * (b[j] + b[DP + j]);
        s = fmaf(t, t, s);
    }
    return __fmul_rd(__fsqrt_rd(s), 1.f - rel_eps<DP>());
}

// Ball bound between two nodes: |C_a - C_b| - lambda_a - lambda_b (>= 0).
template <int DP>
__device__ __forceinline__ float ball_dmin_down(const float* a, float la, const float* b, float lb) {
    return fmaxf(__fsub_rd(__fsub_rd(centre_dist_down<DP>(a, b), la), lb), 0.f);
}

// Point-to-box distance (the box's nearest point), rounded down.
template <int DP>
__device__ __forceinline__ float point_box_dmin_down(const float* q, const float* bx) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < DP; ++j) {
        float g = fmaxf(fmaxf(bx[j] - q[j], q[j] - bx[DP + j]), 0.f);
        s = fmaf(g, g, s);
    }
    return __fmul_rd(__fsqrt_rd(s), 1.f - rel_eps<DP>());
}

// Point-to-ball distance |q - C| - lambda (>= 0), rounded down.
template <int DP>
__device__ __forceinline__ float point_ball_dmin_down(const float* q, const float* bx, float lam) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < DP; ++j) {
        const float t = q[j] - 0.5f * (bx[j] + bx[DP + j]);
        s = fmaf(t, t, s);
    }
    return fmaxf(__fsub_rd(__fmul_rd(__fsqrt_rd(s), 1.f - rel_eps<DP>()), lam), 0.f);
}

// A point's lower bound against a node under the search's dtree_bound.
template <int DP>
__device__ __forceinline__ float point_dmin_down(int bound, const float* q, const float* bx, float lam) {
    if (bound == DTREE_BOUND_BOX) return point_box_dmin_down<DP>(q, bx);
    const float b = point_ball_dmin_down<DP>(q, bx, lam);
    return bound == DTREE_BOUND_BALL ? b : fmaxf(b, point_box_dmin_down<DP>(q, bx));
}

// Largest distance between the points of two boxes, rounded up and negated: a
// lower bound on every negated distance.
template <int DP>
__device__ __forceinline__ float box_dmax_neg(const float* a, const float* b) {
    const float4* al = reinterpret_cast<const float4*>(a);
    const float4* ah = reinterpret_cast<const float4*>(a + DP);
    const float4* bl = reinterpret_cast<const float4*>(b);
    const float4* bh = reinterpret_cast<const float4*>(b + DP);
    float s = 0.f;
#pragma unroll 4
    for (int j = 0; j < DP / 4; ++j) {
        const float4 x = al[j], y = ah[j], u = bl[j], v = bh[j];
        const float g0 = fmaxf(y.x - u.x, v.x - x.x), g1 = fmaxf(y.y - u.y, v.y - x.y);
        const float g2 = fmaxf(y.z - u.z, v.z - x.z), g3 = fmaxf(y.w - u.w, v.w - x.w);
        s = fmaf(g0, g0, s);
        s = fmaf(g1, g1, s);
        s = fmaf(g2, g2, s);
        s = fmaf(g3, g3, s);
    }
    return -__fmul_ru(__fsqrt_ru(s), 1.f + rel_eps<DP>());
}

// A range search's range, the floats around its squared ends that settle a
// float32 key (range.cuh), and where its results go.
struct RangeOut {
    double d_lo, d_hi;
    float hi_up;                  // a float above d_hi
    float lo2_dn, lo2_up;
    float hi2_dn, hi2_up;
    int fill;                     // 0: counts per caller row; 1: the segments at offsets
    int64_t* counts;
    const int64_t* offsets;
    int64_t* out_idx;
    float* out_dist;
};

// What the one-warp-per-query furthest-neighbour kernels read and write.
struct KfnArgs {
    // query points in query-tree order (DP floats each) and their caller rows
    const float* qpts;
    const int32_t* qidx;
    int64_t nq;
    // reference tree
    const float* rpts;
    const int32_t* ridx;
    const int32_t* rbeg;
    const int32_t* rcnt;
    const float* rbox;
    int hr;
    int k;
    int mono;
    int64_t* out_idx;   // (rows in the caller's query order) x k
    float* out_dist;
    const int* in_list;   // a list pass: the queries to serve, *in_count of them
    const int* in_count;
    int* fb_list;         // float pass: appends the queries whose band overflowed
    int* fb_count;
    unsigned long long* stats;  // [0] point distances, [1] leaves visited, [2] nodes pruned
    const int* gate;      // (all queries) set on the device: the block search serves them; or null
};

struct TileArgs {
    const ProbDev* probs;       // the batch's problems
    const int32_t* blk_prob;    // per block: its problem
    const int2* items;          // per work item: (block, chunk of 128 queries)
    int nitems;
    int64_t nq_all;             // rows of the per-query arrays (all problems' queries)
    // candidates
    const int32_t* seed_leaf0;  // per block and seed slot: first leaf of the slot's subtree
    const int32_t* seed_nleaf;  // per block and seed slot: its leaves (0: an unused slot)
    int seed_slots;             // seed slots per block (the greedy subtree, proposed cells)
    int seed_eval_slots;        // of those, the first this many are evaluated by the seed pass;
                                //   the tensor-core main pass evaluates the rest first
    const int64_t* csr_off;     // per block: [off[b], off[b+1]) in csr_leaf / csr_dmin, in
                                //   evaluation order (windows sorted by box-centre distance)
    const int32_t* csr_leaf;
    const float* csr_dmin;
    const float* Bn;            // per query node: B from the bounds pass (or null)
    // approximate candidate lists, [kc_rows][nq_all] layout
    int kc_rows;
    float* cand_d;
    int32_t* cand_i;
    float* qub;                 // per query: upper bound on its true k-th distance (seed pass)
    const float* qcap;          // per query: the cap pass's upper bound on it (or null)
    int* work_ctr;
    int4* fbq_list;    // queries whose error band overflowed: (tree position, block, ub bits, 0)
    int* fbq_count;
    int4* fbq2_list;   // of those, queries whose float32 band overflowed too
    int* fbq2_count;
    // the recomputation's slices per query (1: one CTA per query) and, for
    // more, their lists: queries x slices x KC keys (float64), then as many
    // indices
    int fb_slices;
    void* fb_part;
    unsigned long long* stats;
    RangeOut range;    // (OP_RANGE)
    // the tensor-core pass's slices per work item (1: one CTA per item), their
    // lists ([item][slice][entry][query] keys, then as many positions) and, per
    // item, how many slices are done
    int slices;
    float* slice_d;
    int32_t* slice_i;
    int* slice_done;
};

template <int DP>
int launch_tile_cc(const TileArgs& a, int kc, int mode, int items, cudaStream_t s);

// Per-query caps on the k-th distance: a best-first search of up to `budget`
// reference leaves per query, merged into its candidate list of kc (=
// a.kc_rows) entries; writes qcap and lowers qub.
template <int DP>
int launch_query_cap(const TileArgs& a, int kc, int budget, float* qcap, cudaStream_t s);

template <int DP>
int launch_query_fb(const TileArgs& a, int kc, int nfbq, bool exact, cudaStream_t s);

// The tensor-core BaseCase pass (main mode): fmt 1 = BF16 (split), 2 = TF32;
// wide: a block's chunks are taken two at a time.
template <int DP>
int launch_tile_tc(const TileArgs& a, int fmt, int kc, int items, bool wide, int* err, int spin,
                   cudaStream_t s);

// The furthest-neighbour search's seed tile, cap and tensor-core passes (BF16),
// with lists of 24, 32 or 64 entries.
template <int DP>
int launch_far_seed(const TileArgs& a, int kc, int items, cudaStream_t s);
template <int DP>
int launch_far_cap(const TileArgs& a, int kc, int budget, float* qcap, cudaStream_t s);
template <int DP>
int launch_far_tile(const TileArgs& a, int kc, int items, bool wide, int* err, int spin, cudaStream_t s);
// ... and the one-warp-per-query search (kfn.cuh): of all queries with float32
// keys, of the first words of the 16-byte entries of a.in_list with float32 keys,
// or of its words in float64.
enum KfnPass { KFN_ALL = 0, KFN_LIST = 4, KFN_EXACT = 1 };  // (words per entry)
template <int DP>
int launch_kfn(const KfnArgs& a, int kc, KfnPass pass, int grid, cudaStream_t s);

// The range search's tensor-core pass (BF16).
template <int DP>
int launch_range_tile(const TileArgs& a, int items, int* err, int spin, cudaStream_t s);

// One pass (count or fill) of a range search by block traversal and tensor-core
// tiles; range.cu's look checks that it fits.  Adds to st when given.
int range_by_tiles(const dtree_t* tq, const dtree_t* tr, bool mono, const RangeOut& r, cudaStream_t s,
                   dtree_stats* st);

// A look at a problem before it is searched (probe.cuh), made on the device: the
// walk that follows it on the stream returns at once where gate is set, and the
// host, which waits for the walk anyway, then runs the block search.
constexpr int kProbeQueries = 128, kProbeLeaves = 1024;

struct ProbeOut {
    int gate;  // 1: the block search should serve the problem (zero before the look)
    int done;  // CTAs that have counted (zero before the look)
    int kept[kProbeQueries];  // per sampled query: the sampled leaves a walk would visit
    int near[kProbeQueries];  // and the evaluated points that the tiles would settle exactly,
    int pts[kProbeQueries];   // of this many
};

struct ProbeArgs {
    const float* qpts;
    int64_t nq;
    const float* rpts;
    const int32_t* rbeg;
    const int32_t* rcnt;
    const float* rbox;
    const float* rlam;
    const float* qbox;
    const float* qlam;
    int64_t nr, rleaf0, nleaves;
    int leaves;  // how many of them are scored
    int k;                         // furthest neighbours
    float lo2_dn, hi2_up, hi_up;   // range search: the ends, as in RangeOut
    ProbeOut* out;
};

inline ProbeArgs probe_args(const dtree_t* tq, const dtree_t* tr, ProbeOut* out) {
    ProbeArgs a{};
    a.qpts = tq->pts;
    a.nq = tq->n;
    a.rpts = tr->pts;
    a.rbeg = tr->nbeg;
    a.rcnt = tr->ncnt;
    a.rbox = tr->box;
    a.rlam = tr->lam;
    a.qbox = tq->box;
    a.qlam = tq->lam;
    a.nr = tr->n;
    a.nleaves = tr->nleaves;
    a.rleaf0 = tr->nleaves - 1;
    a.leaves = (int)(tr->nleaves < kProbeLeaves ? tr->nleaves : kProbeLeaves);
    a.out = out;
    return a;
}

// DP = 16, 32 and 64 only.
template <int DP>
int launch_probe_far(const ProbeArgs& a, cudaStream_t s);
template <int DP>
int launch_probe_range(const ProbeArgs& a, cudaStream_t s);

// dtree_kfn by these passes: one problem whose extents keep every squared
// distance inside float32's range (kfn.cu's look checks).  Adds to st when given.
int kfn_by_tiles(const dtree_t* tq, const dtree_t* tr, bool mono, int k, int64_t* out_idx, float* out_dist,
                 cudaStream_t s, dtree_stats* st);

// Bytes per operand row, and the fill of a reference tree's operand array
// (nleaves x ls rows, ls a multiple of 8) for the tensor-core pass.
template <int DP>
size_t tc_ops_row_bytes(int fmt);
template <int DP>
int launch_tc_ops(const dtree_t* t, int fmt, int ls, void* out, cudaStream_t s);

// A block's seed: up to `slots` disjoint subtrees of the reference tree,
// slot s covering leaves [leaf0[s], leaf0[s] + nleaf[s]).
__device__ __forceinline__ int seed_count(const int32_t* sn, int slots, int blk) {
    int t = 0;
    for (int s = 0; s < slots; ++s) t += sn[blk * slots + s];
    return t;
}

// Leaves of a block's first n seed slots.
__device__ __forceinline__ int seed_count_n(const int32_t* sn, int slots, int n, int blk) {
    int t = 0;
    for (int s = 0; s < n; ++s) t += sn[blk * slots + s];
    return t;
}

// The ci-th seed leaf of a block (slots in order).
__device__ __forceinline__ int seed_leaf(const int32_t* sl0, const int32_t* sn, int slots, int blk,
                                         int ci) {
    for (int s = 0; s < slots; ++s) {
        const int n = sn[blk * slots + s];
        if (ci < n) return sl0[blk * slots + s] + ci;
        ci -= n;
    }
    return -1;
}

__device__ __forceinline__ bool in_seed(const int32_t* sl0, const int32_t* sn, int slots, int blk,
                                        int leaf) {
    for (int s = 0; s < slots; ++s) {
        const int l0 = sl0[blk * slots + s];
        if (leaf >= l0 && leaf < l0 + sn[blk * slots + s]) return true;
    }
    return false;
}

// The traversal's frontier holds (global query node, reference node) pairs;
// node_prob gives each global query node's problem.
template <int DP>
int launch_expand(int op, const ProbDev* probs, const int32_t* node_prob, const float* Bn, const int2* fin,
                  const int* nin, int2* fout, int* nout, int64_t cap, int4* outp, int* nout_p,
                  int64_t cap_p, int* bcount, const int32_t* seed_leaf0,
                  const int32_t* seed_nleaf, int seed_slots, int* overflow,
                  unsigned long long* stats, int np, int grid, cudaStream_t s);

template <int DP>
int launch_seed(int op, const ProbDev* probs, const int32_t* blk_prob, int nblocks, int seed_slots,
                int32_t* seed_leaf0, int32_t* seed_nleaf, cudaStream_t s);

int occupancy_grid(const void* kernel, int threads, size_t smem);

}  // namespace dt
