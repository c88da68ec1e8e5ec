// knn_tile.cuh -- the kNN BaseCase (Algorithm 2 of Curtin et al.) on CUDA
// cores, one CTA per work item of <= 128 queries, one thread per query.
//
// For a query block and a list of reference leaves the CTA streams the
// leaves' points through shared memory and each thread keeps its query's
// candidate list (distance key, index) sorted in registers: a reference
// point enters when its key beats the list's last entry, the "d < D[k]"
// test of Algorithm 2 with ties broken by the lower index.
//
// Lists hold KC > k entries.  In float32 the squared distance carries a
// relative error of at most eps = (DP + 8) 2^-24, so
//   - an upper bound on the true k-th distance is sqrt(kth * (1 + 2 eps)),
//     which feeds B_1 and B_2 (Section 5) and the Score test (Algorithm 3)
//     that skips a leaf whose d_min exceeds the block's bound;
//   - every true k-nearest neighbour has a float32 key within
//     band = kth * (1 + 4 eps); at the end those candidates are re-ranked
//     with the exact float64 distance (the same left-to-right sum as the
//     definition) and ordered by (distance, reference index).
// If more than KC - k keys fall inside the band (near-ties or duplicates) the
// list may have dropped a true neighbour: that query is listed and
// recomputed in float64 (k_query_fb), where keys are exact.
//
// Bound by issue slots, not memory (L2 under 2%): per staged point a warp
// issues DP / 4 broadcast loads, DP packed operations and a compare for its 32
// queries.  Keys are taken 32 at a time with no branch between them, a bit
// each for those that may enter the list; inserting inside the key loop
// serialised it (43 instructions per point at d = 8 against 22).  Main pass of
// 10M x 1M points, d = 8, k = 10: 21.4 -> 12.1 ms; whole searches at d = 32
// and 64: 1.1 to 1.9 times faster.
#pragma once

#include <type_traits>

#include "knn_common.cuh"

namespace dt {

template <typename T>
__device__ __forceinline__ bool key_less(T d, int i, T e, int j) {
    return d < e || (d == e && i < j);
}

// Insert (d, i) into the ascending list (bubble through; the last entry falls off).
template <typename T, int KC>
__device__ __forceinline__ void list_insert(T (&ld)[KC], int (&li)[KC], T d, int i) {
#pragma unroll
    for (int j = 0; j < KC; ++j) {
        if (key_less(d, i, ld[j], li[j])) {
            T td = ld[j];
            int ti = li[j];
            ld[j] = d;
            li[j] = i;
            d = td;
            i = ti;
        }
    }
}

// The same insertion by key alone and without a serial chain: every
// comparison against the new key is independent, then each slot either keeps
// its entry, takes the new one or takes its predecessor (descending order
// reads each predecessor before it moves).  Entries of equal keys stay in the
// order they came: the tensor-core lists' order among them never matters,
// since the re-rank settles it and a band that reaches the last key overflows.
template <int KC>
__device__ __forceinline__ void list_insert_key(float (&ld)[KC], int (&li)[KC], float d, int i) {
#pragma unroll
    for (int j = KC - 1; j > 0; --j) {
        const bool here = d < ld[j], before = d < ld[j - 1];
        li[j] = here ? (before ? li[j - 1] : i) : li[j];
        ld[j] = here ? (before ? ld[j - 1] : d) : ld[j];
    }
    if (d < ld[0]) {
        ld[0] = d;
        li[0] = i;
    }
}

// Is i among the list's indices?
template <int KC>
__device__ __forceinline__ bool listed(const int (&li)[KC], int i) {
    bool in = false;
#pragma unroll
    for (int j = 0; j < KC; ++j) in |= li[j] == i;
    return in;
}

template <typename T, int KC>
__device__ __forceinline__ T list_at(const T (&ld)[KC], int j) {
    T v = ld[0];
#pragma unroll
    for (int q = 1; q < KC; ++q)
        if (q == j) v = ld[q];
    return v;
}

// Two float32 values in a register pair, and the packed fused multiply-add
// (each half rounded as fmaf rounds).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
    return ((uint64_t)__float_as_uint(y) << 32) | __float_as_uint(x);
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// The float32 key of a staged row: sum over j of (q_j - r_j)^2, even and odd
// coordinates summed apart (relative error <= rel_eps as before: each half has
// DP / 2 terms, and one more addition joins them).
template <int DP>
__device__ __forceinline__ float packed_d2(const uint64_t (&q)[DP / 2], const float* r) {
    const ulonglong2* r2 = reinterpret_cast<const ulonglong2*>(r);
    const uint64_t minus1 = pack2(-1.f, -1.f);
    uint64_t acc = 0;
#pragma unroll
    for (int j = 0; j < DP / 4; ++j) {
        const ulonglong2 v = r2[j];
        const uint64_t t0 = fma2(v.x, minus1, q[2 * j]), t1 = fma2(v.y, minus1, q[2 * j + 1]);
        acc = fma2(t0, t0, acc);
        acc = fma2(t1, t1, acc);
    }
    return __uint_as_float((uint32_t)acc) + __uint_as_float((uint32_t)(acc >> 32));
}

// Exact squared distance: sum over j of (q_j - r_j)^2 in float64, left to
// right, one rounding per operation (padded dimensions add +0 exactly).
template <int DP>
__device__ __forceinline__ double exact_d2(const float* q, const float* r) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < DP; ++j) {
        double t = __dsub_rn((double)q[j], (double)r[j]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// The same sum in pairs of float32 (value h + l, |l| <= ulp(h) / 2), on the
// FP32 pipe: this GPU's FP64 pipe does two operations per clock and SM, and the
// re-rank's k x DP x 5 of them per query held up every work item (at d = 64,
// k = 50 a fifth of the tile kernel's time).
//   t = q_j - r_j exactly as th + tl; t^2 as a product and its remainder plus
//   2 th tl; the running sum renormalised at each step.
// With S the true sum, |h + l - S| <= (DP + 4) 2^-44 S: per step the remainder
// terms round by at most 2 x 2^-46 of the running sum, tl^2 is left out (2^-48
// of its term).  The float64 sum itself is within (DP + 2) 2^-53 S of S.
// Returns false where the bound does not hold: a sum whose squares may have
// underflowed or overflowed (zero is exact when every difference is zero).
template <int DP>
__device__ __forceinline__ bool pair_d2(const float (&q)[DP], const float* r, float& h, float& l) {
    const float4* r4 = reinterpret_cast<const float4*>(r);
    float sh = 0.f, sl = 0.f, mx = 0.f;
#pragma unroll
    for (int j4 = 0; j4 < DP / 4; ++j4) {
        const float4 v = r4[j4];
        const float rv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float a = q[4 * j4 + u], b = -rv[u];
            const float th = __fadd_rn(a, b), bb = __fsub_rn(th, a);
            const float tl = __fadd_rn(__fsub_rn(a, __fsub_rn(th, bb)), __fsub_rn(b, bb));
            const float p = __fmul_rn(th, th);
            const float e = __fmaf_rn(__fadd_rn(th, th), tl, __fmaf_rn(th, th, -p));
            const float s = __fadd_rn(sh, p), sb = __fsub_rn(s, sh);
            const float se = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, sb)), __fsub_rn(p, sb));
            const float lo = __fadd_rn(sl, __fadd_rn(se, e));
            sh = __fadd_rn(s, lo);
            sl = __fsub_rn(lo, __fsub_rn(sh, s));
            mx = fmaxf(mx, fabsf(th));
        }
    }
    h = sh;
    l = sl;
    return (sh >= 1e-20f && sh <= 1e37f) || mx == 0.f;
}

// The float32 distance of a float64 squared distance D known as h + l within
// (DP + 4) 2^-44 D: (float)sqrt(D) as float64 rounds it, or false where D is
// too close to a rounding boundary to tell.
template <int DP>
__device__ __forceinline__ bool pair_dist(float h, float l, float& out) {
    out = 0.f;
    if (h == 0.f) return true;
    const float s0 = __fsqrt_rn(h);
    // sqrt(h + l) = s0 + c, c small and known to 2^-22 of itself
    const float c = __fmul_rn(__fadd_rn(__fmaf_rn(-s0, s0, h), l), __fdiv_rn(0.5f, s0));
    const float f = __fadd_rn(s0, c);
    const float e = __fsub_rn(c, __fsub_rn(f, s0));  // what the rounding to f left out
    const float half = 0.5f * (__uint_as_float(__float_as_uint(f) + 1u) - f);
    out = f;
    // (a power of two has a nearer boundary below: left to float64)
    return (__float_as_uint(f) & 0x7fffffu) != 0u &&
           half - fabsf(e) > f * ((DP + 4) * 1.1368684e-13f);  // 2^-43
}

// Upper bound on the true k-th value (a distance; for OP_FAR a negated one, of
// the negated key): for the furthest neighbours a lower bound on the k-th
// distance, negated.
template <int DP, int OP>
__device__ __forceinline__ float ub_op(float kth);

template <typename T, int DP>
__device__ __forceinline__ float ub_of(T kth) {
    if (sizeof(T) == 8) return __double2float_ru(__dsqrt_ru((double)kth));
    if (!(kth < INFINITY)) return INFINITY;
    return __fsqrt_ru(__fmul_ru((float)kth, 1.f + 2.f * rel_eps<DP>()));
}

template <int DP, int OP>
__device__ __forceinline__ float ub_op(float kth) {
    if (OP == OP_NEAR) return ub_of<float, DP>(kth);
    if (!(kth < INFINITY)) return INFINITY;
    return -__fsqrt_rd(fmaxf(__fmul_rd(-kth, 1.f - 2.f * rel_eps<DP>()), 0.f));
}

// Warp 0 of a tile CTA: take candidate leaves from the current window, in
// order, skip those whose d_min exceeds the block's bound (Algorithm 3:
// Score = infinity), and pack the rows of the rest (whole leaves, or the
// part of a leaf that fits) into a stage of at most TN points.  stab gets one
// (first row, rows, stage offset) entry per run of rows.
template <int TN, int MODE, int OP>
__device__ __forceinline__ void stage_fill(const TileArgs& a, const ProbDev& P, int64_t w0,
                                           int wn, int nseed, int blk, int64_t c0, int3* stab,
                                           unsigned long long& n_skip, unsigned long long& n_eval,
                                           int& s_cur, int& s_part, int& s_nst, int& s_ntab,
                                           const float Bc) {
    const int lane = threadIdx.x & 31;
    int cur = s_cur, part = s_part, nst = 0, ntab = 0;
    while (cur < wn && nst < TN) {
        int c = cur + lane;
        bool valid = c < wn;
        int leaf = 0;
        float dmin = -INFINITY;  // (a seed leaf is never pruned)
        if (valid) {
            if (MODE == MODE_MAIN) {  // the block's candidates, sorted nearest-first
                const int64_t ci = c0 + w0 + c;
                leaf = a.csr_leaf[ci];
                dmin = a.csr_dmin[ci];
            } else {
                int64_t ci = w0 + c;
                if (ci < nseed) {
                    leaf = seed_leaf(a.seed_leaf0, a.seed_nleaf, a.seed_slots, blk, (int)ci);
                } else {
                    leaf = a.csr_leaf[c0 + ci - nseed];
                    dmin = a.csr_dmin[c0 + ci - nseed];
                }
            }
        }
        bool keep = valid && !(dmin > Bc);
        int lb = 0, lc = 0;
        if (keep) {
            int64_t ln = P.rleaf0 + leaf;
            lb = P.rbeg[ln];
            lc = P.rcnt[ln];
        }
        if (lane == 0 && part > 0 && keep) {  // rest of a split leaf
            lb += part;
            lc -= part;
        }
        int incl = lc;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        int excl = incl - lc;
        int take = min(max(TN - nst - excl, 0), lc);
        bool full = valid && take == lc;
        unsigned fm = __ballot_sync(0xffffffffu, full);
        int nlead = fm == 0xffffffffu ? 32 : __ffs(~fm) - 1;
        bool put = take > 0 && lane <= nlead;
        unsigned tm = __ballot_sync(0xffffffffu, put);
        if (put) stab[ntab + __popc(tm & ((1u << lane) - 1u))] = make_int3(lb, take, nst + excl);
        unsigned sk = __ballot_sync(0xffffffffu, valid && !keep && lane < nlead);
        unsigned ev = __ballot_sync(0xffffffffu, keep && lane < nlead);
        if (lane == 0) {
            n_skip += __popc(sk);
            n_eval += __popc(ev);
        }
        int taken = put ? take : 0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) taken += __shfl_xor_sync(0xffffffffu, taken, off);
        int pn = __shfl_sync(0xffffffffu, take, nlead & 31);
        nst += taken;
        ntab += __popc(tm);
        if (nlead < 32) {
            part = (nlead == 0 ? part : 0) + pn;
            cur += nlead;
            if (!(cur < wn)) part = 0;
            break;  // stage full, or the window is exhausted
        }
        cur += 32;
        part = 0;
    }
    if (lane == 0) {
        s_cur = cur;
        s_part = part;
        s_nst = nst;
        s_ntab = ntab;
    }
}

template <int DP, int KC, int MODE, int OP = OP_NEAR>
__global__ void __launch_bounds__(kQB) k_tile(const TileArgs a) {
    constexpr int TN = 4096 / DP;       // staged reference points (16 KB)
    constexpr int WINDOW = 2048;        // candidates per window of the main pass
    __shared__ __align__(16) float rs[TN * DP];
    __shared__ int32_t spos[TN];
    __shared__ int3 stab[TN];
    __shared__ int s_item, s_ntab, s_nst, s_cur, s_part;
    __shared__ float s_B;
    __shared__ float s_rmax[kQB / 32], s_rmin[kQB / 32];
    __shared__ ProbDev s_prob;

    constexpr float sgn = OP == OP_FAR ? -1.f : 1.f;  // keys are negated squared distances for OP_FAR
    static_assert(OP == OP_NEAR || MODE == MODE_SEED, "the furthest neighbours' main pass is the tensor-core one");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nitems = a.nitems;
    unsigned long long n_skip = 0, n_eval = 0, n_pp = 0, n_re = 0;
    const ProbDev& P = s_prob;

    for (;;) {
        if (tid == 0) {
            s_item = atomicAdd(a.work_ctr, 1);
            if (s_item < nitems) s_prob = a.probs[a.blk_prob[a.items[s_item].x]];
        }
        __syncthreads();
        const int item = s_item;
        if (item >= nitems) break;
        const int2 wi = a.items[item];
        const int blk = wi.x, chunk = wi.y;  // global block, chunk of its queries
        const int64_t qnode = P.qblock0 + (blk - P.block0);
        const int nq = min(kQB, P.qcnt[qnode] - chunk * kQB);
        if (nq > 0) {
            const bool act = tid < nq;
            const int myq = P.qbeg[qnode] + chunk * kQB + tid;
            const int64_t row = P.q0 + myq;  // the query's row in the per-query arrays
            const int kq = P.k;                // read once: stores below could alias P
            const bool mono = P.mono != 0;
            uint64_t q[DP / 2];
            {
                const ulonglong2* q2 = reinterpret_cast<const ulonglong2*>(P.qpts + (int64_t)myq * DP);
#pragma unroll
                for (int j = 0; j < DP / 4; ++j) {
                    const ulonglong2 v = act ? q2[j] : make_ulonglong2(0, 0);
                    q[2 * j] = v.x;
                    q[2 * j + 1] = v.y;
                }
            }
            float ld[KC];
            int li[KC];
#pragma unroll
            for (int j = 0; j < KC; ++j) {
                ld[j] = INFINITY;
                li[j] = kEmptyIdx;
                if (MODE == MODE_MAIN && act) {
                    ld[j] = a.cand_d[(int64_t)j * a.nq_all + row];
                    li[j] = a.cand_i[(int64_t)j * a.nq_all + row];
                }
            }
            const float lam2 = 2.f * P.qlam[qnode];
            const float Bq = a.Bn ? a.Bn[P.node0 + qnode] : INFINITY;
            // the cap pass's bound on the query's k-th distance (main pass only)
            const float qc = MODE == MODE_MAIN && act && a.qcap ? a.qcap[row] : INFINITY;

            // the block's live bound: min(B from the traversal, B_1, B_2)
            auto refresh_bound = [&]() {
                float ub = fminf(ub_op<DP, OP>(list_at(ld, kq - 1)), qc);
                float vmax = act ? ub : -INFINITY, vmin = act ? ub : INFINITY;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
                    vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
                }
                if (lane == 0) {
                    s_rmax[warp] = vmax;
                    s_rmin[warp] = vmin;
                }
                __syncthreads();
                if (tid == 0) {
                    for (int w = 1; w < kQB / 32; ++w) {
                        vmax = fmaxf(vmax, s_rmax[w]);
                        vmin = fminf(vmin, s_rmin[w]);
                    }
                    float b2 = __fadd_ru(vmin, lam2);
                    s_B = fminf(Bq, fminf(vmax, b2));
                }
                __syncthreads();
            };
            refresh_bound();

            const int nseed = MODE == MODE_MAIN ? 0 : seed_count_n(a.seed_nleaf, a.seed_slots, a.seed_eval_slots, blk);
            const int64_t c0 = MODE == MODE_SEED ? 0 : a.csr_off[blk];
            const int64_t c1 = MODE == MODE_SEED ? 0 : a.csr_off[blk + 1];
            const int64_t ntot = nseed + (c1 - c0);
            const int64_t win = MODE == MODE_MAIN ? WINDOW : (ntot > 0 ? ntot : 1);

            for (int64_t w0 = 0; w0 < ntot; w0 += win) {
                const int wn = (int)(ntot - w0 < win ? ntot - w0 : win);
                if (tid == 0) {
                    s_cur = 0;
                    s_part = 0;
                }
                __syncthreads();
                while (s_cur < wn) {
                    // ---- warp 0 fills the stage with whole or partial leaves
                    if (warp == 0)
                        stage_fill<TN, MODE, OP>(a, P, w0, wn, nseed, blk, c0, stab, n_skip,
                                             n_eval, s_cur, s_part, s_nst, s_ntab, s_B);
                    __syncthreads();
                    // ---- all warps copy the staged rows
                    const int ntab = s_ntab, nst = s_nst;
                    for (int t = warp; t < ntab; t += kQB / 32) {
                        int3 e = stab[t];
                        const float4* src = reinterpret_cast<const float4*>(P.rpts) + (int64_t)e.x * (DP / 4);
                        float4* dst = reinterpret_cast<float4*>(rs) + e.z * (DP / 4);
                        for (int f = lane; f < e.y * (DP / 4); f += 32) dst[f] = src[f];
                        for (int i = lane; i < e.y; i += 32) {
                            spos[e.z + i] = e.x + i;
                        }
                    }
                    __syncthreads();
                    // ---- BaseCase over the stage
                    if (act) {
                        for (int e0 = 0; e0 < nst; e0 += 32) {
                            // 32 keys without branches, then the few that may
                            // enter (a bit each), the warp's lanes together
                            const float* rows = rs + e0 * DP;
                            const float tail = ld[KC - 1];
                            uint32_t m = 0;
                            if (nst - e0 >= 32) {
#pragma unroll (DP <= 8 ? 8 : DP <= 16 ? 4 : 2)
                                for (int i = 0; i < 32; ++i)
                                    m |= (sgn * packed_d2<DP>(q, rows + i * DP) <= tail ? 1u : 0u) << i;
                            } else {
                                for (int i = 0; i < nst - e0; ++i)
                                    m |= (sgn * packed_d2<DP>(q, rows + i * DP) <= tail ? 1u : 0u) << i;
                            }
                            while (m) {
                                const int i = __ffs(m) - 1;
                                m &= m - 1;
                                const float key = sgn * packed_d2<DP>(q, rows + i * DP);
                                const int rp = spos[e0 + i];
                                // (the cap pass may have listed this point already)
                                if (key_less(key, rp, ld[KC - 1], li[KC - 1]) && !(mono && rp == myq) &&
                                    !(MODE == MODE_MAIN && listed(li, rp)))
                                    list_insert(ld, li, key, rp);
                            }
                        }
                    }
                    if (tid == 0) n_pp += (unsigned long long)nst * nq;
                    refresh_bound();
                }
                __syncthreads();
            }

            // ---- finish the work item
            if (MODE == MODE_SEED) {
                if (act) {
#pragma unroll
                    for (int j = 0; j < KC; ++j) {
                        a.cand_d[(int64_t)j * a.nq_all + row] = ld[j];
                        a.cand_i[(int64_t)j * a.nq_all + row] = li[j];
                    }
                    // the main pass may keep longer lists: their other rows start empty
                    for (int j = KC; j < a.kc_rows; ++j) {
                        a.cand_d[(int64_t)j * a.nq_all + row] = INFINITY;
                        a.cand_i[(int64_t)j * a.nq_all + row] = kEmptyIdx;
                    }
                    a.qub[row] = ub_op<DP, OP>(list_at(ld, kq - 1));
                }
            } else {
                const float kth = list_at(ld, kq - 1);
                const float band = __fmul_ru(kth, 1.f + 4.f * rel_eps<DP>());
                const bool ovf = act && li[KC - 1] != kEmptyIdx && !(ld[KC - 1] > band);
                if (ovf) {
                    a.fbq_list[atomicAdd(a.fbq_count, 1)] =
                        make_int4(myq, blk, __float_as_int(ub_op<DP, OP>(list_at(ld, kq - 1))), 0);
                } else if (act) {
                    // float64 distances of the band; the float32 order is
                    // theirs but for near-ties, so that sorting them is mostly
                    // one pass that finds nothing to swap
                    double rd[KC];
                    int ri[KC];
                    const float* qp = P.qpts + (int64_t)myq * DP;
#pragma unroll
                    for (int j = 0; j < KC; ++j) {
                        rd[j] = (double)INFINITY;
                        ri[j] = kEmptyIdx;
                        if (li[j] != kEmptyIdx && !(ld[j] > band)) {
                            rd[j] = exact_d2<DP>(qp, P.rpts + (int64_t)li[j] * DP);
                            ri[j] = P.ridx[li[j]];
                            ++n_re;
                        }
                    }
                    for (bool again = true; again;) {
                        again = false;
#pragma unroll
                        for (int j = 0; j + 1 < KC; ++j) {
                            if (key_less(rd[j + 1], ri[j + 1], rd[j], ri[j])) {
                                const double td = rd[j];
                                const int ti = ri[j];
                                rd[j] = rd[j + 1];
                                ri[j] = ri[j + 1];
                                rd[j + 1] = td;
                                ri[j + 1] = ti;
                                again = true;
                            }
                        }
                    }
                    int64_t base = (int64_t)P.qidx[myq] * kq;
#pragma unroll
                    for (int j = 0; j < KC; ++j)
                        if (j < kq) {
                            P.out_idx[base + j] = ri[j];
                            P.out_dist[base + j] = (float)sqrt(rd[j]);
                        }
                }
            }
        }
        __syncthreads();
    }
    // counters: one atomic per thread that holds any
    if (n_skip) atomicAdd(&a.stats[ST_SKIPPED], n_skip);
    if (n_eval) atomicAdd(&a.stats[ST_EVALUATED], n_eval);
    if (n_pp) atomicAdd(&a.stats[MODE == MODE_SEED ? ST_SEED_PAIRS : ST_POINT_PAIRS], n_pp);
    if (n_re) atomicAdd(&a.stats[ST_RERANK], n_re);
}

// Recomputation of one query whose error band overflowed its list, one CTA
// per query.  The candidate leaves are its block's seed leaves and traversal
// candidates; each is kept only if the distance from the query to the leaf's
// box (rounded down) does not exceed the query's upper bound on its k-th
// distance (the single-tree form of Algorithm 3's Score), so the work follows
// the query's own ball, not its block's.  Kept leaves gather in a shared
// buffer; when it fills, the 128 threads evaluate its points, one point each
// in turn, each keeping a candidate list, and the lists are merged.
//   EXACT = false  float32 keys (relative error <= rel_eps): the merged KC
//                  best keys give a band of possible k-th neighbours; if the
//                  band fits the list, its members are re-ranked in float64
//                  and written, else the query goes on to the exact pass.
//   EXACT = true   float64 (distance, index) keys, the result itself.
constexpr int kFbLeafBuf = 512;

template <int DP>
__device__ __forceinline__ float approx_d2(const float* q, const float* r) {
    const float4* r4 = reinterpret_cast<const float4*>(r);
    float f = 0.f;
#pragma unroll
    for (int j = 0; j < DP / 4; ++j) {
        const float4 v = r4[j];
        const float t0 = q[4 * j] - v.x, t1 = q[4 * j + 1] - v.y;
        const float t2 = q[4 * j + 2] - v.z, t3 = q[4 * j + 3] - v.w;
        f = fmaf(t0, t0, f);
        f = fmaf(t1, t1, f);
        f = fmaf(t2, t2, f);
        f = fmaf(t3, t3, f);
    }
    return f;
}

//   stage 0  one CTA per query over all of its candidate leaves (many queries)
//   stage 1  S CTAs per query, each over 1/S of the candidates, each writing
//            the KC best keys of its slice to part (few queries: the scan of
//            one query's candidates then spreads over the GPU)
//   stage 2  one CTA per query merges its S slices' lists and finishes as
//            stage 0 does
template <int DP, int KC, bool EXACT>
__global__ void __launch_bounds__(kQB) k_query_fb(const TileArgs a, int stage, int S, void* part) {
    using T = typename std::conditional<EXACT, double, float>::type;
    extern __shared__ __align__(16) unsigned char fsm[];
    T* md = reinterpret_cast<T*>(fsm);                           // KC x 128
    int32_t* mi = reinterpret_cast<int32_t*>(md + KC * kQB);     // KC x 128
    __shared__ int s_lb[kFbLeafBuf], s_pre[kFbLeafBuf + 1];
    __shared__ int s_n, s_nb;
    __shared__ float s_fd[KC];
    __shared__ int s_fi[KC];
    __shared__ double s_rd[KC];
    __shared__ int s_ri[KC];
    const int fq = stage == 1 ? blockIdx.x / S : blockIdx.x;  // the query's slot in its list
    const int sl = stage == 1 ? blockIdx.x % S : 0;           // stage 1: the CTA's slice
    T* part_d = reinterpret_cast<T*>(part);                   // [query][slice][KC]
    int32_t* part_i = reinterpret_cast<int32_t*>(part_d + (size_t)gridDim.x * (stage == 1 ? 1 : S) * KC);
    const int4 e = (EXACT ? a.fbq2_list : a.fbq_list)[fq];
    const int myq = e.x, blk = e.y;  // query (tree position in its problem), global block
    const ProbDev& P = a.probs[a.blk_prob[blk]];
    const int kq = P.k;  // read once: stores below could alias P
    const bool mono = P.mono != 0;
    const float ub = __int_as_float(e.z);
    const int tid = threadIdx.x;
    float q[DP];
    {
        const float4* q4 = reinterpret_cast<const float4*>(P.qpts + (int64_t)myq * DP);
#pragma unroll
        for (int j = 0; j < DP / 4; ++j) {
            float4 v = q4[j];
            q[4 * j] = v.x;
            q[4 * j + 1] = v.y;
            q[4 * j + 2] = v.z;
            q[4 * j + 3] = v.w;
        }
    }
    T ld[KC];
    int li[KC];
#pragma unroll
    for (int j = 0; j < KC; ++j) {
        ld[j] = (T)INFINITY;
        li[j] = kEmptyIdx;
    }
    if (stage != 2) {
        const int nseed = seed_count(a.seed_nleaf, a.seed_slots, blk);
        const int bound = P.bound;  // read once
        const int64_t c0 = a.csr_off[blk], c1 = a.csr_off[blk + 1];
        const int64_t ntot = nseed + (c1 - c0);
        // this CTA's candidates: all of them, or slice sl of S
        const int64_t c_lo = stage == 1 ? ntot * sl / S : 0, c_hi = stage == 1 ? ntot * (sl + 1) / S : ntot;
        if (tid == 0) s_n = 0;
        __syncthreads();
        for (int64_t base = c_lo; base < c_hi; base += kQB) {
            // 1. test one candidate leaf per thread against the query's ball
            const int64_t c = base + tid;
            int leaf = -1;
            if (c < c_hi) {
                if (c < nseed) {
                    leaf = seed_leaf(a.seed_leaf0, a.seed_nleaf, a.seed_slots, blk, (int)c);
                } else if (!(a.csr_dmin[c0 + c - nseed] > ub)) {
                    leaf = a.csr_leaf[c0 + c - nseed];
                }
                if (leaf >= 0) {
                    const float* bx = P.rbox + (P.rleaf0 + leaf) * 2 * DP;
                    const float dl = bound == DTREE_BOUND_BOX
                                         ? point_box_dmin_down<DP>(q, bx)
                                         : point_dmin_down<DP>(bound, q, bx, P.rlam[P.rleaf0 + leaf]);
                    if (dl > ub) leaf = -1;
                }
            }
            if (leaf >= 0) s_lb[atomicAdd(&s_n, 1)] = leaf;
            __syncthreads();
            // 2. evaluate the buffered leaves once the next round might not fit
            const int nb = s_n;
            const bool flush = nb > 0 && (base + kQB >= c_hi || nb + kQB > kFbLeafBuf);
            __syncthreads();  // every thread has read s_n before the next round adds to it
            if (flush) {
                if (tid == 0) {
                    int acc = 0;
                    for (int i = 0; i < nb; ++i) {
                        s_pre[i] = acc;
                        acc += P.rcnt[P.rleaf0 + s_lb[i]];
                    }
                    s_pre[nb] = acc;
                }
                __syncthreads();
                const int npts = s_pre[nb];
                for (int p = tid; p < npts; p += kQB) {
                    int lo = 0, hi = nb - 1;  // the buffered leaf holding point p
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (s_pre[mid] <= p) lo = mid;
                        else hi = mid - 1;
                    }
                    const int r = P.rbeg[P.rleaf0 + s_lb[lo]] + (p - s_pre[lo]);
                    if (mono && r == myq) continue;
                    if constexpr (EXACT) {
                        const double d2 = exact_d2<DP>(q, P.rpts + (int64_t)r * DP);
                        const int orig = P.ridx[r];
                        if (key_less(d2, orig, ld[KC - 1], li[KC - 1])) list_insert(ld, li, d2, orig);
                    } else {
                        const float d2 = approx_d2<DP>(q, P.rpts + (int64_t)r * DP);
                        if (key_less(d2, r, ld[KC - 1], li[KC - 1])) list_insert(ld, li, d2, r);
                    }
                }
                __syncthreads();
                if (tid == 0) s_n = 0;
                __syncthreads();
            }
        }
    }
    if (stage == 2) {
        // the S slices' lists are the columns to merge (the rest are empty)
        for (int j = 0; j < KC; ++j) {
            md[j * kQB + tid] = tid < S ? part_d[((size_t)fq * S + tid) * KC + j] : (T)INFINITY;
            mi[j * kQB + tid] = tid < S ? part_i[((size_t)fq * S + tid) * KC + j] : kEmptyIdx;
        }
    } else {
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            md[j * kQB + tid] = ld[j];
            mi[j * kQB + tid] = li[j];
        }
    }
    __syncthreads();
    if (stage == 1) {
        // the slice's KC best keys (a merge of the 128 sorted thread lists)
        if (tid == 0) {
            int head[kQB];
            for (int t = 0; t < kQB; ++t) head[t] = 0;
            for (int j = 0; j < KC; ++j) {
                int best = -1;
                T bd = (T)INFINITY;
                int bi = kEmptyIdx;
                for (int t = 0; t < kQB; ++t) {
                    if (head[t] >= KC) continue;
                    const T d = md[head[t] * kQB + t];
                    const int i = mi[head[t] * kQB + t];
                    if (best < 0 || key_less(d, i, bd, bi)) {
                        best = t;
                        bd = d;
                        bi = i;
                    }
                }
                head[best]++;
                part_d[(size_t)blockIdx.x * KC + j] = bd;
                part_i[(size_t)blockIdx.x * KC + j] = bi;
            }
        }
        return;
    }
    const int64_t obase = (int64_t)P.qidx[myq] * kq;
    const int nout = EXACT ? kq : KC;
    if (tid == 0) {
        // merge the 128 sorted lists: the first nout keys overall
        int head[kQB];
        for (int t = 0; t < kQB; ++t) head[t] = 0;
        for (int j = 0; j < nout; ++j) {
            int best = -1;
            T bd = (T)INFINITY;
            int bi = kEmptyIdx;
            for (int t = 0; t < kQB; ++t) {
                if (head[t] >= KC) continue;
                const T d = md[head[t] * kQB + t];
                const int i = mi[head[t] * kQB + t];
                if (best < 0 || key_less(d, i, bd, bi)) {
                    best = t;
                    bd = d;
                    bi = i;
                }
            }
            head[best]++;
            if constexpr (EXACT) {
                P.out_idx[obase + j] = bi;
                P.out_dist[obase + j] = (float)sqrt(bd);
            } else {
                s_fd[j] = bd;
                s_fi[j] = bi;
            }
        }
        if constexpr (!EXACT) {
            // every true k-nearest neighbour has a key <= band; the band must
            // end inside the list, else the float64 pass takes the query
            const float band = __fmul_ru(s_fd[kq - 1], 1.f + 4.f * rel_eps<DP>());
            int n = 0;
            while (n < KC && s_fi[n] != kEmptyIdx && !(s_fd[n] > band)) ++n;
            if (n == KC) {
                a.fbq2_list[atomicAdd(a.fbq2_count, 1)] = e;
                n = -1;
            }
            s_nb = n;
        }
    }
    if constexpr (!EXACT) {
        __syncthreads();
        const int n = s_nb;
        if (n < 0) return;  // uniform: the float64 pass recomputes this query
        if (tid < n) {
            s_rd[tid] = exact_d2<DP>(q, P.rpts + (int64_t)s_fi[tid] * DP);
            s_ri[tid] = P.ridx[s_fi[tid]];
        }
        __syncthreads();
        if (tid == 0) {
            double rd[KC];
            int ri[KC];
#pragma unroll
            for (int j = 0; j < KC; ++j) {
                rd[j] = (double)INFINITY;
                ri[j] = kEmptyIdx;
            }
            for (int j = 0; j < n; ++j) list_insert(rd, ri, s_rd[j], s_ri[j]);
            for (int j = 0; j < kq; ++j) {
                P.out_idx[obase + j] = ri[j];
                P.out_dist[obase + j] = (float)sqrt(rd[j]);
            }
        }
        if (tid == 0) atomicAdd(&a.stats[ST_RERANK], (unsigned long long)n);
    }
}

template <int DP>
int launch_query_fb(const TileArgs& a, int kc, int nfbq, bool exact, cudaStream_t s) {
#define DT_FB_CASE(KCV)                                                                       \
    case KCV: {                                                                               \
        auto kern = exact ? k_query_fb<DP, KCV, true> : k_query_fb<DP, KCV, false>;           \
        const size_t smem = (size_t)KCV * kQB * ((exact ? 8 : 4) + 4);                      \
        DT_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                                      (int)smem));                                            \
        const int S = a.fb_slices > 1 ? a.fb_slices : 1;                                       \
        if (S > 1) {                                                                          \
            DT_LAUNCH(kern, nfbq * S, kQB, smem, s, a, 1, S, a.fb_part);                      \
            DT_LAUNCH(kern, nfbq, kQB, smem, s, a, 2, S, a.fb_part);                          \
        } else {                                                                              \
            DT_LAUNCH(kern, nfbq, kQB, smem, s, a, 0, 1, a.fb_part);                          \
        }                                                                                     \
        return DTREE_OK;                                                                      \
    }
    switch (kc) {
        DT_FB_CASE(4)
        DT_FB_CASE(8)
        DT_FB_CASE(16)
        DT_FB_CASE(24)
        DT_FB_CASE(32)
        DT_FB_CASE(48)
        DT_FB_CASE(64)
        default:
            return DTREE_ERR_UNSUPPORTED;
    }
#undef DT_FB_CASE
}

template <class K>
inline int tile_grid(K kern, int items) {
    int g = occupancy_grid((const void*)kern, kQB, 0);
    return items < g ? (items > 0 ? items : 1) : g;
}

// The cap pass: a budgeted best-first search of the reference tree for every
// query, merged into the query's candidate list.  One warp serves one query
// at a time.  The list starts as the seed pass left it.  From the root the
// search walks down to a leaf, always into the child whose box is nearer
// (the left one on a tie), queueing the farther child with its box
// distance; it offers the leaf's points (itself excluded in a monochromatic
// search) to the list with their float32 keys, the seed pass's keys, then
// resumes from the nearest queued node, until it has evaluated `budget`
// leaves or no queued box is nearer than the list's k-th key.  The block's
// seed leaves are skipped (the seed pass offered their points already), and
// no leaf is reached twice, so no point enters the list twice.  The list
// goes back to cand_d / cand_i, and ub_of of its k-th key, a valid bound on
// the true k-th distance, lowers the query's qub (so B of Section 5 shrinks
// before the traversal) and caps the BaseCase's thresholds.  The BaseCase
// still evaluates every candidate leaf, these included: its insertions skip
// points already listed.
//
// Lane layout: list entry 32 s + lane in (ld[s], li[s]); queue entry `lane`
// in (pd, pn), ascending (32 entries, more than a budget can reach); box
// element e = lane + 32 t of the two children (child e / DP, coordinate
// e % DP), whose query coordinate is qd[t]; point rb + lane (+ 32 u) of a leaf.
constexpr int kCapMaxLeaves = 17;

template <int DP, int KC, int OP = OP_NEAR>
__global__ void __launch_bounds__(kQB) k_query_cap(const TileArgs a, float* qcap, int budget) {
    constexpr int NE = (KC + 31) / 32;      // list entries per lane
    constexpr int NT = (2 * DP + 31) / 32;  // box elements per lane
    constexpr int LPR = DP / 4;             // lanes per point of a leaf
    const int item = blockIdx.x;
    if (item >= a.nitems) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2 wi = a.items[item];
    const int blk = wi.x;
    const ProbDev& P = a.probs[a.blk_prob[blk]];
    const int64_t qnode = P.qblock0 + (blk - P.block0);
    const int nq = min(kQB, P.qcnt[qnode] - wi.y * kQB);
    const int kq = P.k, hr = P.hr;
    const bool mono = P.mono != 0;
    for (int qi = warp + blockIdx.y * (kQB / 32); qi < nq; qi += gridDim.y * (kQB / 32)) {
        const int myq = P.qbeg[qnode] + wi.y * kQB + qi;
        const int64_t row = P.q0 + myq;
        const float* qp = P.qpts + (int64_t)myq * DP;
        // this lane's four coordinates of the query in the leaf evaluation
        const float4 qv = reinterpret_cast<const float4*>(qp)[lane % LPR];
        float qd[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int e = lane + 32 * t;
            qd[t] = e < 2 * DP ? qp[e % DP] : 0.f;
        }
        float ld[NE];
        int li[NE];
#pragma unroll
        for (int s = 0; s < NE; ++s) {
            const int e = 32 * s + lane;
            ld[s] = e < KC ? a.cand_d[(int64_t)e * a.nq_all + row] : INFINITY;
            li[s] = e < KC ? a.cand_i[(int64_t)e * a.nq_all + row] : kEmptyIdx;
        }
        // list entry e (uniform e), broadcast to the warp
        auto entry_d = [&](int e) {
            float v = ld[0];
#pragma unroll
            for (int s = 1; s < NE; ++s)
                if ((e >> 5) == s) v = ld[s];
            return __shfl_sync(0xffffffffu, v, e & 31);
        };
        auto entry_i = [&](int e) {
            int v = li[0];
#pragma unroll
            for (int s = 1; s < NE; ++s)
                if ((e >> 5) == s) v = li[s];
            return __shfl_sync(0xffffffffu, v, e & 31);
        };
        float pd = INFINITY;
        int32_t pn = 0;
        int64_t n = 0;
        int lev = 0;
        float kth = entry_d(kq - 1);
        for (int used = 0;;) {
            for (; lev < hr; ++lev) {
                const int64_t l = 2 * n + 1;
                const float* bx = P.rbox + l * 2 * DP;  // the boxes of children l and l + 1
                // per child: squared distance to its box (s) and to its box
                // centre (u, for the ball bound)
                float s0 = 0.f, s1 = 0.f, u0 = 0.f, u1 = 0.f;
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    const int e = lane + 32 * t;
                    if (e < 2 * DP) {
                        const int c = e / DP, d = e % DP;
                        const float lo = bx[c * 2 * DP + d], hi = bx[c * 2 * DP + DP + d];
                        const float g = OP == OP_FAR ? fmaxf(qd[t] - lo, hi - qd[t])
                                                     : fmaxf(fmaxf(lo - qd[t], qd[t] - hi), 0.f);
                        const float w = qd[t] - 0.5f * (lo + hi);
                        if (c == 0) {
                            s0 = fmaf(g, g, s0);
                            u0 = fmaf(w, w, u0);
                        } else {
                            s1 = fmaf(g, g, s1);
                            u1 = fmaf(w, w, u1);
                        }
                    }
                }
                const bool ball = OP == OP_NEAR && P.bound != DTREE_BOUND_BOX;  // uniform over the warp
                float dl, dr;
                if (2 * DP <= 32) {
                    // child c's coordinates sit in lanes [c DP, c DP + DP)
                    float sv = s0 + s1, uv = u0 + u1;
#pragma unroll
                    for (int off = DP / 2; off > 0; off >>= 1) {
                        sv += __shfl_xor_sync(0xffffffffu, sv, off);
                        if (ball) uv += __shfl_xor_sync(0xffffffffu, uv, off);
                    }
                    dl = __shfl_sync(0xffffffffu, sv, 0);
                    dr = __shfl_sync(0xffffffffu, sv, DP);
                    u0 = __shfl_sync(0xffffffffu, uv, 0);
                    u1 = __shfl_sync(0xffffffffu, uv, DP);
                } else {
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) {
                        s0 += __shfl_xor_sync(0xffffffffu, s0, off);
                        s1 += __shfl_xor_sync(0xffffffffu, s1, off);
                        if (ball) {
                            u0 += __shfl_xor_sync(0xffffffffu, u0, off);
                            u1 += __shfl_xor_sync(0xffffffffu, u1, off);
                        }
                    }
                    dl = s0;
                    dr = s1;
                }
                if (ball) {
                    // squared ball distances max(0, |q - C| - lambda)^2 (an
                    // order and a stopping rule only: any choice is exact)
                    const float gl = fmaxf(sqrtf(u0) - P.rlam[l], 0.f), gr = fmaxf(sqrtf(u1) - P.rlam[l + 1], 0.f);
                    const bool both = P.bound == DTREE_BOUND_BOTH;
                    dl = both ? fmaxf(dl, gl * gl) : gl * gl;
                    dr = both ? fmaxf(dr, gr * gr) : gr * gr;
                }
                if (OP == OP_FAR) {  // negated squared d_max: the farther child is the smaller
                    dl = -dl;
                    dr = -dr;
                }
                const bool right = dr < dl;
                const float df = right ? dl : dr;
                if (df < kth) {
                    // sorted insertion of the farther child (the last entry drops)
                    const int32_t nf = (int32_t)(right ? l : l + 1);
                    const int pos = __popc(__ballot_sync(0xffffffffu, pd <= df));
                    const float upd = __shfl_up_sync(0xffffffffu, pd, 1);
                    const int32_t upn = __shfl_up_sync(0xffffffffu, pn, 1);
                    if (lane > pos) {
                        pd = upd;
                        pn = upn;
                    } else if (lane == pos) {
                        pd = df;
                        pn = nf;
                    }
                }
                n = right ? l + 1 : l;
            }
            if (!in_seed(a.seed_leaf0, a.seed_nleaf, a.seed_slots, blk, (int)(n - P.rleaf0))) {
                const int rb = P.rbeg[n], rc = P.rcnt[n];
                float td = entry_d(KC - 1);
                int ti = entry_i(KC - 1);
                for (int r0 = 0; r0 < rc; r0 += 32) {
                    const int r = rb + r0 + lane;
                    // 32 points, LPR lanes each, in LPR steps: the group that
                    // starts at lane g takes points g, g + 1, ..., so that lane l
                    // ends up with point l's key, and a step's loads are whole
                    // rows.  (A lane per point touched 32 lines with every load
                    // and was bound by L1: seed and cap of 500k queries, d = 64,
                    // 16 leaves 29.2 -> 23.7 ms; of 131k, d = 27 3.6 -> 2.7; d = 16
                    // 11.0 -> 10.8.)
                    float key = 0.f;
#pragma unroll
                    for (int s = 0; s < LPR; ++s) {
                        const int row = min(r0 + lane - lane % LPR + s, rc - 1);
                        const float4 v = reinterpret_cast<const float4*>(P.rpts + (int64_t)(rb + row) * DP)[lane % LPR];
                        const float t0 = qv.x - v.x, t1 = qv.y - v.y, t2 = qv.z - v.z, t3 = qv.w - v.w;
                        float f = fmaf(t3, t3, fmaf(t2, t2, fmaf(t1, t1, t0 * t0)));
#pragma unroll
                        for (int off = LPR / 2; off > 0; off >>= 1) f += __shfl_xor_sync(0xffffffffu, f, off);
                        key = lane % LPR == s ? f : key;
                    }
                    float d = INFINITY;
                    if (r0 + lane < rc && !(mono && r == myq)) d = (OP == OP_FAR ? -1.f : 1.f) * key;
                    uint32_t m = __ballot_sync(0xffffffffu, d < INFINITY && key_less(d, r, td, ti));
                    while (m) {
                        const int src = __ffs(m) - 1;
                        m &= m - 1;
                        const float cd = __shfl_sync(0xffffffffu, d, src);
                        const int ci = __shfl_sync(0xffffffffu, r, src);
                        if (!key_less(cd, ci, td, ti)) continue;
                        // insert (cd, ci): entries from its position on move up one
                        int pos = 0;
#pragma unroll
                        for (int s = 0; s < NE; ++s)
                            pos += __popc(__ballot_sync(0xffffffffu, key_less(ld[s], li[s], cd, ci)));
#pragma unroll
                        for (int s = NE - 1; s >= 0; --s) {
                            float pv = __shfl_up_sync(0xffffffffu, ld[s], 1);
                            int pi = __shfl_up_sync(0xffffffffu, li[s], 1);
                            if (s > 0) {
                                const float cv = __shfl_sync(0xffffffffu, ld[s > 0 ? s - 1 : 0], 31);
                                const int cix = __shfl_sync(0xffffffffu, li[s > 0 ? s - 1 : 0], 31);
                                if (lane == 0) {
                                    pv = cv;
                                    pi = cix;
                                }
                            }
                            const int e = 32 * s + lane;
                            if (e < KC) {
                                if (e > pos) {
                                    ld[s] = pv;
                                    li[s] = pi;
                                } else if (e == pos) {
                                    ld[s] = cd;
                                    li[s] = ci;
                                }
                            }
                        }
                        td = entry_d(KC - 1);
                        ti = entry_i(KC - 1);
                    }
                }
            }
            kth = entry_d(kq - 1);
            const float head = __shfl_sync(0xffffffffu, pd, 0);
            if (++used >= budget || !(head < kth)) break;
            // resume from the nearest queued node
            n = __shfl_sync(0xffffffffu, pn, 0);
            lev = 63 - __clzll((long long)n + 1);
            pd = __shfl_down_sync(0xffffffffu, pd, 1);
            pn = __shfl_down_sync(0xffffffffu, pn, 1);
            if (lane == 31) pd = INFINITY;
        }
#pragma unroll
        for (int s = 0; s < NE; ++s) {
            const int e = 32 * s + lane;
            if (e < KC) {
                a.cand_d[(int64_t)e * a.nq_all + row] = ld[s];
                a.cand_i[(int64_t)e * a.nq_all + row] = li[s];
            }
        }
        if (lane == 0) {
            const float cap = ub_op<DP, OP>(kth);
            qcap[row] = cap;
            a.qub[row] = fminf(a.qub[row], cap);
        }
    }
}

// One CTA per work item, or, where the items alone do not fill the GPU, as many
// as do (a warp then serves a few of the item's queries instead of 32 in a row:
// 64 items at d = 16, 0.60 -> 0.08 ms).
template <int DP, int KC, int OP>
int launch_query_cap_as(const TileArgs& a, int budget, float* qcap, cudaStream_t s) {
    auto kern = k_query_cap<DP, KC, OP>;
    const int split = std::max(1, std::min(32, occupancy_grid((const void*)kern, kQB, 0) / a.nitems));
    DT_LAUNCH(kern, dim3(a.nitems, split), kQB, 0, s, a, qcap, std::min(budget, kCapMaxLeaves));
    return DTREE_OK;
}

template <int DP>
int launch_query_cap(const TileArgs& a, int kc, int budget, float* qcap, cudaStream_t s) {
    if (a.nitems <= 0) return DTREE_OK;
    if (budget < 1 || kc != a.kc_rows) return DTREE_ERR_UNSUPPORTED;
    switch (kc) {
        case 4: return launch_query_cap_as<DP, 4, OP_NEAR>(a, budget, qcap, s);
        case 8: return launch_query_cap_as<DP, 8, OP_NEAR>(a, budget, qcap, s);
        case 16: return launch_query_cap_as<DP, 16, OP_NEAR>(a, budget, qcap, s);
        case 24: return launch_query_cap_as<DP, 24, OP_NEAR>(a, budget, qcap, s);
        case 32: return launch_query_cap_as<DP, 32, OP_NEAR>(a, budget, qcap, s);
        case 48: return launch_query_cap_as<DP, 48, OP_NEAR>(a, budget, qcap, s);
        case 64: return launch_query_cap_as<DP, 64, OP_NEAR>(a, budget, qcap, s);
        default: return DTREE_ERR_UNSUPPORTED;
    }
}

template <int DP>
int launch_tile_cc(const TileArgs& a, int kc, int mode, int items, cudaStream_t s) {
#define DT_TILE_CASE(KCV)                                                                 \
    case KCV:                                                                             \
        if (mode == MODE_SEED) {                                                          \
            auto kern = k_tile<DP, KCV, MODE_SEED>;                                \
            DT_LAUNCH(kern, tile_grid(kern, items), kQB, 0, s, a);                        \
        } else if (mode == MODE_MAIN) {                                                   \
            auto kern = k_tile<DP, KCV, MODE_MAIN>;                                \
            DT_LAUNCH(kern, tile_grid(kern, items), kQB, 0, s, a);                        \
        }                                                                                 \
        return DTREE_OK;
    switch (kc) {
        DT_TILE_CASE(4)
        DT_TILE_CASE(8)
        DT_TILE_CASE(16)
        DT_TILE_CASE(24)
        DT_TILE_CASE(32)
        DT_TILE_CASE(48)
        DT_TILE_CASE(64)
        default:
            return DTREE_ERR_UNSUPPORTED;
    }
#undef DT_TILE_CASE
}

}  // namespace dt
