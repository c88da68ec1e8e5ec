// scan.cuh -- exclusive prefix sums of int64 counts (range search's offsets,
// the spanning tree's edge slots).
//
// Memory-bound: read once, written twice (block-local sums, then the blocks'
// offsets added).  One CTA whose threads each walk a chunk of their own reads
// uncoalesced, with one load in flight per thread: its time grew with n / 1024
// serial steps (part of what made the spanning tree's rounds on 1M points cost
// a millisecond each beside their search).
#pragma once

#include "dtree_internal.cuh"

namespace dt {

constexpr int kScanThreads = 1024, kScanEach = 4, kScanBlock = kScanThreads * kScanEach;

inline int64_t scan_blocks(int64_t n) { return (n + kScanBlock - 1) / kScanBlock; }

// Exclusive prefix of v over the CTA; total is the CTA's sum.
__device__ __forceinline__ int64_t scan_cta(int64_t v, int64_t& total) {
    __shared__ int64_t ws[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t t = ws[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t u = __shfl_up_sync(0xffffffffu, t, off);
            if (lane >= off) t += u;
        }
        ws[lane] = t;
    }
    __syncthreads();
    total = ws[kScanThreads / 32 - 1];
    const int64_t excl = incl - v + (warp > 0 ? ws[warp - 1] : 0);
    __syncthreads();  // ws may be written again
    return excl;
}

// Each CTA scans its kScanBlock counts in place; sums[b] is its total.
static __global__ void __launch_bounds__(kScanThreads) k_scan_local(int64_t* a, int64_t n, int64_t* sums) {
    const int64_t i0 = (int64_t)blockIdx.x * kScanBlock + threadIdx.x * kScanEach;
    int64_t v[kScanEach], s = 0;
#pragma unroll
    for (int e = 0; e < kScanEach; ++e) {
        v[e] = i0 + e < n ? a[i0 + e] : 0;
        s += v[e];
    }
    int64_t total;
    int64_t run = scan_cta(s, total);
#pragma unroll
    for (int e = 0; e < kScanEach; ++e) {
        if (i0 + e < n) a[i0 + e] = run;
        run += v[e];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// The block sums, in place (one CTA), and the grand total.
static __global__ void __launch_bounds__(kScanThreads) k_scan_sums(int64_t* sums, int64_t nb, int64_t* grand) {
    int64_t carry = 0;
    for (int64_t b = 0; b < nb; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        int64_t total;
        const int64_t excl = scan_cta(i < nb ? sums[i] : 0, total);
        if (i < nb) sums[i] = carry + excl;
        carry += total;
    }
    if (threadIdx.x == 0) *grand = carry;
}

static __global__ void __launch_bounds__(kScanThreads) k_scan_add(int64_t* a, int64_t n, const int64_t* sums) {
    const int64_t base = sums[blockIdx.x];
    const int64_t i0 = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
#pragma unroll
    for (int e = 0; e < kScanEach; ++e)
        if (i0 + e * kScanThreads < n) a[i0 + e * kScanThreads] += base;
}

// In place: a[0..n) -> exclusive prefix sums, a[n] = the total; sums holds
// scan_blocks(n) values.
static inline int exclusive_scan(int64_t* a, int64_t n, int64_t* sums, cudaStream_t s) {
    const int nb = (int)scan_blocks(n);
    DT_LAUNCH(k_scan_local, nb, kScanThreads, 0, s, a, n, sums);
    DT_LAUNCH(k_scan_sums, 1, kScanThreads, 0, s, sums, (int64_t)nb, a + n);
    if (nb > 1) DT_LAUNCH(k_scan_add, nb, kScanThreads, 0, s, a, n, sums);
    return DTREE_OK;
}

}  // namespace dt
