// range.cu -- dtree_range_count / dtree_range_fill: exact range search, host
// side (the kernels and their reading of Section 6 are in range.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "range.cuh"
#include "scan.cuh"

namespace dt {
namespace {

int range_launch(int dp, const RangeArgs& a, bool fill, int grid, cudaStream_t s) {
    switch (dp) {
        case 4: return launch_range<4>(a, fill, grid, s);
        case 8: return launch_range<8>(a, fill, grid, s);
        case 16: return launch_range<16>(a, fill, grid, s);
        case 32: return launch_range<32>(a, fill, grid, s);
        default: return launch_range<64>(a, fill, grid, s);
    }
}

// Shared argument checks; fills the tree fields and the float bounds.
int range_setup(const dtree_t* query, const dtree_t* ref, double d_lo, double d_hi,
                const dtree_opts* o, RangeArgs* a) {
    if (!ref) return DTREE_ERR_INVALID_ARG;
    const bool mono = query == nullptr || query == ref;
    const dtree_t* tq = mono ? ref : query;
    if (tq->d != ref->d) return DTREE_ERR_INVALID_ARG;
    if (!(d_lo >= 0.0) || !(d_hi >= d_lo)) return DTREE_ERR_INVALID_ARG;  // (NaN fails both)
    if (o) {
        for (int i = 0; i < 8; ++i)
            if (o->reserved[i]) return DTREE_ERR_INVALID_ARG;
        if (o->precision != DTREE_PREC_FP32 || o->bound != DTREE_BOUND_BOX) return DTREE_ERR_UNSUPPORTED;
    }
    if (ref->height > 30) return DTREE_ERR_UNSUPPORTED;  // the depth-first stack: one entry per lane
    int dev = 0;
    cudaGetDevice(&dev);
    if (ref->device != dev || tq->device != dev) return DTREE_ERR_INVALID_ARG;
    memset(a, 0, sizeof(*a));
    a->qpts = tq->pts;
    a->qidx = tq->idx;
    a->nq = tq->n;
    a->rpts = ref->pts;
    a->ridx = ref->idx;
    a->rbeg = ref->nbeg;
    a->rcnt = ref->ncnt;
    a->rbox = ref->box;
    a->hr = ref->height;
    a->mono = mono ? 1 : 0;
    a->d_lo = d_lo;
    a->d_hi = d_hi;
    // floats below and above the squared ends, 1e-12 apart from them
    const double lo2 = d_lo * d_lo, hi2 = d_hi * d_hi;
    a->lo2_dn = std::nextafter((float)(lo2 * (1.0 - 1e-12)), -INFINITY);
    a->lo2_up = std::nextafter((float)(lo2 * (1.0 + 1e-12)), INFINITY);
    a->hi2_dn = std::isinf(hi2) ? INFINITY : std::nextafter((float)(hi2 * (1.0 - 1e-12)), -INFINITY);
    a->hi2_up = std::isinf(hi2) ? INFINITY : std::nextafter((float)(hi2 * (1.0 + 1e-12)), INFINITY);
    if (a->lo2_dn < 0.f) a->lo2_dn = 0.f;
    return DTREE_OK;
}

int range_grid(int64_t nq) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)std::max<int64_t>(1, std::min<int64_t>((nq + 3) / 4, (int64_t)sms * 16));
}

RangeOut range_out(const RangeArgs& a, bool fill) {
    RangeOut r{};
    r.d_lo = a.d_lo;
    r.d_hi = a.d_hi;
    const float hi = (float)(a.d_hi * (1.0 + 1e-12));
    r.hi_up = std::isinf(hi) ? hi : std::nextafter(hi, INFINITY);
    r.lo2_dn = a.lo2_dn;
    r.lo2_up = a.lo2_up;
    r.hi2_dn = a.hi2_dn;
    r.hi2_up = a.hi2_up;
    r.fill = fill ? 1 : 0;
    r.counts = a.counts;
    r.offsets = a.offsets;
    r.out_idx = a.out_idx;
    r.out_dist = a.out_dist;
    return r;
}

// Whether the block search may serve a range: enough work that its passes pay
// (d > 8, 10k queries and 1e9 pairs) and a candidate bit per (block, leaf) in at
// most 1 GB.  A look at the points then decides (probe.cuh: their extents, what a
// walk would visit, and how many of the points it evaluates are results).  Both
// passes of a search decide alike.
//
// A walk per query visits few leaves where the box bound prunes well (d <= 8),
// and a few queries make too few blocks for the GPU (mixture, d = 16, radius
// 2.4: 1M x 2k points 5.3 against 6.9 ms, 300k x 5k 4.4 against 4.6).  Above,
// blocks share the visits and the tensor cores do the distances: 100k x 20k
// 4.2 -> 3.9 ms, 1M x 20k 16.5 -> 6.9, 1M x 100k 64 -> 10.3; 300k x 100k in d =
// 32 91 -> 13; 100k x 20k in d = 64 179 -> 21.
bool range_tiles_fit(const dtree_t* tq, const dtree_t* tr) {
    if (tr->dp < 16 || tq->n < 10000 || (double)tq->n * (double)tr->n < 1e9) return false;
    if ((double)tq->n / 64.0 * (double)tr->nleaves / 8.0 > 1e9) return false;
    int major = 0, minor = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, tr->device);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, tr->device);
    return major == 10 && minor == 3;  // the tiles are tcgen05 code
}

int range_look(const dtree_t* tq, const dtree_t* tr, const RangeArgs& r, ProbeOut* out, cudaStream_t s) {
    ProbeArgs a = probe_args(tq, tr, out);
    a.lo2_dn = r.lo2_dn;
    a.hi2_up = r.hi2_up;
    a.hi_up = range_out(r, false).hi_up;
    if (cudaMemsetAsync(out, 0, 8, s) != cudaSuccess) return cuda_status(cudaGetLastError());
    switch (tr->dp) {
        case 16: return launch_probe_range<16>(a, s);
        case 32: return launch_probe_range<32>(a, s);
        default: return launch_probe_range<64>(a, s);
    }
}

}  // namespace
}  // namespace dt

extern "C" int dtree_range_count(const dtree_t* query, const dtree_t* ref, double d_lo, double d_hi,
                                 int64_t* offsets, int64_t* total, const dtree_opts* o, void* stream,
                                 dtree_stats* st) {
    using namespace dt;
    if (st) memset(st, 0, sizeof(*st));
    RangeArgs a;
    int rc = range_setup(query, ref, d_lo, d_hi, o, &a);
    if (rc != DTREE_OK) return rc;
    if (!offsets || !total) return DTREE_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t launches0 = g_launches.load();
    const dtree_t* tq = query ? query : ref;
    // scratch: four counters, the look's result and the scan's block sums
    unsigned long long* cnt = nullptr;
    constexpr size_t n_look = (sizeof(ProbeOut) + 7) / 8;
    DT_CHECK(cudaMallocAsync((void**)&cnt, (4 + n_look + (size_t)scan_blocks(a.nq)) * sizeof(unsigned long long), s));
    ProbeOut* look = reinterpret_cast<ProbeOut*>(cnt + 4);
    int64_t* sums = reinterpret_cast<int64_t*>(cnt + 4 + n_look);
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    a.counts = offsets;
    a.stats = cnt;
    unsigned long long h[5] = {0, 0, 0, 0, 0};  // the counters, and the look's verdict (its low half)
    dtree_stats tst{};  // the block search's counters
    cudaEvent_t ev[2] = {};
    const bool timed = st && cudaEventCreate(&ev[0]) == cudaSuccess && cudaEventCreate(&ev[1]) == cudaSuccess;
    cudaGetLastError();
    bool ask = range_tiles_fit(tq, ref), tiles = false;
    for (;;) {
        a.gate = ask ? &look->gate : nullptr;
        if (cudaMemsetAsync(cnt, 0, 5 * sizeof(unsigned long long), s) != cudaSuccess) {
            rc = cuda_status(cudaGetLastError());
            break;
        }
        if (timed) cudaEventRecord(ev[0], s);
        if (ask && (rc = range_look(tq, ref, a, look, s)) != DTREE_OK) break;
        if (tiles) {
            rc = range_by_tiles(tq, ref, a.mono != 0, range_out(a, false), s, st ? &tst : nullptr);
            if (rc == DTREE_ERR_OOM || rc == DTREE_ERR_TIMEOUT) tiles = false;  // (the walk needs no memory and has no waits)
            else if (rc != DTREE_OK) break;
        }
        if (!tiles && (rc = range_launch(ref->dp, a, false, range_grid(a.nq), s)) != DTREE_OK) break;
        // (before the verdict is known: sums of nothing in particular where the
        // walks stood back)
        rc = exclusive_scan(offsets, a.nq, sums, s);
        if (rc != DTREE_OK) break;
        if (timed) cudaEventRecord(ev[1], s);
        if (cudaMemcpyAsync(total, offsets + a.nq, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            rc = cuda_status(cudaGetLastError());
            break;
        }
        if (!ask || (uint32_t)h[4] == 0) break;
        ask = false;
        tiles = true;
    }
    cudaFreeAsync(cnt, s);
    if (cudaStreamSynchronize(s) != cudaSuccess && rc == DTREE_OK) rc = cuda_status(cudaGetLastError());
    if (st && rc == DTREE_OK) {
        float ms = 0.f;
        if (tiles) {
            *st = tst;  // its counters and phases
        } else {
            st->point_pairs = (int64_t)h[0];
            st->leaf_pairs_evaluated = (int64_t)h[1];
            st->node_pairs_pruned = (int64_t)h[2];
            st->rerank_candidates = (int64_t)h[3];
            if (timed && cudaEventElapsedTime(&ms, ev[0], ev[1]) == cudaSuccess) st->ns_basecase = (int64_t)(ms * 1e6);
        }
        st->kernel_launches = g_launches.load() - launches0;
    }
    if (timed) {
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
    }
    cudaGetLastError();
    return rc;
}

extern "C" int dtree_range_fill(const dtree_t* query, const dtree_t* ref, double d_lo, double d_hi,
                                const int64_t* offsets, int64_t* out_idx, float* out_dist,
                                const dtree_opts* o, void* stream) {
    using namespace dt;
    RangeArgs a;
    int rc = range_setup(query, ref, d_lo, d_hi, o, &a);
    if (rc != DTREE_OK) return rc;
    if (!offsets || !out_idx || !out_dist) return DTREE_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    a.offsets = offsets;
    a.out_idx = out_idx;
    a.out_dist = out_dist;
    const dtree_t* tq = query ? query : ref;
    int verdict = 0;
    ProbeOut* look = nullptr;
    if (range_tiles_fit(tq, ref) && scratch(&look, 1, s) == DTREE_OK) {
        a.gate = &look->gate;
        rc = range_look(tq, ref, a, look, s);
    }
    if (rc == DTREE_OK) rc = range_launch(ref->dp, a, true, range_grid(a.nq), s);
    if (rc == DTREE_OK && look && (cudaMemcpyAsync(&verdict, &look->gate, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                                   cudaStreamSynchronize(s) != cudaSuccess))
        rc = cuda_status(cudaGetLastError());
    if (look) cudaFreeAsync(look, s);
    if (rc == DTREE_OK && verdict) {
        a.gate = nullptr;
        rc = range_by_tiles(tq, ref, a.mono != 0, range_out(a, true), s, nullptr);
        if (rc == DTREE_ERR_OOM || rc == DTREE_ERR_TIMEOUT) rc = range_launch(ref->dp, a, true, range_grid(a.nq), s);
    }
    if (cudaStreamSynchronize(s) != cudaSuccess && rc == DTREE_OK) rc = cuda_status(cudaGetLastError());
    return rc;
}
