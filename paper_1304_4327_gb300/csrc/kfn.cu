// kfn.cu -- dtree_kfn: exact k-furthest-neighbour search, host side (the
// kernels and their reading of Section 5 are in kfn.cuh).
#include <algorithm>
#include <cstring>

#include "kfn.cuh"

namespace dt {
namespace {

int kfn_launch(int dp, const KfnArgs& a, int kc, KfnPass pass, int grid, cudaStream_t s) {
    switch (dp) {
        case 4: return launch_kfn<4>(a, kc, pass, grid, s);
        case 8: return launch_kfn<8>(a, kc, pass, grid, s);
        case 16: return launch_kfn<16>(a, kc, pass, grid, s);
        case 32: return launch_kfn<32>(a, kc, pass, grid, s);
        default: return launch_kfn<64>(a, kc, pass, grid, s);
    }
}

// Whether the block search may serve a problem: enough work that its passes pay
// (d > 8, 4096 queries and 1e9 pairs) and lists of at most 64 that hold the 14
// entries beyond k its band wants.  A look at the points then decides
// (probe.cuh: their extents, and what a walk per query would visit).
//
// A walk per query visits few leaves where the box bound prunes well (d <= 8:
// 1M x 100k uniform points in d = 3 3.6 ms against 5.4; 1M x 30k in d = 8 5.9
// against 9.6) and has no passes to pay for (2k queries of 5k points, d = 16:
// 1.1 against 1.7 ms).  Above, blocks of queries share the visits and the
// tensor cores do the distances: 1M x 20k points of the mixture, d = 12, 16,
// 32: 26.5 -> 11.3, 40.8 -> 11.6, 195 -> 19.6 ms; 50k x 20k, d = 16: 5.5 ->
// 3.9; 300k x 5k, d = 10 and 20: 5.4 -> 4.9, 14.7 -> 6.5.
// A band that overflows costs the walk on top: 300k x 50k Gaussian points in d =
// 16, k = 63 took 3608 ms by tiles (nearly all bands overflow a list of 64) and
// take 276 by walks; k = 50 on 20k queries 8.5 by tiles, 93 by walks.
bool kfn_tiles_fit(const dtree_t* tq, const dtree_t* tr, int k) {
    if (tr->dp < 16 || k + 14 > 64 || tq->n < 4096 || (double)tq->n * (double)tr->n < 1e9) return false;
    int major = 0, minor = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, tr->device);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, tr->device);
    return major == 10 && minor == 3;  // the tiles are tcgen05 code
}

int kfn_look(const dtree_t* tq, const dtree_t* tr, int k, ProbeOut* out, cudaStream_t s) {
    ProbeArgs a = probe_args(tq, tr, out);
    a.k = k;
    switch (tr->dp) {
        case 16: return launch_probe_far<16>(a, s);
        case 32: return launch_probe_far<32>(a, s);
        default: return launch_probe_far<64>(a, s);
    }
}

}  // namespace
}  // namespace dt

extern "C" int dtree_kfn(const dtree_t* query, const dtree_t* ref, int32_t k, int64_t* out_idx,
                         float* out_dist, const dtree_opts* o, void* stream, dtree_stats* st) {
    using namespace dt;
    if (st) memset(st, 0, sizeof(*st));
    if (!ref) return DTREE_ERR_INVALID_ARG;
    const bool mono = query == nullptr || query == ref;
    const dtree_t* tq = mono ? ref : query;
    const int64_t m = ref->n, nq = tq->n;
    if (k <= 0 || (mono ? (int64_t)k > m - 1 : (int64_t)k >= m)) return DTREE_ERR_INVALID_K;
    if (!out_idx || !out_dist || tq->d != ref->d) return DTREE_ERR_INVALID_ARG;
    if (o) {
        for (int i = 0; i < 8; ++i)
            if (o->reserved[i]) return DTREE_ERR_INVALID_ARG;
        if (o->precision != DTREE_PREC_FP32 || o->bound != DTREE_BOUND_BOX) return DTREE_ERR_UNSUPPORTED;
    }
    // lists of up to 64 entries; the depth-first stack holds one entry per lane
    if (k > 63 || ref->height > 30) return DTREE_ERR_UNSUPPORTED;
    int dev = 0;
    cudaGetDevice(&dev);
    if (ref->device != dev || tq->device != dev) return DTREE_ERR_INVALID_ARG;
    const int kc = k + 1 <= 16 ? 16 : k + 1 <= 32 ? 32 : 64;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t launches0 = g_launches.load();
    // scratch: three counters, the fallback count, the look's result, and the
    // fallback list
    unsigned char* scratch = nullptr;
    constexpr size_t o_count = 32, o_look = 36, o_list = (o_look + sizeof(ProbeOut) + 15) & ~(size_t)15;
    DT_CHECK(cudaMallocAsync((void**)&scratch, o_list + (size_t)nq * sizeof(int), s));
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    ProbeOut* look = reinterpret_cast<ProbeOut*>(scratch + o_look);
    KfnArgs a{};
    a.qpts = tq->pts;
    a.qidx = tq->idx;
    a.nq = nq;
    a.rpts = ref->pts;
    a.ridx = ref->idx;
    a.rbeg = ref->nbeg;
    a.rcnt = ref->ncnt;
    a.rbox = ref->box;
    a.hr = ref->height;
    a.k = k;
    a.mono = mono ? 1 : 0;
    a.out_idx = out_idx;
    a.out_dist = out_dist;
    a.stats = reinterpret_cast<unsigned long long*>(scratch);
    a.fb_count = reinterpret_cast<int*>(scratch + o_count);
    a.fb_list = reinterpret_cast<int*>(scratch + o_list);
    bool ask = kfn_tiles_fit(tq, ref, k);
    a.gate = ask ? &look->gate : nullptr;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaEvent_t ev[2] = {};
    const bool timed = st && cudaEventCreate(&ev[0]) == cudaSuccess && cudaEventCreate(&ev[1]) == cudaSuccess;
    cudaGetLastError();
    int rc = DTREE_OK;
    int hv[2] = {0, 0};  // the fallback count, and whether the block search serves the call
    int& nfb = hv[0];
    unsigned long long cnt[3] = {0, 0, 0};
    bool tiles = false;
    for (;; ask = false, a.gate = nullptr) {
        if (cudaMemsetAsync(scratch, 0, o_look + 8, s) != cudaSuccess) { rc = cuda_status(cudaGetLastError()); break; }
        if (timed) cudaEventRecord(ev[0], s);
        if (ask && (rc = kfn_look(tq, ref, k, look, s)) != DTREE_OK) break;
        // one warp per query, four per CTA; a grid of whole waves of CTAs
        const int64_t want = (nq + 3) / 4;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 16));
        rc = kfn_launch(ref->dp, a, kc, KFN_ALL, grid, s);
        if (rc != DTREE_OK) break;
        if (cudaMemcpyAsync(hv, a.fb_count, sizeof(hv), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            rc = cuda_status(cudaGetLastError());
            break;
        }
        if (ask && hv[1]) {
            rc = kfn_by_tiles(tq, ref, mono, k, out_idx, out_dist, s, st);
            tiles = rc == DTREE_OK;
            // (its operand rows or candidate pairs may not fit where the walks,
            // which need 4 bytes a query, do, and its waits are bounded where the
            // walks wait for nothing)
            if (rc != DTREE_ERR_OOM && rc != DTREE_ERR_TIMEOUT) break;
            if (st) memset(st, 0, sizeof(*st));
            continue;
        }
        if (nfb > 0) {
            a.in_list = a.fb_list;
            a.in_count = a.fb_count;
            const int g2 = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)nfb + 3) / 4, (int64_t)sms * 16));
            rc = kfn_launch(ref->dp, a, kc, KFN_EXACT, g2, s);
            if (rc != DTREE_OK) break;
        }
        if (timed) cudaEventRecord(ev[1], s);
        if (st && cudaMemcpyAsync(cnt, a.stats, sizeof(cnt), cudaMemcpyDeviceToHost, s) != cudaSuccess) {
            rc = cuda_status(cudaGetLastError());
            break;
        }
        if (cudaStreamSynchronize(s) != cudaSuccess) rc = cuda_status(cudaGetLastError());
        break;
    }
    cudaFreeAsync(scratch, s);
    if (rc == DTREE_OK && cudaStreamSynchronize(s) != cudaSuccess) rc = cuda_status(cudaGetLastError());
    if (st && tiles) {
        st->point_pairs += st->seed_point_pairs;
        st->kernel_launches = g_launches.load() - launches0;
    } else if (st && rc == DTREE_OK) {
        st->point_pairs = (int64_t)cnt[0];
        st->leaf_pairs_evaluated = (int64_t)cnt[1];
        st->node_pairs_pruned = (int64_t)cnt[2];
        st->fallback_queries = nfb;
        st->fallback64_queries = nfb;
        float ms = 0.f;
        if (timed && cudaEventElapsedTime(&ms, ev[0], ev[1]) == cudaSuccess) st->ns_basecase = (int64_t)(ms * 1e6);
        st->kernel_launches = g_launches.load() - launches0;
    }
    if (timed) {
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
    }
    cudaGetLastError();
    return rc;
}
