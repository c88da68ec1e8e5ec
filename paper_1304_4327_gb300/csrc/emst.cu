// emst.cu -- dtree_emst: the Euclidean minimum spanning tree by Boruvka
// rounds, host side and the round's small kernels (the nearest-edge search
// and the reading of Section 7 are in emst.cuh).
#include <algorithm>
#include <cstring>

#include "emst.cuh"
#include "scan.cuh"

namespace dt {
namespace {

// The start: every point its own component.
__global__ void k_emst_iota(int32_t* v, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) v[i] = (int32_t)i;
}

// Labels of the lowest levels: a CTA labels up to kLabLeaves leaves (one per
// thread: the component all its points share, else -1) and the nodes above
// them, up to the one that covers them all.
constexpr int kLabLeaves = 256;

__device__ __forceinline__ int32_t lab_join(int32_t a, int32_t b) { return a == b && a >= 0 ? a : -1; }

__global__ void __launch_bounds__(kLabLeaves) k_emst_labels(const int32_t* comp, const int32_t* nbeg,
                                                            const int32_t* ncnt, int h, int up, int32_t* nlab) {
    __shared__ int32_t lab[kLabLeaves];
    const int64_t leaf0 = ((int64_t)1 << h) - 1;
    const int64_t first = (int64_t)blockIdx.x << up;  // this CTA's first leaf, of 2^up
    const int t = threadIdx.x;
    if (t < (1 << up)) {
        const int64_t nd = leaf0 + first + t;
        const int b = nbeg[nd], c = ncnt[nd];
        int32_t l = c > 0 ? comp[b] : -1;
        for (int j = 1; j < c && l >= 0; ++j)
            if (comp[b + j] != l) l = -1;
        nlab[nd] = lab[t] = l;
    }
    for (int v = 1; v <= up; ++v) {
        __syncthreads();
        const int cnt = 1 << (up - v);
        const int32_t l = t < cnt ? lab_join(lab[2 * t], lab[2 * t + 1]) : -1;
        __syncthreads();
        if (t < cnt) {
            lab[t] = l;
            nlab[((int64_t)1 << (h - v)) - 1 + (first >> v) + t] = l;
        }
    }
}

// The levels above, from `level` up to the root (one CTA).
__global__ void __launch_bounds__(1024) k_emst_labels_top(int level, int32_t* nlab) {
    for (int L = level; L >= 0; --L) {
        const int64_t cnt = (int64_t)1 << L;
        for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
            const int64_t nd = cnt - 1 + i;
            nlab[nd] = lab_join(nlab[2 * nd + 1], nlab[2 * nd + 2]);
        }
        __syncthreads();
    }
}

// What a round's components start with.
__global__ void k_emst_reset(int64_t n, unsigned long long* ck1, unsigned long long* ck2, int32_t* pick,
                             uint32_t* cub) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    ck1[i] = ck2[i] = ~0ull;
    pick[i] = -1;
    cub[i] = 0x7f800000u;  // +inf
}

// Among the points that reach their component's shortest length: the lowest
// pair of endpoints ...
__global__ void k_emst_min2(const int32_t* comp, const double* bd, const int32_t* br,
                            const int32_t* idx, int64_t n, const unsigned long long* ck1,
                            unsigned long long* ck2) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || br[i] < 0 || dkey(bd[i]) != ck1[comp[i]]) return;
    const uint32_t a = (uint32_t)idx[i], b = (uint32_t)idx[br[i]];
    atomicMin(&ck2[comp[i]], ((unsigned long long)min(a, b) << 32) | max(a, b));
}

// ... and the one point of the component that holds it.
__global__ void k_emst_pick(const int32_t* comp, const double* bd, const int32_t* br,
                            const int32_t* idx, int64_t n, const unsigned long long* ck1,
                            const unsigned long long* ck2, int32_t* pick) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || br[i] < 0) return;
    const int32_t c = comp[i];
    if (dkey(bd[i]) != ck1[c]) return;
    const uint32_t a = (uint32_t)idx[i], b = (uint32_t)idx[br[i]];
    if ((((unsigned long long)min(a, b) << 32) | max(a, b)) == ck2[c]) pick[c] = (int32_t)i;
}

// Hooks: a component points to the one across its edge; of two components
// that chose the same edge, the lower id stays a root and writes the edge.
// adds[b] counts the edges that components [1024 b, 1024 (b + 1)) write.
constexpr int kHookCta = 1024;

__device__ __forceinline__ bool emst_hook_of(int64_t c, int64_t n, const int32_t* comp, const int32_t* br,
                                             const int32_t* pick, const unsigned long long* ck1,
                                             const unsigned long long* ck2, int32_t* par) {
    if (c >= n) return false;
    const int32_t p = pick[c];
    if (p < 0) {
        if (par) par[c] = (int32_t)c;
        return false;
    }
    const int32_t o = comp[br[p]];
    const bool mutual = pick[o] >= 0 && ck1[o] == ck1[c] && ck2[o] == ck2[c];
    if (par) par[c] = (mutual && c < o) ? (int32_t)c : o;
    return !mutual || c < o;
}

__global__ void __launch_bounds__(kHookCta) k_emst_hook(const int32_t* comp, const int32_t* br, const int32_t* pick,
                                                        const unsigned long long* ck1,
                                                        const unsigned long long* ck2, int64_t n, int32_t* par,
                                                        int64_t* adds) {
    const int64_t c = blockIdx.x * (int64_t)kHookCta + threadIdx.x;
    const int cnt = __syncthreads_count(emst_hook_of(c, n, comp, br, pick, ck1, ck2, par));
    if (threadIdx.x == 0) adds[blockIdx.x] = cnt;
}

// The round's edges, in component-id order after the ones written before.
__global__ void __launch_bounds__(kHookCta) k_emst_emit(const int32_t* comp, const int32_t* pick, const int32_t* br,
                                                        const double* bd, const int32_t* idx,
                                                        const unsigned long long* ck1, const unsigned long long* ck2,
                                                        const int64_t* offs, int64_t n, int64_t base, int64_t* edges,
                                                        float* dist) {
    __shared__ int before[kHookCta / 32];
    const int64_t c = blockIdx.x * (int64_t)kHookCta + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool add = emst_hook_of(c, n, comp, br, pick, ck1, ck2, nullptr);
    const unsigned m = __ballot_sync(0xffffffffu, add);
    if (lane == 0) before[warp] = __popc(m);
    __syncthreads();
    if (!add) return;
    int64_t slot = base + offs[blockIdx.x] + __popc(m & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) slot += before[w];
    if (slot >= n - 1) return;  // (cannot happen: the host reports a count other than n - 1)
    const int32_t p = pick[c];
    const int32_t a = idx[p], b = idx[br[p]];
    edges[2 * slot] = min(a, b);
    edges[2 * slot + 1] = max(a, b);
    dist[slot] = (float)sqrt(bd[p]);
}

// Every component's root.  Each thread moves its own pointer to its
// grandparent until that is a root; the others' moves shorten its way, so
// that a chain of n takes about log n steps, and since a pointer only ever
// moves to an ancestor the order of the moves does not matter.
__global__ void k_emst_roots(int32_t* par, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    volatile int32_t* v = par;
    int32_t p = v[i];
    for (int64_t step = 0; step < n; ++step) {  // (a root is fewer than n steps away)
        const int32_t g = v[p];
        if (g == p) break;
        v[i] = p = g;
    }
}

__global__ void k_emst_relabel(int32_t* comp, const int32_t* par, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) comp[i] = par[comp[i]];
}

int emst_nn(int dp, const EmstArgs& a, cudaStream_t s) {
    switch (dp) {
        case 4: return launch_emst_nn<4>(a, s);
        case 8: return launch_emst_nn<8>(a, s);
        case 16: return launch_emst_nn<16>(a, s);
        case 32: return launch_emst_nn<32>(a, s);
        default: return launch_emst_nn<64>(a, s);
    }
}

inline int g256(int64_t n) { return (int)std::max<int64_t>(1, (n + 255) / 256); }

}  // namespace
}  // namespace dt

extern "C" int dtree_emst(const dtree_t* t, int64_t* out_edges, float* out_dist, const dtree_opts* o,
                          void* stream, dtree_stats* st) {
    using namespace dt;
    if (st) memset(st, 0, sizeof(*st));
    if (!t) return DTREE_ERR_INVALID_ARG;
    const int64_t n = t->n;
    if (n > 1 && (!out_edges || !out_dist)) return DTREE_ERR_INVALID_ARG;
    if (o) {
        for (int i = 0; i < 8; ++i)
            if (o->reserved[i]) return DTREE_ERR_INVALID_ARG;
        if (o->precision != DTREE_PREC_FP32 || o->bound != DTREE_BOUND_BOX) return DTREE_ERR_UNSUPPORTED;
    }
    if (t->height > 30) return DTREE_ERR_UNSUPPORTED;  // the depth-first stack: one entry per lane
    int dev = 0;
    cudaGetDevice(&dev);
    if (t->device != dev) return DTREE_ERR_INVALID_ARG;
    if (n < 2) return DTREE_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t launches0 = g_launches.load();
    const int64_t nn = t->nnodes;
    const int64_t nhook = (n + kHookCta - 1) / kHookCta;
    // scratch, one block: comp, br, pick, par, lb, cub (4 n bytes each), nlab
    // (4 bytes per node), bd, ck1, ck2 (8 n bytes each), done (n bytes), adds
    // (8 bytes per 1024 components, and one), counters
    const size_t b4 = (size_t)n * 4, b8 = (size_t)n * 8;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t bytes = 0;
    auto room = [&](size_t x) {
        const size_t at = bytes;
        bytes = al(bytes + x);
        return at;
    };
    const size_t o_comp = room(b4), o_br = room(b4), o_pick = room(b4), o_par = room(b4), o_lb = room(b4),
                 o_cub = room(b4), o_nlab = room((size_t)nn * 4), o_bd = room(b8), o_ck1 = room(b8),
                 o_ck2 = room(b8), o_done = room((size_t)n), o_adds = room((size_t)(nhook + 1) * 8),
                 o_cnt = room(16);
    unsigned char* m = nullptr;
    DT_CHECK(cudaMallocAsync((void**)&m, bytes, s));
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    int32_t* comp = reinterpret_cast<int32_t*>(m + o_comp);
    int32_t* br = reinterpret_cast<int32_t*>(m + o_br);
    int32_t* pick = reinterpret_cast<int32_t*>(m + o_pick);
    int32_t* par = reinterpret_cast<int32_t*>(m + o_par);
    uint32_t* cub = reinterpret_cast<uint32_t*>(m + o_cub);
    int32_t* nlab = reinterpret_cast<int32_t*>(m + o_nlab);
    double* bd = reinterpret_cast<double*>(m + o_bd);
    unsigned long long* ck1 = reinterpret_cast<unsigned long long*>(m + o_ck1);
    unsigned long long* ck2 = reinterpret_cast<unsigned long long*>(m + o_ck2);
    int64_t* adds = reinterpret_cast<int64_t*>(m + o_adds);
    unsigned long long* cstats = reinterpret_cast<unsigned long long*>(m + o_cnt);
    EmstArgs a{};
    a.pts = t->pts;
    a.idx = t->idx;
    a.nbeg = t->nbeg;
    a.ncnt = t->ncnt;
    a.box = t->box;
    a.n = n;
    a.hr = t->height;
    a.pk1 = make_packets(t, 0);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    a.pk = make_packets(t, packet_lanes(n, sms));
    a.first = 1;
    a.comp = comp;
    a.nlab = nlab;
    a.bd = bd;
    a.br = br;
    a.lb = reinterpret_cast<float*>(m + o_lb);
    a.done = m + o_done;
    a.cub = cub;
    a.ck1 = ck1;
    a.stats = cstats;
    // leaves per CTA of the label kernel: a power of two
    const int up = std::min<int>(t->height, 8);
    const int nlabcta = 1 << (t->height - up);
    cudaEvent_t ev[2] = {};
    const bool timed = st && cudaEventCreate(&ev[0]) == cudaSuccess && cudaEventCreate(&ev[1]) == cudaSuccess;
    cudaGetLastError();
    int rc = DTREE_OK;
    int64_t base = 0;
    unsigned long long hs[2] = {0, 0};
    auto launch_ok = [&](int launches) {
        g_launches.fetch_add(launches, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess;
    };
    do {
        if (cudaMemsetAsync(cstats, 0, 16, s) != cudaSuccess) { rc = DTREE_ERR_CUDA; break; }
        if (timed) cudaEventRecord(ev[0], s);
        k_emst_iota<<<g256(n), 256, 0, s>>>(comp, n);
        if (!launch_ok(1)) { rc = DTREE_ERR_CUDA; break; }
        // each round at least halves the number of components
        for (int round = 0; round < 64 && base < n - 1 && rc == DTREE_OK; ++round) {
            k_emst_labels<<<nlabcta, kLabLeaves, 0, s>>>(comp, t->nbeg, t->ncnt, t->height, up, nlab);
            if (t->height > up) k_emst_labels_top<<<1, 1024, 0, s>>>(t->height - up - 1, nlab);
            k_emst_reset<<<g256(n), 256, 0, s>>>(n, ck1, ck2, pick, cub);
            if (!launch_ok(t->height > up ? 3 : 2)) { rc = DTREE_ERR_CUDA; break; }
            rc = emst_nn(t->dp, a, s);
            if (rc != DTREE_OK) break;
            a.first = 0;
            k_emst_min2<<<g256(n), 256, 0, s>>>(comp, bd, br, t->idx, n, ck1, ck2);
            k_emst_pick<<<g256(n), 256, 0, s>>>(comp, bd, br, t->idx, n, ck1, ck2, pick);
            k_emst_hook<<<(int)nhook, kHookCta, 0, s>>>(comp, br, pick, ck1, ck2, n, par, adds);
            k_scan_sums<<<1, kScanThreads, 0, s>>>(adds, nhook, adds + nhook);
            k_emst_emit<<<(int)nhook, kHookCta, 0, s>>>(comp, pick, br, bd, t->idx, ck1, ck2, adds, n, base,
                                                        out_edges, out_dist);
            k_emst_roots<<<g256(n), 256, 0, s>>>(par, n);
            k_emst_relabel<<<g256(n), 256, 0, s>>>(comp, par, n);
            if (!launch_ok(7)) { rc = DTREE_ERR_CUDA; break; }
            int64_t added = 0;
            if (cudaMemcpyAsync(&added, adds + nhook, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess) {
                rc = DTREE_ERR_CUDA;
                break;
            }
            if (added <= 0) rc = DTREE_ERR_CUDA;  // no edge left to add: cannot happen with >= 2 components
            base += added;
        }
        if (rc == DTREE_OK && base != n - 1) rc = DTREE_ERR_CUDA;
        if (timed) cudaEventRecord(ev[1], s);
        if (st && cudaMemcpyAsync(hs, cstats, sizeof(hs), cudaMemcpyDeviceToHost, s) != cudaSuccess) rc = DTREE_ERR_CUDA;
    } while (false);
    cudaFreeAsync(m, s);
    if (cudaStreamSynchronize(s) != cudaSuccess && rc == DTREE_OK) rc = cuda_status(cudaGetLastError());
    if (st && rc == DTREE_OK) {
        st->point_pairs = (int64_t)hs[0];
        st->leaf_pairs_evaluated = (int64_t)hs[1];
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
