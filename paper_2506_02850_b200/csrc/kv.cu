// metok_kv_compact: per-layer keep lists (section 3.3 policy, top-k policy, or given)
// and the in-place, order-preserving gather of K and V rows.
//
// In-place safety.  Row i receives old row keep[i] with keep ascending, hence
// keep[i] >= i, and after the call only rows [0, n) matter (n = list length).
//
// Fast path.  A source row at or beyond n is never written by anybody, so it can be
// read at any time.  Only the first h rows of the list, h = #{i : keep[i] < n}, have
// their source inside the destination region.  Those h rows are read, into registers or a
// staging area in the workspace, by the CTAs of the slab's cluster before a cluster barrier behind
// which every row is written.  With a keep ratio r about r*n rows are concerned.
//
// General path (h larger than the staging area: lists that keep most rows).  Rows are
// moved in rounds of consecutive destination rows; a round's sources all lie at or
// beyond the round's first destination row, so
//   * a round only has to finish READING before any of its rows are WRITTEN, and
//   * later rounds' sources are never touched by earlier rounds' writes, so the
//     next round can be prefetched before the current one is stored.
// One thread-block cluster owns one (layer, K|V, head) slab; the read->write
// ordering inside a round is a hardware cluster barrier (no spinning on memory).
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "launchers.h"

namespace cg = cooperative_groups;

namespace metok {

constexpr int kKvCluster = 4;        // CTAs per slab
constexpr int kKvThreads = 256;
constexpr int kKvUnroll = 4;         // 16-byte chunks per thread per round
constexpr int kKvMaxLayersPerLaunch = 64;

struct KvPtrs {
    void* k[kKvMaxLayersPerLaunch];
    void* v[kKvMaxLayersPerLaunch];
};

// PAPER policy lists: layers below l1 keep everything, the others drop the visual span.
__global__ void __launch_bounds__(256)
kv_paper_lists_kernel(int S_cur, int vis_start, int n_vis, int l1, int32_t* __restrict__ keep_idx,
                      int32_t* __restrict__ keep_len, int32_t* __restrict__ new_len) {
    grid_dep_wait();
    const int layer = blockIdx.x;
    int32_t* keep = keep_idx + (size_t)layer * S_cur;
    int n;
    if (layer < l1) {
        for (int i = threadIdx.x; i < S_cur; i += blockDim.x) keep[i] = i;
        n = S_cur;
    } else {
        for (int i = threadIdx.x; i < vis_start; i += blockDim.x) keep[i] = i;
        const int tail = S_cur - (vis_start + n_vis);
        for (int i = threadIdx.x; i < tail; i += blockDim.x) keep[vis_start + i] = vis_start + n_vis + i;
        n = vis_start + tail;
    }
    if (threadIdx.x == 0) { keep_len[layer] = n; new_len[layer] = n; }
}

// PAPER policy when no more rows follow the visual span than it holds (the rule: a question is shorter than its video):
// every row that moves comes from beyond the new length, so one kernel writes the lists and moves the rows, a
// contiguous piece per slab.  (Three launches, the lists read back row by row: 12.3 us for 6272 + 80 rows in 28 layers;
// 4.2 now, one pass of a replayed graph.)  The CTAs of a layer's slabs share the writing of its list.
__global__ void __launch_bounds__(256)
kv_paper_kernel(KvPtrs ptrs, int layer0, int Hkv, int S_cap, int S_cur, int row_chunks, int vis_start, int n_vis, int l1,
                int32_t* __restrict__ keep_idx, int32_t* __restrict__ keep_len, int32_t* __restrict__ new_len,
                int32_t* __restrict__ status) {
    grid_dep_wait();
    const int slab = blockIdx.y, head = slab % Hkv, which = (slab / Hkv) & 1, ll = slab / (2 * Hkv), layer = layer0 + ll;
    const int tail = S_cur - (vis_start + n_vis), n = layer < l1 ? S_cur : vis_start + tail;
    if (layer >= l1) {
        uint4* base = reinterpret_cast<uint4*>(which ? ptrs.v[ll] : ptrs.k[ll]) + (size_t)head * S_cap * row_chunks;
        uint4* dst = base + (size_t)vis_start * row_chunks;
        const uint4* src = dst + (size_t)n_vis * row_chunks;
        const int total = n_vis > 0 ? tail * row_chunks : 0;
        constexpr int U = 4;
        for (int g0 = blockIdx.x * 256 * U + threadIdx.x; g0 < total; g0 += gridDim.x * 256 * U) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (g0 + u * 256 < total) v[u] = src[g0 + u * 256];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (g0 + u * 256 < total) dst[g0 + u * 256] = v[u];
        }
    }
    int32_t* keep = keep_idx + (size_t)layer * S_cur;
    const int part = (which * Hkv + head) * gridDim.x + blockIdx.x, parts = 2 * Hkv * gridDim.x;
    for (int i = part * 256 + threadIdx.x; i < n; i += parts * 256) keep[i] = layer < l1 || i < vis_start ? i : i + n_vis;
    if (part == 0 && threadIdx.x == 0) {
        keep_len[layer] = n;
        new_len[layer] = n;
        if (layer == 0) *status = METOK_OK;
    }
}

// GIVEN policy: the caller's lists are checked before anything is indexed through them.  One CTA
// per layer reads only the list itself: 0 <= length <= S_cur, entries strictly ascending inside
// [0, S_cur).  valid[layer] says whether the layer may be compacted; a layer with a bad list is
// left untouched and reports S_cur rows.
__global__ void __launch_bounds__(256)
kv_check_lists_kernel(int S_cur, const int32_t* __restrict__ keep_idx, const int32_t* __restrict__ keep_len,
                      int32_t* __restrict__ new_len, int32_t* __restrict__ valid) {
    grid_dep_wait();
    __shared__ int s_bad;
    const int layer = blockIdx.x;
    const int n = keep_len[layer];
    if (threadIdx.x == 0) s_bad = (n < 0 || n > S_cur) ? 1 : 0;
    __syncthreads();
    if (!s_bad) {
        const int32_t* keep = keep_idx + (size_t)layer * S_cur;
        int bad = 0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int v = keep[i];
            const int prev = i > 0 ? keep[i - 1] : -1;
            bad |= (v <= prev) | (v >= S_cur);           // prev >= -1, so v > prev also gives v >= 0
        }
        if (bad) s_bad = 1;                               // same value from every writer
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        valid[layer] = s_bad ? 0 : 1;
        new_len[layer] = s_bad ? S_cur : n;
    }
}

// ---- fast path ------------------------------------------------------------------
constexpr int kKvFastThreads = 256;
constexpr int kKvFastUnroll = 8;          // 16-byte chunks in flight per thread
constexpr int kKvCtasPerSm = 4;           // (64 registers)
constexpr int kKvMaxSplit = 8;            // most CTAs per slab, a cluster
constexpr size_t kKvStageBudget = (size_t)128 << 20;   // bytes of workspace the staging area may take

// First index of the ascending list keep[0..n) whose value is >= n; whole warp, 32-ary search.
__device__ __forceinline__ int warp_lower_bound(const int32_t* __restrict__ keep, int n, int lane) {
    int lo = 0, hi = n;                                   // answer in [lo, hi]
    while (hi > lo) {
        const int step = (hi - lo + 31) / 32;
        const int idx = lo + lane * step;
        const bool ge = idx < hi ? keep[idx] >= n : true;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, ge);
        const int f = bal ? __ffs(bal) - 1 : 32;          // first probe that is >= n; 32: none was
        const int new_hi = f < 32 ? min(hi, lo + f * step) : hi;   // keep[new_hi] >= n (or new_hi == hi)
        const int new_lo = f > 0 ? lo + (f - 1) * step + 1 : lo;   // the probe before it was < n
        hi = new_hi;
        lo = new_lo;
    }
    return lo;
}

struct SlabId { int ll, which, head; };
__device__ __forceinline__ SlabId slab_of(int slab, int Hkv) {
    SlabId s;
    s.head = slab % Hkv;
    s.which = (slab / Hkv) & 1;
    s.ll = slab / (2 * Hkv);
    return s;
}

// A cluster per slab moves the slab's rows; its CTAs take runs of 2048 pieces of 16 bytes in turn.  Rows whose
// source lies at or beyond the new length (all but the first h) are never written before they are read.  The others are
// read by everybody before anybody writes: those of a CTA's first run into registers, later ones into the staging area,
// which the same thread reads again; then a cluster barrier, behind which the first run's loads of all rows land.
// Records h per layer (-1: too many for the staging area, the general path takes the layer).
// What bounds it is HBM, with scattered rows of 256 bytes.  Staging and copying as two kernels, the copy with four CTAs
// per slab in one and a half waves, took (call, cold, us) for 28 layers x 4 heads of 18 432 + 64 rows, 6.5 / 15 / 30 / 50 %
// kept: 52.2 / 98.3 / 196.6 / 469.0, this 46.0 / 87.0 / 185.3 / 472.1; 40 layers x 40 heads of 2751 rows 108.5 and 85.0, one
// layer of one head of 63 606 rows 148.4 and 70.6.
__global__ void __launch_bounds__(kKvFastThreads, kKvCtasPerSm)
kv_move_kernel(KvPtrs ptrs, int layer0, int Hkv, int S_cap, int S_cur, int row_chunks,
               const int32_t* __restrict__ keep_idx, const int32_t* __restrict__ keep_len, int stage_rows,
               int32_t* __restrict__ haz, uint4* stage, const int32_t* __restrict__ valid,
               int n_layers, int32_t* __restrict__ status) {
    grid_dep_wait();
    __shared__ int s_h;
    const SlabId id = slab_of(blockIdx.y, Hkv);
    const int layer = layer0 + id.ll;
    const bool lead = blockIdx.x == 0 && id.which == 0 && id.head == 0 && threadIdx.x == 0;   // one thread per layer
    // the call's status word: a rejected list (GIVEN policy) is an invalid argument
    if (layer0 == 0 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        int st = METOK_OK;
        if (valid)
            for (int l = 0; l < n_layers; ++l)
                if (!valid[l]) st = METOK_ERR_INVALID_ARG;
        *status = st;
    }
    if (valid && !valid[layer]) {                          // nothing is indexed through a rejected list (uniform per cluster)
        if (lead) haz[layer] = -2;
        return;
    }
    const int32_t* keep = keep_idx + (size_t)layer * S_cur;
    const int n = keep_len[layer];
    if (n <= 0 || n >= S_cur) {                            // nothing to keep, or nothing dropped
        if (lead) haz[layer] = 0;
        return;
    }
    uint4* base = reinterpret_cast<uint4*>(id.which ? ptrs.v[id.ll] : ptrs.k[id.ll]) +
                  (size_t)id.head * S_cap * row_chunks;
    uint4* stg = stage + ((size_t)(layer * 2 + id.which) * Hkv + id.head) * (size_t)stage_rows * row_chunks;
    const int total = n * row_chunks;
    constexpr int kStep = kKvFastThreads * kKvFastUnroll;
    uint4 v[kKvFastUnroll];
    unsigned some = 0;                                     // which of them there are to store
    auto load = [&](int g0, int h) {
        some = 0;
#pragma unroll
        for (int u = 0; u < kKvFastUnroll; ++u) {
            const int gc = g0 + u * kKvFastThreads + threadIdx.x;
            if (gc < total) {
                const int i = gc / row_chunks, c = gc - i * row_chunks;
                const int src = keep[i];
                if (src != i) {
                    v[u] = i < h ? stg[gc] : base[(size_t)src * row_chunks + c];
                    some |= 1u << u;
                }
            }
        }
    };
    const int g_first = blockIdx.x * kStep, stride = gridDim.x * kStep;
    load(g_first, 0);                                      // all from their sources
    if (threadIdx.x < 32) {
        const int h = warp_lower_bound(keep, n, threadIdx.x);
        if (threadIdx.x == 0) s_h = h;
    }
    __syncthreads();
    const int h = s_h;
    if (lead) haz[layer] = h <= stage_rows ? h : -1;
    if (h > stage_rows) return;                            // uniform per cluster
    for (int gc = g_first + stride + (int)threadIdx.x, u = 0; gc < h * row_chunks;) {
        const int i = gc / row_chunks, c = gc - i * row_chunks, src = keep[i];
        if (src != i) stg[gc] = base[(size_t)src * row_chunks + c];
        if (++u < kKvFastUnroll) {
            gc += kKvFastThreads;
        } else {
            u = 0;
            gc += stride - (kKvFastUnroll - 1) * kKvFastThreads;
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int g0 = g_first;;) {
#pragma unroll
        for (int u = 0; u < kKvFastUnroll; ++u)
            if (some >> u & 1u) base[g0 + u * kKvFastThreads + threadIdx.x] = v[u];
        g0 += stride;
        if (g0 >= total) break;
        load(g0, h);
    }
}

// ---- general path -----------------------------------------------------------------
__global__ void __cluster_dims__(kKvCluster, 1, 1) __launch_bounds__(kKvThreads)
kv_gather_kernel(KvPtrs ptrs, int layer0, int Hkv, int S_cap, int S_cur, int row_chunks,
                 const int32_t* __restrict__ keep_idx, const int32_t* __restrict__ keep_len,
                 const int32_t* __restrict__ haz) {
    grid_dep_wait();
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int slab = blockIdx.x / kKvCluster;            // (layer_local, which, head)
    const int head = slab % Hkv;
    const int which = (slab / Hkv) & 1;
    const int ll = slab / (2 * Hkv);
    if (haz[layer0 + ll] != -1) return;                  // the fast path took this layer, or its list was rejected (uniform per cluster)
    uint4* base = reinterpret_cast<uint4*>(which ? ptrs.v[ll] : ptrs.k[ll]) + (size_t)head * S_cap * row_chunks;
    const int32_t* keep = keep_idx + (size_t)(layer0 + ll) * S_cur;
    const int n = keep_len[layer0 + ll];
    if (n >= S_cur) return;                              // nothing dropped: every row stays (uniform per cluster)
    const long long total = (long long)n * row_chunks;
    constexpr int kPerCta = kKvThreads * kKvUnroll;
    const long long per_round = (long long)kKvCluster * kPerCta;
    const int rounds = (int)((total + per_round - 1) / per_round);

    struct Buf {
        uint4 v[kKvUnroll];
        int row[kKvUnroll];      // -1: nothing to store
        int c[kKvUnroll];
    } b0, b1;

    auto issue = [&](int r, Buf& b) {
#pragma unroll
        for (int u = 0; u < kKvUnroll; ++u) {
            const long long gc = ((long long)r * kKvCluster + crank) * kPerCta + u * kKvThreads + threadIdx.x;
            b.row[u] = -1;
            if (gc < total) {
                const int i = (int)(gc / row_chunks);
                const int c = (int)(gc % row_chunks);
                const int src = keep[i];
                if (src != i) {
                    b.v[u] = base[(size_t)src * row_chunks + c];
                    b.row[u] = i;
                    b.c[u] = c;
                }
            }
        }
    };
    auto store = [&](const Buf& b) {
#pragma unroll
        for (int u = 0; u < kKvUnroll; ++u)
            if (b.row[u] >= 0) base[(size_t)b.row[u] * row_chunks + b.c[u]] = b.v[u];
    };
    if (rounds > 0) issue(0, b0);
    for (int r = 0; r < rounds; r += 2) {
        cluster.sync();                                  // every CTA has read round r
        if (r + 1 < rounds) issue(r + 1, b1);            // its sources lie beyond round r's rows
        store(b0);
        if (r + 1 < rounds) {
            cluster.sync();
            if (r + 2 < rounds) issue(r + 2, b0);
            store(b1);
        }
    }
}

struct KvWs {
    int32_t* status;          // device status word, first in the workspace
    int32_t* haz;
    int32_t* valid;           // GIVEN policy: per layer, whether the caller's list passed the check
    uint4* stage;
    int stage_rows;
};
static KvWs carve_kv(Carver& cv, int L, int Hkv, int S_cur, int row_chunks) {
    KvWs w;
    w.status = cv.take<int32_t>(64);
    w.haz = cv.take<int32_t>((size_t)L);
    w.valid = cv.take<int32_t>((size_t)L);
    const size_t per_row = (size_t)L * 2 * Hkv * row_chunks * sizeof(uint4);
    size_t rows = kKvStageBudget / per_row;
    if (rows > (size_t)S_cur) rows = (size_t)S_cur;
    w.stage_rows = (int)rows;
    w.stage = cv.take<uint4>((size_t)L * 2 * Hkv * rows * row_chunks);
    return w;
}

static KvPtrs kv_ptrs(void* const* k_layers, void* const* v_layers, int l0, int nl) {
    KvPtrs p;
    for (int l = 0; l < kKvMaxLayersPerLaunch; ++l) {
        p.k[l] = l < nl ? k_layers[l0 + l] : nullptr;
        p.v[l] = l < nl ? v_layers[l0 + l] : nullptr;
    }
    return p;
}

}  // namespace metok

using namespace metok;

extern "C" size_t metok_kv_compact_workspace_bytes(int dtype, int L, int Hkv, int S_cur, int dh, int policy,
                                                   int n_vis) {
    (void)policy; (void)n_vis;
    if (L < 1 || Hkv < 1 || S_cur < 1 || dh < 1) return 0;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    const int row_chunks = (int)((long long)dh * eb / 16);
    if (row_chunks < 1) return 0;
    Carver cv(nullptr);
    carve_kv(cv, L, Hkv, S_cur, row_chunks);
    return cv.total();
}

extern "C" int metok_kv_compact(void* const* k_layers, void* const* v_layers, int dtype, int L, int Hkv, int S_cap,
                                int S_cur, int dh, int policy, int l1, double keep_ratio, int vis_start, int n_vis,
                                const float* scores, int scores_per_layer, int32_t* keep_idx, int32_t* keep_len,
                                int32_t* new_len, void* ws, size_t ws_bytes, void* stream) {
    if (!k_layers || !v_layers || !keep_idx || !keep_len || !new_len) return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (L < 1 || Hkv < 1 || S_cap < 1 || S_cur < 1 || S_cur > S_cap || dh < 1) return METOK_ERR_INVALID_ARG;
    if (policy != METOK_KV_PAPER && policy != METOK_KV_TOPK && policy != METOK_KV_GIVEN) return METOK_ERR_INVALID_ARG;
    if (vis_start < 0 || n_vis < 0 || (long long)vis_start + n_vis > S_cur) return METOK_ERR_INVALID_ARG;
    if (policy == METOK_KV_PAPER && l1 < 0) return METOK_ERR_INVALID_ARG;
    if (policy == METOK_KV_TOPK && (!scores || !(keep_ratio >= 0.0 && keep_ratio <= 1.0) || n_vis < 1))
        return METOK_ERR_INVALID_ARG;
    for (int l = 0; l < L; ++l) {
        if (!k_layers[l] || !v_layers[l] || !aligned16(k_layers[l]) || !aligned16(v_layers[l]))
            return METOK_ERR_INVALID_ARG;
    }
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (((long long)dh * eb) % 16 != 0) return METOK_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < metok_kv_compact_workspace_bytes(dtype, L, Hkv, S_cur, dh, policy, n_vis) || !aligned16(ws))
        return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int row_chunks = (int)((long long)dh * eb / 16);
    Carver cv(ws);
    const KvWs w = carve_kv(cv, L, Hkv, S_cur, row_chunks);

    // an upper bound, known on the host, of the length of every list that drops anything
    // (-1: not known); lists that keep all rows cause no copying
    int kept_bound = -1;
    if (policy == METOK_KV_PAPER) {
        if (S_cur - (vis_start + n_vis) <= n_vis) {                // one kernel: nothing moves into a row that is still to be read
            for (int l0 = 0; l0 < L; l0 += kKvMaxLayersPerLaunch) {
                const int nl = (L - l0) < kKvMaxLayersPerLaunch ? (L - l0) : kKvMaxLayersPerLaunch;
                const KvPtrs ptrs = kv_ptrs(k_layers, v_layers, l0, nl);
                const int slabs = nl * 2 * Hkv;
                // a CTA per 1024 chunks of a slab, up to eight CTAs per SM
                const long long want = ((long long)(S_cur - vis_start - n_vis) * row_chunks + 1023) / 1024, room = 8 * kNumSMs / slabs;
                const int split = (int)(want < 1 || room < 1 ? 1 : want < room ? want : room);
                {
                    METOK_TIMED("kv_paper_kernel", st);
                    launch_chained(kv_paper_kernel, dim3(split, slabs), dim3(256), 0, st, ptrs, l0, Hkv, S_cap, S_cur, row_chunks,
                                   vis_start, n_vis, l1, keep_idx, keep_len, new_len, w.status);
                }
                METOK_LAUNCH_CHECK();
            }
            return METOK_OK;
        }
        kept_bound = S_cur - n_vis;
        {
            METOK_TIMED("kv_paper_lists_kernel", st);
            launch_chained(kv_paper_lists_kernel, dim3(L), dim3(256), 0, st, S_cur, vis_start, n_vis, l1, keep_idx, keep_len, new_len);
        }
        METOK_LAUNCH_CHECK();
    } else if (policy == METOK_KV_TOPK) {
        int32_t budget = ceilq(keep_ratio * (double)n_vis);
        if (budget > n_vis) budget = n_vis;
        // shared scores give the same list in every layer: select once, write it L times
        const int problems = scores_per_layer ? L : 1;
        const int rc = launch_class_topk(scores, scores_per_layer ? (size_t)n_vis : 0, nullptr, n_vis, 1, &budget,
                                         S_cur, vis_start, keep_idx, (size_t)S_cur, scores_per_layer ? 1 : L,
                                         keep_len, new_len, problems, st);
        if (rc != METOK_OK) return rc;
        kept_bound = budget + (S_cur - n_vis);
    } else {
        {
            METOK_TIMED("kv_check_lists_kernel", st);
            launch_chained(kv_check_lists_kernel, dim3(L), dim3(256), 0, st, S_cur, keep_idx, keep_len, new_len, w.valid);
        }
        METOK_LAUNCH_CHECK();
    }
    const int32_t* valid = policy == METOK_KV_GIVEN ? w.valid : nullptr;
    for (int l0 = 0; l0 < L; l0 += kKvMaxLayersPerLaunch) {
        const int nl = (L - l0) < kKvMaxLayersPerLaunch ? (L - l0) : kKvMaxLayersPerLaunch;
        const KvPtrs ptrs = kv_ptrs(k_layers, v_layers, l0, nl);
        const int slabs = nl * 2 * Hkv;
        // a cluster of as many CTAs per slab as keep all of them resident at once: two waves cost more than fewer loads in
        // flight (224 slabs with clusters of four: 58.4 us instead of 46.0), and clusters that are no power of two leave SMs
        // unused (192 slabs with clusters of three: 50.2 us instead of 44.6)
        int split = 1;
        while (2 * split <= kKvMaxSplit && 2 * split * slabs <= kNumSMs * kKvCtasPerSm) split *= 2;
        {
            METOK_TIMED("kv_move_kernel", st);
            launch_chained_clusters(split, kv_move_kernel, dim3(split, slabs), dim3(kKvFastThreads), 0, st,
                ptrs, l0, Hkv, S_cap, S_cur, row_chunks, keep_idx, keep_len, w.stage_rows, w.haz, w.stage, valid, L,
                w.status);
        }
        METOK_LAUNCH_CHECK();
        // h <= list length: when every list is known to fit the staging area, no layer takes the general path
        if (kept_bound < 0 || kept_bound > w.stage_rows) {
            {
                METOK_TIMED("kv_gather_kernel", st);
                launch_chained(kv_gather_kernel, dim3(slabs * kKvCluster), dim3(kKvThreads), 0, st, ptrs, l0, Hkv, S_cap, S_cur, row_chunks,
                                                                        keep_idx, keep_len, w.haz);
            }
            METOK_LAUNCH_CHECK();
        }
    }
    return METOK_OK;
}
