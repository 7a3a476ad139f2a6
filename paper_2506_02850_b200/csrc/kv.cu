// metok_kv_compact: per-layer keep lists (section 3.3 policy, top-k policy, or given)
// and the in-place, order-preserving gather of K and V rows.
//
// In-place safety.  Row i receives old row keep[i] with keep ascending, hence
// keep[i] >= i, and after the call only rows [0, n) matter (n = list length).
//
// Fast path.  A source row at or beyond n is never written by anybody, so it can be
// read at any time.  Only the first h rows of the list, h = #{i : keep[i] < n}, have
// their source inside the destination region.  Those h rows are read, into shared memory or a
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
#include "sm100.cuh"

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
constexpr int kKvMoveWarps = 16;          // most warps of a CTA (64 registers, two such CTAs per SM)
constexpr int kKvPieceBytes = 2048, kKvRing = 3;   // a warp's ring: pieces on their way
constexpr int kKvMaxSplit = 8;            // most CTAs per slab, a cluster
constexpr size_t kKvStageBudget = (size_t)128 << 20;   // bytes of workspace the staging area may take

// First index of [0, n) with f(index), which stays true from there on; n if there is none.  Whole warp, 32-ary search.
template <typename F>
__device__ __forceinline__ int warp_first(int n, int lane, F f) {
    int lo = 0;
    while (n > 0) {                                        // it lies in [lo, lo + n]
        const int step = (n + 31) >> 5, at = lane * step + step - 1;
        const uint32_t yes = __ballot_sync(0xFFFFFFFFu, at >= n ? true : f(lo + at));
        if (!yes) return lo + n;
        const int skip = (__ffs(yes) - 1) * step;
        lo += skip;
        n = min(step - 1, n - skip);
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

// A cluster per slab moves the slab's rows; the warps of its CTAs take pieces of up to kKvPieceBytes of consecutive destination rows in
// turn.  Rows at the front that stay where they are (keep[i] == i: the first p) are left alone.  Rows whose source lies at or
// beyond the new length (all from the h-th on) are never written before they are read.  The others are read by everybody before
// anybody writes: those of a warp's first pieces into its ring, later ones into the staging area, which the same warp reads
// again; then a cluster barrier, behind which a piece leaves by one bulk copy as soon as it has landed.
// Records h per layer (-1: too many for the staging area, the general path takes the layer, before anything is read).
// What bounds it is HBM, with scattered rows of 256 bytes.  Rows through registers, all CTAs of 256 threads resident to the end,
// were a tenth slower, and other streams' kernels waited for the whole of it: an attention or selection CTA wants most of an SM.
// The call, cold, with two kernels (stage, copy) / through registers / this, in us, 28 layers x 4 heads of 18 432 + 72 rows, 6.5 / 15 / 30 / 50 %
// kept: 48.4 / 94.8 / 193.9 / 463.7; 43.6 / 86.0 / 183.2 / 469.8; 39.1 / 82.0 / 176.4 / 466.0.  40 layers x 40 heads of 2751 rows, 10 %:
// 139.6; 117.5; 111.4.  One layer of one head of 63 614 rows: 69.8; 39.1; 26.8.  One 128-frame video with the call beside pruning
// levels 2 and 3: 264.6; 268.5; 255.  The first of them with rings of 2 x 2 / 6 x 1 / 3 x 4 KB (eight warps) / 3 x 8 KB (four): 38.7 / 46.1 /
// 41.5 / 40.2 against 36.6 warm.
__global__ void __launch_bounds__(kKvMoveWarps * 32, 2)
kv_move_kernel(KvPtrs ptrs, int layer0, int Hkv, int S_cap, int S_cur, int row_chunks,
               const int32_t* __restrict__ keep_idx, const int32_t* __restrict__ keep_len, int stage_rows,
               int32_t* __restrict__ haz, uint4* stage, const int32_t* __restrict__ valid,
               int n_layers, int32_t* __restrict__ status) {
    grid_dep_wait();
    extern __shared__ uint8_t kv_dyn[];
    const SlabId id = slab_of(blockIdx.y, Hkv);
    const int layer = layer0 + id.ll, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool lead = id.which == 0 && id.head == 0 && blockIdx.x == 0 && threadIdx.x == 0;
    // the call's status: METOK_OK, or INVALID_ARG if any caller-given list failed its check
    if (layer0 == 0 && blockIdx.y == 0 && blockIdx.x == 0 && threadIdx.x == 0) {
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
    const uint32_t ring = ((sm100::smem_u32(kv_dyn) + 127u) & ~127u) + (uint32_t)(warp * kKvRing * kKvPieceBytes);
    // pieces: `rows` whole rows, or one of the `segs` parts of a row that is wider
    constexpr int kPiece = kKvPieceBytes / 16;
    const int rows = max(1, kPiece / row_chunks), segs = (row_chunks + kPiece - 1) / kPiece;
    int p = 0;                                             // rows that stay
    {
        const bool too_many = stage_rows < n && keep[stage_rows] < n;   // h > stage_rows: uniform per cluster
        const uint32_t stay = __ballot_sync(0xFFFFFFFFu, lane < n && keep[lane] == lane);
        if (too_many) {
            if (lead) haz[layer] = -1;
            return;
        }
        p = stay == 0xFFFFFFFFu ? warp_first(n, lane, [&](int i) { return keep[i] > i; }) : __ffs(~stay) - 1;
    }
    const int pieces = ((n - p) + rows - 1) / rows * segs;
    const int warps = blockDim.x >> 5, first = blockIdx.x * warps + warp, stride = gridDim.x * warps;
    struct Piece { int row0, nrows, c0, nc; };
    auto piece = [&](int q) {
        Piece x;
        const int g = q / segs, sg = q - g * segs;
        x.row0 = p + g * rows;
        x.nrows = min(rows, n - x.row0);
        x.c0 = sg * kPiece;
        x.nc = min(kPiece, row_chunks - x.c0);             // (all chunks where a piece is whole rows)
        return x;
    };
    // the sources of a piece's first 32 rows, one per lane
    auto sources = [&](int q) {
        if (q >= pieces) return 0;
        const int i = p + q / segs * rows + lane;
        return i < n ? keep[i] : 0;
    };
    auto load = [&](int q, int src, int slot, int h) {
        if (q < pieces) {
            const Piece x = piece(q);
            const uint32_t dst = ring + (uint32_t)(slot * kKvPieceBytes + lane * 16);
            int r = lane / x.nc, c = lane - r * x.nc;
            const int dr = 32 / x.nc, dc = 32 - dr * x.nc, total = x.nrows * x.nc;
#pragma unroll 4
            for (int t = 0; t < total; t += 32) {
                int from = __shfl_sync(0xFFFFFFFFu, src, r & 31);
                if (t + lane < total) {
                    const int i = x.row0 + r;
                    if (r >= 32) from = keep[i];
                    const uint4* at = i < h ? stg + (size_t)i * row_chunks : base + (size_t)from * row_chunks;
                    sm100::cp_async16_zfill(dst + (uint32_t)t * 16u, at + x.c0 + c, 16u);
                }
                r += dr;
                c += dc;
                if (c >= x.nc) { c -= x.nc; ++r; }
            }
        }
        sm100::cp_async_commit();
    };
#pragma unroll 1
    for (int k = 0; k < kKvRing; ++k) load(first + k * stride, sources(first + k * stride), k, 0);   // all from their sources
    int ahead = sources(first + kKvRing * stride);
    const int h = warp_first(n, lane, [&](int i) { return keep[i] >= n; });
    if (lead) haz[layer] = h;
    if (h > p) {
#pragma unroll 1
        for (int q = first + kKvRing * stride; q < pieces; q += stride) {
            const Piece x = piece(q);
            if (x.row0 >= h) break;
            for (int t = lane; t < x.nrows * x.nc; t += 32) {
                const int i = x.row0 + t / x.nc, c = x.c0 + t % x.nc;
                if (i < h) stg[(size_t)i * row_chunks + c] = base[(size_t)keep[i] * row_chunks + c];
            }
        }
        sm100::cp_async_wait_all();
        __syncwarp();
    }
    if (gridDim.x > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
    int slot = 0;
#pragma unroll 1
    for (int q = first; q < pieces; q += stride) {
        sm100::cp_async_wait<kKvRing - 2>();               // this piece has landed: kKvRing - 2 were asked for after it, and one more at first
        sm100::fence_proxy_async();
        __syncwarp();
        const Piece x = piece(q);
        if (lane == 0) {
            sm100::bulk_store(base + (size_t)x.row0 * row_chunks + x.c0, ring + (uint32_t)slot * kKvPieceBytes, (uint32_t)(x.nrows * x.nc) * 16u);
            sm100::bulk_commit();
            sm100::bulk_wait_read<1>();                    // the piece before has left its slot
        }
        __syncwarp();
        if (q != first) {
            const int next = q + (kKvRing - 1) * stride;
            const int src = ahead;
            ahead = sources(next + stride);
            load(next, src, slot == 0 ? kKvRing - 1 : slot - 1, h);
        }
        slot = slot + 1 == kKvRing ? 0 : slot + 1;
    }
    if (lane == 0) sm100::bulk_wait_all();
    sm100::cp_async_wait_all();
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
        // a cluster of as many CTAs per slab as keep all of them resident at once (clusters that are no power of two leave SMs
        // unused); where there are more slabs than places, smaller CTAs and more of them, so that one's reads run beside
        // another's writes (3200 slabs of 311 rows: 125 us with 16 warps, 111 with four)
        int split = 1;
        while (2 * split <= kKvMaxSplit && 2 * split * slabs <= 2 * kNumSMs) split *= 2;
        const int warps = slabs <= 2 * kNumSMs ? kKvMoveWarps : slabs <= 4 * kNumSMs ? kKvMoveWarps / 2 : kKvMoveWarps / 4;
        const size_t smem = (size_t)warps * kKvPieceBytes * kKvRing + 128;
        METOK_ALLOW_SMEM(kv_move_kernel, smem);
        {
            METOK_TIMED("kv_move_kernel", st);
            launch_chained_clusters(split, kv_move_kernel, dim3(split, slabs), dim3(warps * 32), smem, st,
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
