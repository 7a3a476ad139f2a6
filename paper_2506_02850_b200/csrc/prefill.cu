// metok_prefill_prune: text->visual attention scores at a pruning layer, class-wise
// top-k under the Eq. 6/7 budgets, and compaction of the surviving hidden states.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "select.cuh"
#include "select_cluster.cuh"
#include "launchers.h"
#include "simt_tile.cuh"
#include "sm100.cuh"

namespace metok {

// --------------------------------------------------------------------------- //
// Attention scores, generic CUDA-core path.
//
// Per KV head g the rep = Hq/Hkv query heads of the group form R = rep*Lt rows
// (row r = local head * Lt + q) that all multiply the same K[g].  The softmax
// normaliser of a row needs every visible key, the column sums need the
// normaliser, and the R x S probability matrix is never stored: pass 1 computes
// per-row running (max, sum) over a split of the columns, pass 2 recomputes the
// logits, normalises, and sums each column over the rows of the tile.
// Everything is reduced in a fixed order (no float atomics).
//
// A CTA of 64 threads takes a tile of 32 rows and a run of tiles of 32 keys (SimtTile with 4 x 4 outputs per thread); a
// thread keeps the running (max, sum) of its four rows over its own keys and they meet once, at the end of the run.  What
// bounds it is the rate of multiply-adds and shared-memory reads together, at small sizes the chain over the head
// dimension.  Tiles of 64 x 64 read less but fill the chip worse (28 heads x 30 rows x 6080 keys, fp32, the whole pruning
// call: 222 us with 64 x 64 tiles of 4 x 4 scalar reads per thread and 256 threads, 133 with SimtTile<8>, 126 as it is;
// 40 heads x 16 rows x 3016 keys: 265, 166, 100; 14 heads x 7 rows x 2041 keys: 30.8, 33.5, 27); of 16 x 16 only
// where a KV head has 16 rows or fewer (92 for the second case).
// --------------------------------------------------------------------------- //
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kNegInf = -3.0e38f;   // finite stand-in: keeps (m_old - m_new) free of inf - inf
constexpr int kAtPT = 4, kAtTile = 8 * kAtPT;   // outputs per thread and tile (a side of the square)
constexpr int kAtMaxSplits = 128;

struct AttnDims {
    int Hq, Hkv, Lt, S, dh, vis_start, n_vis, rep, R, nrt, nsplit, per, tiles_n;   // nsplit runs of `per` key tiles
    float scale_log2;
};

// This thread's copies of a tile's query rows (they stay the same) and of the key rows from u0 on; rows past the end are
// copies of the last one, whose results nobody uses.
template <typename Tile, typename T>
__device__ __forceinline__ void attn_tile_sources(const T* Qg, const T* Kg, const AttnDims& dm, int rt, int u0, bool first,
                                                  const uint4* (&src)[Tile::kCopies]) {
    const size_t row_chunks = (size_t)(dm.dh / Tile::CE);
#pragma unroll
    for (int i = 0; i < Tile::kCopies; ++i) {
        const int r = Tile::copy_row(i);
        if (r >= kAtTile)
            src[i] = reinterpret_cast<const uint4*>(Kg) + (size_t)min(u0 + r - kAtTile, dm.S - 1) * row_chunks + Tile::copy_chunk();
        else if (first)
            src[i] = reinterpret_cast<const uint4*>(Qg) + (size_t)min(rt * kAtTile + r, dm.R - 1) * row_chunks + Tile::copy_chunk();
    }
}

template <typename T>
__global__ void __launch_bounds__(kSaThreads, sizeof(T) == 4 ? sa_ctas_per_sm(kAtPT) : 4)
attn_stats_kernel(const T* __restrict__ q_text, const T* __restrict__ k_all, AttnDims dm,
                  float* __restrict__ part_m, float* __restrict__ part_l, int32_t* __restrict__ status) {
    grid_dep_wait();
    using Tile = SimtTile<T, kAtPT>;
    constexpr int PT = kAtPT;
    __shared__ __align__(16) Tile tile;
    const int split = blockIdx.x, rt = blockIdx.y, g = blockIdx.z;
    if (status && split == 0 && rt == 0 && g == 0 && threadIdx.x == 0) {     // as in attn_stats_mma_kernel
        *status = 0;
        status[kStatusCounts] = status[kStatusCounts + 1] = 0;
    }
    const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7;
    const T* Qg = q_text + (size_t)g * dm.R * dm.dh;
    const T* Kg = k_all + (size_t)g * dm.S * dm.dh;
    const int text_start = dm.S - dm.Lt;
    int limit[PT];
    float m_run[PT], l_run[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int r = rt * kAtTile + ty + 8 * i;
        limit[i] = r < dm.R ? text_start + (r % dm.Lt) : -1;    // last visible key
        m_run[i] = kNegInf;
        l_run[i] = 0.f;
    }
    const int t_lo = split * dm.per, t_hi = min(dm.tiles_n, t_lo + dm.per);
    const int ksteps = Tile::steps(dm.dh);
    const uint32_t dst0 = tile.copy_dst();
    const uint4* src[Tile::kCopies];
    for (int tn = t_lo; tn < t_hi; ++tn) {
        const int u0 = tn * kAtTile;
        attn_tile_sources<Tile>(Qg, Kg, dm, rt, u0, tn == t_lo, src);
        __syncthreads();
        float acc[PT][PT];
        tile.dots(src, dm.dh / Tile::CE, ksteps, dst0, acc);
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            float m_new = m_run[i];
#pragma unroll
            for (int j = 0; j < PT; ++j) {
                acc[i][j] = (u0 + tx + 8 * j <= limit[i]) ? acc[i][j] * dm.scale_log2 : kNegInf;
                m_new = fmaxf(m_new, acc[i][j]);
            }
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < PT; ++j) s += (acc[i][j] > kNegInf) ? exp2f(acc[i][j] - m_new) : 0.f;
            l_run[i] = l_run[i] * exp2f(m_run[i] - m_new) + s;
            m_run[i] = m_new;
        }
    }
#pragma unroll
    for (int i = 0; i < PT; ++i) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {                       // the eight threads of the row
            const float m2 = __shfl_xor_sync(0xFFFFFFFFu, m_run[i], o), l2 = __shfl_xor_sync(0xFFFFFFFFu, l_run[i], o);
            const float m = fmaxf(m_run[i], m2);
            l_run[i] = l_run[i] * exp2f(m_run[i] - m) + l2 * exp2f(m2 - m);
            m_run[i] = m;
        }
        const int r = rt * kAtTile + ty + 8 * i;
        if (tx == 0 && r < dm.R) {
            const size_t o = ((size_t)g * dm.nsplit + split) * dm.R + r;
            part_m[o] = m_run[i];
            part_l[o] = l_run[i];
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kSaThreads, sizeof(T) == 4 ? sa_ctas_per_sm(kAtPT) : 4)
attn_colsum_kernel(const T* __restrict__ q_text, const T* __restrict__ k_all, AttnDims dm,
                   const float* __restrict__ part_m, const float* __restrict__ part_l,
                   float* __restrict__ part_col) {
    grid_dep_wait();
    using Tile = SimtTile<T, kAtPT>;
    constexpr int PT = kAtPT;
    __shared__ __align__(16) Tile tile;
    __shared__ float s_M[kAtTile], s_invZ[kAtTile];
    __shared__ float s_col[2][kAtTile];
    const int split = blockIdx.x, rt = blockIdx.y, g = blockIdx.z;
    const int tid = threadIdx.x, ty = tid >> 3, tx = tid & 7, warp = tid >> 5, lane = tid & 31;
    const T* Qg = q_text + (size_t)g * dm.R * dm.dh;
    const T* Kg = k_all + (size_t)g * dm.S * dm.dh;
    const int text_start = dm.S - dm.Lt, vis_end = dm.vis_start + dm.n_vis;
    const int t_lo = max(split * dm.per, dm.vis_start / kAtTile);                                    // tiles with a visual column
    const int t_hi = min(min(dm.tiles_n, split * dm.per + dm.per), (vis_end + kAtTile - 1) / kAtTile);
    if (t_lo >= t_hi) return;
    {
        // The rows' normalisers, two threads per row (its even and its odd runs of keys): every CTA goes through all runs' partials,
        // up to 128 per row, in round trips to L2 of sixteen runs per thread.  (A thread per row, eight runs a trip: 14 heads
        // x 7 rows x 2041 keys in 64 runs, this kernel 15.3 us under ncu, 11.6 now; the call 28.4 -> 24.1.)  Up to eight
        // runs are four per thread, without the instructions for twelve that are not there: 14 heads x 8 rows x 64 keys, the call
        // 10.1 -> 9.4 us, 40 heads x 30 rows x 150 keys 15.7 -> 14.9.
        static_assert(kSaThreads == 2 * kAtTile, "two threads per row");
        const int rl = tid >> 1, odd = tid & 1, r = rt * kAtTile + rl;
        const int runs = r < dm.R ? dm.nsplit : 0;
        const size_t o = (size_t)g * dm.nsplit * dm.R + r;
        float M = kNegInf, Z = 0.f;
        auto add = [&](auto trip) {
            constexpr int kTrip = decltype(trip)::value;
            for (int s0 = odd; s0 < runs; s0 += 2 * kTrip) {
                float m[kTrip], l[kTrip], Mn = M;
#pragma unroll
                for (int x = 0; x < kTrip; ++x) {
                    const bool in = s0 + 2 * x < runs;
                    m[x] = in ? part_m[o + (size_t)(s0 + 2 * x) * dm.R] : kNegInf;
                    l[x] = in ? part_l[o + (size_t)(s0 + 2 * x) * dm.R] : 0.f;
                }
#pragma unroll
                for (int x = 0; x < kTrip; ++x) Mn = fmaxf(Mn, m[x]);
                Z *= exp2f(M - Mn);
#pragma unroll
                for (int x = 0; x < kTrip; ++x) Z += l[x] * exp2f(m[x] - Mn);
                M = Mn;
            }
        };
        if (dm.nsplit <= 8) add(std::integral_constant<int, 4>());
        else add(std::integral_constant<int, 16>());
        const float Mo = __shfl_xor_sync(0xFFFFFFFFu, M, 1), Zo = __shfl_xor_sync(0xFFFFFFFFu, Z, 1), Mn = fmaxf(M, Mo);
        Z = Z * exp2f(M - Mn) + Zo * exp2f(Mo - Mn);             // read from the even thread
        if (!odd) {
            s_M[rl] = Mn;
            s_invZ[rl] = Z > 0.f ? 1.0f / Z : 0.f;
        }
    }
    __syncthreads();
    int limit[PT];
    float rM[PT], rI[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int rl = ty + 8 * i;
        const int r = rt * kAtTile + rl;
        limit[i] = r < dm.R ? text_start + (r % dm.Lt) : -1;
        rM[i] = s_M[rl];
        rI[i] = s_invZ[rl];
    }
    const int ksteps = Tile::steps(dm.dh);
    const uint32_t dst0 = tile.copy_dst();
    const uint4* src[Tile::kCopies];
    for (int tn = t_lo; tn < t_hi; ++tn) {
        const int u0 = tn * kAtTile;
        attn_tile_sources<Tile>(Qg, Kg, dm, rt, u0, tn == t_lo, src);
        float acc[PT][PT];
        tile.dots(src, dm.dh / Tile::CE, ksteps, dst0, acc);      // (the barrier below: nobody reads the tile before)
#pragma unroll
        for (int j = 0; j < PT; ++j) {
            const int u = u0 + tx + 8 * j;
            float c = 0.f;
#pragma unroll
            for (int i = 0; i < PT; ++i)
                c += (u <= limit[i]) ? exp2f(acc[i][j] * dm.scale_log2 - rM[i]) * rI[i] : 0.f;
            c += __shfl_xor_sync(0xFFFFFFFFu, c, 8);             // the warp's four row groups
            c += __shfl_xor_sync(0xFFFFFFFFu, c, 16);
            if (lane < 8) s_col[warp][tx + 8 * j] = c;
        }
        __syncthreads();
        if (tid < kAtTile) {
            const int u = u0 + tid;
            if (u >= dm.vis_start && u < vis_end)
                part_col[((size_t)g * dm.nrt + rt) * dm.n_vis + (u - dm.vis_start)] = s_col[0][tid] + s_col[1][tid];
        }
    }
}

// scores[j] = inv_rows * (sum of the planes, in their order), for one level or for all levels of a schedule.  With several,
// the blocks of the first also write origin[j] = j and count the tokens of classes 0 and 1.  (The kernel is so short that what
// one level does not need is left out at compile time: 2.8 us with one, 3.6 with the levels looked up.)
struct ReduceLevel { const float* part_col; float* scores; int n_vis, block0; };   // block0: the level's first block
template <int NL>
struct ReduceArgs {
    ReduceLevel lv[NL];
    int nparts;
    float inv_rows;
    const int32_t* group;                                     // several levels, else null
    int32_t *origin, *counts;
};
template <int NL>
__global__ void __launch_bounds__(256)
attn_score_reduce_kernel(const __grid_constant__ ReduceArgs<NL> ra) {
    grid_dep_wait();
    int level = 0;
#pragma unroll
    for (int l = 1; l < NL; ++l) level += (int)blockIdx.x >= ra.lv[l].block0;
    const float* __restrict__ part_col = ra.lv[level].part_col;
    const int n_vis = ra.lv[level].n_vis, nparts = ra.nparts;
    const int j = ((int)blockIdx.x - (NL > 1 ? ra.lv[level].block0 : 0)) * 256 + (int)threadIdx.x;
    if (NL > 1 && level == 0) {
        const int g = j < n_vis ? ra.group[j] : -1;
        const int c0 = __syncthreads_count(g == 0), c1 = __syncthreads_count(g == 1);
        if (threadIdx.x < 2) atomicAdd(&ra.counts[threadIdx.x], threadIdx.x == 0 ? c0 : c1);
        if (j < n_vis) ra.origin[j] = j;
    }
    if (j >= n_vis) return;
    float a = 0.f;
    int p = 0;
    for (; p + 8 <= nparts; p += 8) {                          // eight loads in flight, added in plane order
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = part_col[(size_t)(p + u) * n_vis + j];
#pragma unroll
        for (int u = 0; u < 8; ++u) a += v[u];
    }
    for (; p < nparts; ++p) a += part_col[(size_t)p * n_vis + j];
    ra.lv[level].scores[j] = a * ra.inv_rows;
}

// --------------------------------------------------------------------------- //
// Class-wise top-k + ordered keep list.  One CTA per problem (blockIdx.x): the
// prefill step launches one, the KV TOPK policy one per layer.
// --------------------------------------------------------------------------- //
struct TopkBudgets { int v[METOK_MAX_GROUPS]; };

__global__ void __cluster_dims__(kSelCluster, 1, 1) __launch_bounds__(kSelThreads)
class_topk_kernel(const float* __restrict__ scores, size_t score_stride, const int32_t* __restrict__ token_group,
                  int n_vis, int G, SelectLayout lay, TopkBudgets budgets, int S, int vis_start,
                  int32_t* __restrict__ keep_idx, size_t keep_stride, int replicas,
                  int32_t* __restrict__ count_a, int32_t* __restrict__ count_b) {
    grid_dep_wait();
    __shared__ SelectSmem sm;
    __shared__ int s_budget[METOK_MAX_GROUPS];
    extern __shared__ __align__(16) unsigned char sel_dyn[];
    const int problem = blockIdx.x / kSelCluster;
    const float* sc = scores + (size_t)problem * score_stride;
    int32_t* keep = keep_idx + (size_t)problem * keep_stride;
    const int vis_end = vis_start + n_vis;
    SelectCtx cx;
    cx.rank = (int)cx.cl.block_rank();
    cx.G = G;
    cx.nb_log2 = lay.nb_log2;
    int p_lo, p_hi;
    select_slice(S, cx.rank, &p_lo, &p_hi);
    const int v_lo = max(p_lo, vis_start), v_hi = min(p_hi, vis_end);   // scored positions of this slice
    cx.item_lo = v_lo - vis_start;
    cx.m = v_hi > v_lo ? v_hi - v_lo : 0;
    cx.cached = cx.m <= lay.cache_cap;
    cx.hist = reinterpret_cast<uint32_t*>(sel_dyn + lay.hist_off);
    cx.merged = reinterpret_cast<uint32_t*>(sel_dyn + lay.merged_off);
    cx.keys = reinterpret_cast<uint32_t*>(sel_dyn + lay.keys_off);
    cx.cls = sel_dyn + lay.cls_off;
    for (int g = threadIdx.x; g < G; g += blockDim.x) s_budget[g] = budgets.v[g];
    __syncthreads();
    auto cls = [=](int i) {
        if (!token_group) return 0;
        const int g = token_group[i];
        return (g >= 0 && g < G) ? g : -1;
    };
    auto val = [=](int i) { return sc[i]; };
    cluster_select(cx, n_vis, cls, val, s_budget, sm);
    auto flag = [&](int u) {
        if (u < vis_start || u >= vis_end) return true;
        const int i = u - vis_start;
        const SelItem it = item_at(cx, i - cx.item_lo, cls, val);
        return it.cls >= 0 && is_selected(sm, it.cls, it.key, i);
    };
    // one list may serve several layers: `replicas` copies, keep_stride apart
    auto emit = [&](int u, int rank) {
        for (int r = 0; r < replicas; ++r) keep[(size_t)r * keep_stride + rank] = u;
    };
    const int total = cluster_compact(cx, p_lo, p_hi, flag, emit, [](int, int) {}, sm);
    if (cx.rank == 0) {
        for (int r = threadIdx.x; r < replicas; r += blockDim.x) {
            if (count_a) count_a[problem + r] = total;
            if (count_b) count_b[problem + r] = total;
        }
    }
}

// Where the selection adds the planes itself, a launch less: few planes, of which four are in flight (40 of 200 tokens: 18.1
// us the call with the sum apart, 19.5 inside), and little to read per CTA (bytes).  14 heads in two planes, 6272 tokens:
// 23.3 -> 22.3 us replayed; 28 in eight, 800 tokens: 21.7 -> 21.5, 8000: 32.5 -> 32.2, 18 432: the same, and left apart.
constexpr int kPlanesInside = 8, kPlaneBytesInside = 64 * 1024;
// The scores of one level as the attention passes leave them: n planes to be added in their order (n 0: they are added already).
struct ScorePlanes { const float* part_col; int n; float inv_rows; float* scores; };
// This thread's items i_first + 32 j < i_hi of the n_vis: their planes added and the scores written.
template <int IT>
__device__ __forceinline__ void add_planes(const ScorePlanes& pl, int n_vis, int i_first, int i_hi, float (&v)[IT]) {
#pragma unroll
    for (int j = 0; j < IT; ++j) v[j] = 0.f;
    constexpr int U = 4;                                      // planes whose loads are in flight
    for (int p0 = 0; p0 < pl.n; p0 += U) {
        float x[U][IT];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < IT; ++j)
                x[u][j] = p0 + u < pl.n && i_first + 32 * j < i_hi ? pl.part_col[(size_t)(p0 + u) * n_vis + i_first + 32 * j] : 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < IT; ++j)
                if (p0 + u < pl.n) v[j] += x[u][j];
    }
#pragma unroll
    for (int j = 0; j < IT; ++j) {
        v[j] *= pl.inv_rows;
        if (i_first + 32 * j < i_hi) pl.scores[i_first + 32 * j] = v[j];
    }
}

// The same for up to 81 920 items (select_cluster.cuh): a CTA or a cluster per problem.
template <int IT, bool kCl, bool kOne, bool kPlanes>   // kOne: one class and no class array; kPlanes: the scores are still in planes
__global__ void __launch_bounds__(IT == kCsMaxItems ? kCsMaxItemsThreads : 1024)
cs_topk_kernel(const float* __restrict__ scores, size_t score_stride, const int32_t* __restrict__ token_group,
               int n_vis, int G, CsLayout lay, TopkBudgets budgets, int S, int vis_start,
               int32_t* __restrict__ keep_idx, size_t keep_stride, int replicas,
               int32_t* __restrict__ count_a, int32_t* __restrict__ count_b, ScorePlanes pl) {
    cs_enter<kCl>();
    grid_dep_wait();
    __shared__ CsShared sm;
    extern __shared__ __align__(16) unsigned char sel_dyn[];
    constexpr int C = kCl ? kCsMaxCluster : 1;
    const int problem = blockIdx.x / C, rank = blockIdx.x - problem * C;
    const float* sc = scores + (size_t)problem * score_stride;
    int32_t* keep = keep_idx + (size_t)problem * keep_stride;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const CsSlice sl = cs_slice<IT>(n_vis, rank, C);
    float added[kPlanes ? IT : 1] = {};
    if constexpr (kPlanes) add_planes<IT>(pl, n_vis, sl.i_first, sl.i_hi, added);
    auto load = [&](int j, int i, float& v, int& c) {
        v = kPlanes ? added[j] : sc[i];
        c = 0;
        if (!kOne) {
            c = token_group[i];
            if (c >= G) c = -1;
        }
    };
    int before, kept;
    const uint32_t bits = cs_select<IT, kCl, kOne>(sm, sel_dyn, lay, G, budgets.v, rank, sl.i_first, sl.i_hi, load, &before, &kept);
    // The kept positions in order; positions before and after the visual span are always kept.
    const int outside = S - n_vis;
    if (replicas == 1) {
        cs_for_items<IT>(bits, vis_start + before, sl.i_first, sl.i_hi, [&](int, int i, int place, bool k) {
            if (k) keep[place] = vis_start + i;
        });
        for (int i = rank * nthr + tid; i < outside; i += C * nthr)
            keep[i < vis_start ? i : kept + i] = i < vis_start ? i : i + n_vis;
    } else {
        // One list serves several layers (`replicas` copies, keep_stride apart): the CTA's part of it is packed in
        // shared memory (over the histograms, as much as they hold at a time), so that every copy leaves in
        // coalesced stores.
        int32_t* pack = reinterpret_cast<int32_t*>(sel_dyn);
        const int room = 2 * G << lay.nb_log2;
        int mine = 0;                                        // what this CTA keeps, and the place of its first item
        for (int w = 0; w < (nthr >> 5); ++w) mine += sm.warp_tot[w];
        const int first = sm.before;
        for (int p0 = 0; p0 < mine; p0 += room) {
            cs_for_items<IT>(bits, before - first - p0, sl.i_first, sl.i_hi, [&](int, int i, int place, bool k) {
                if (k && place >= 0 && place < room) pack[place] = vis_start + i;
            });
            __syncthreads();
            for (int i = tid; i < min(room, mine - p0); i += nthr) {
                const int v = pack[i];
                for (int l = 0; l < replicas; ++l) keep[(size_t)l * keep_stride + vis_start + first + p0 + i] = v;
            }
            __syncthreads();
        }
        for (int i = rank * nthr + tid; i < outside; i += C * nthr)
            for (int l = 0; l < replicas; ++l)
                keep[(size_t)l * keep_stride + (i < vis_start ? i : kept + i)] = i < vis_start ? i : i + n_vis;
    }
    if (rank == 0) {
        for (int l = tid; l < replicas; l += nthr) {
            if (count_a) count_a[problem + l] = outside + kept;
            if (count_b) count_b[problem + l] = outside + kept;
        }
    }
}

static int class_topk(const float* scores, size_t score_stride, const int32_t* token_group, int n_vis, int G,
                      const int32_t* budgets_host, int S, int vis_start, int32_t* keep_idx, size_t keep_stride,
                      int replicas, int32_t* count_a, int32_t* count_b, int problems, const ScorePlanes& pl, cudaStream_t st);
int launch_class_topk(const float* scores, size_t score_stride, const int32_t* token_group, int n_vis, int G,
                      const int32_t* budgets_host, int S, int vis_start, int32_t* keep_idx, size_t keep_stride,
                      int replicas, int32_t* count_a, int32_t* count_b, int problems, cudaStream_t st) {
    return class_topk(scores, score_stride, token_group, n_vis, G, budgets_host, S, vis_start, keep_idx, keep_stride, replicas, count_a,
                      count_b, problems, {}, st);
}
static int class_topk(const float* scores, size_t score_stride, const int32_t* token_group, int n_vis, int G,
                      const int32_t* budgets_host, int S, int vis_start, int32_t* keep_idx, size_t keep_stride,
                      int replicas, int32_t* count_a, int32_t* count_b, int problems, const ScorePlanes& pl, cudaStream_t st) {
    TopkBudgets b;
    for (int g = 0; g < METOK_MAX_GROUPS; ++g) b.v[g] = g < G ? budgets_host[g] : 0;
    const CsPlan plan = cs_plan(n_vis);
    if (plan.fits) {
        const CsLayout lay = cs_layout(G, n_vis);
        auto launch = [&](auto kernel) -> int {
            if (lay.bytes > 40 * 1024) METOK_ALLOW_SMEM(kernel, lay.bytes);
            METOK_TIMED("class_topk_kernel", st);
            launch_chained_clusters(plan.C, kernel, dim3(problems * plan.C), dim3(plan.threads), lay.bytes, st, scores,
                                    score_stride, token_group, n_vis, G, lay, b, S, vis_start, keep_idx, keep_stride,
                                    replicas, count_a, count_b, pl);
            METOK_LAUNCH_CHECK();
            return METOK_OK;
        };
        const bool one = G == 1 && !token_group;
        if (pl.n > 0) return plan.C == 1 ? launch(cs_topk_kernel<4, false, false, true>) : launch(cs_topk_kernel<4, true, false, true>);
        if (plan.C == 1)
            return one ? launch(cs_topk_kernel<4, false, true, false>) : launch(cs_topk_kernel<4, false, false, false>);
        if (plan.items == 4)
            return one ? launch(cs_topk_kernel<4, true, true, false>) : launch(cs_topk_kernel<4, true, false, false>);
        return one ? launch(cs_topk_kernel<kCsMaxItems, true, true, false>) : launch(cs_topk_kernel<kCsMaxItems, true, false, false>);
    }
    const SelectLayout lay = select_layout(G, select_items_per_cta((long long)S));
    const int nthreads = select_threads(select_items_per_cta((long long)S));
    if (lay.bytes > 32 * 1024)                        // static + dynamic beyond 48 KiB needs the opt-in
        METOK_ALLOW_SMEM(class_topk_kernel, lay.bytes);
    {
        METOK_TIMED("class_topk_kernel", st);
        launch_chained(class_topk_kernel, dim3(problems * kSelCluster), dim3(nthreads), lay.bytes, st,
            scores, score_stride, token_group, n_vis, G, lay, b, S, vis_start, keep_idx, keep_stride, replicas,
            count_a, count_b);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

// --------------------------------------------------------------------------- //
// hidden_out[i] = hidden[keep_idx[i]], i < *S_out.  Rows are whole 16-byte chunks.
// The gather is driven by the copy engine: a worker is one thread, which moves (row, 8 KiB segment)
// items global -> shared -> global with bulk copies, kGbStages items in flight; no registers
// or warps are spent on the data.
constexpr int kGbStages = 4;
constexpr uint32_t kGbSegBytes = 8192;
constexpr size_t kGbWorkerBytes = (size_t)kGbStages * kGbSegBytes;
constexpr size_t kGbSmemBytes = kGbWorkerBytes + 128;

constexpr int kGatherWorkersMax = 6;      // workers of a CTA, and of an SM
struct GatherRows {
    const uint8_t* src;
    uint8_t* dst;
    const int32_t *keep_idx, *n_rows;
    uint32_t row_bytes;
    int src_rows;
    int32_t *status, *call_status;       // METOK_ERR_TIMEOUT to the first, and to the second if that is given and still 0
};

// Worker `first` of `stride`; stage0: its kGbWorkerBytes of shared memory, bars and abort_flag its own.
__device__ __forceinline__ void gather_rows_worker(const GatherRows& ga, long long first, long long stride, uint32_t stage0,
                                                   uint64_t* bars, volatile int* abort_flag) {
    using namespace sm100;
    for (int j = 0; j < kGbStages; ++j) mbar_init(smem_u32(&bars[j]), 1);
    *abort_flag = 0;
    mbar_fence_init();
    const int nseg = (int)((ga.row_bytes + kGbSegBytes - 1) / kGbSegBytes);
    const long long items = (long long)(*ga.n_rows) * nseg;
    const long long mine = first < items ? (items - first + stride - 1) / stride : 0;   // items of this worker
    auto issue_load = [&](long long k) {
        const long long it = first + k * stride;
        const int i = (int)(it / nseg), sg = (int)(it - (long long)i * nseg);
        const uint32_t off = (uint32_t)sg * kGbSegBytes;
        const uint32_t bytes = min(kGbSegBytes, ga.row_bytes - off);
        const uint32_t bar = smem_u32(&bars[k % kGbStages]);
        mbar_arrive_expect_tx(bar, bytes);
        const long long row = dbg_bound(ga.keep_idx[i], ga.src_rows, ga.status);
        if (!(dbg_withhold(ga.status, kDbgGatherRows) && first == 0 && k == 0))   // debug builds: one copy never sent
            bulk_load(stage0 + (uint32_t)(k % kGbStages) * kGbSegBytes, ga.src + (size_t)row * ga.row_bytes + off, bytes, bar);
    };
    for (long long k = 0; k < mine && k < kGbStages; ++k) issue_load(k);
    bool ok = true;
    for (long long k = 0; k < mine; ++k) {
        const int s = (int)(k % kGbStages);
        if (!mbar_wait(smem_u32(&bars[s]), (uint32_t)(k / kGbStages) & 1u, abort_flag)) { ok = false; break; }
        const long long it = first + k * stride;
        const int i = (int)(it / nseg), sg = (int)(it - (long long)i * nseg);
        const uint32_t off = (uint32_t)sg * kGbSegBytes;
        const uint32_t bytes = min(kGbSegBytes, ga.row_bytes - off);
        fence_proxy_async();
        bulk_store(ga.dst + (size_t)i * ga.row_bytes + off, stage0 + (uint32_t)s * kGbSegBytes, bytes);
        bulk_commit();
        // the stage of the item before this one is free once its store has read it
        if (k >= 1 && k - 1 + kGbStages < mine) {
            bulk_wait_read<1>();
            issue_load(k - 1 + kGbStages);
        }
    }
    bulk_wait_all();
    if (!ok) {
        // loads still in flight must land before the shared memory goes away
        for (int j = 0; j < kGbStages; ++j) mbar_wait(smem_u32(&bars[j]), 0u, abort_flag);
        *ga.status = METOK_ERR_TIMEOUT;
        if (ga.call_status) atomicCAS(ga.call_status, METOK_OK, METOK_ERR_TIMEOUT);
    }
}

__global__ void __launch_bounds__(32)
gather_rows_bulk_kernel(const __grid_constant__ GatherRows ga) {
    grid_dep_wait();
    extern __shared__ uint8_t gb_dyn[];
    __shared__ __align__(8) uint64_t s_bar[kGbStages];
    __shared__ int s_abort;
    if (threadIdx.x != 0) return;
    gather_rows_worker(ga, blockIdx.x, gridDim.x, (sm100::smem_u32(gb_dyn) + 127u) & ~127u, s_bar, &s_abort);
}

static int launch_gather(const GatherRows& ga, const char* timer_name, cudaStream_t st) {
    METOK_ALLOW_SMEM(gather_rows_bulk_kernel, kGbSmemBytes);
    {
        METOK_TIMED(timer_name, st);
        launch_chained(gather_rows_bulk_kernel, dim3(kNumSMs * 6), dim3(32), kGbSmemBytes, st, ga);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}
int launch_gather_rows_bulk(const void* src, void* dst, const int32_t* idx, const int32_t* n_rows, size_t row_bytes,
                            int src_rows, int32_t* status, const char* timer_name, cudaStream_t st) {
    return launch_gather({reinterpret_cast<const uint8_t*>(src), reinterpret_cast<uint8_t*>(dst), idx, n_rows, (uint32_t)row_bytes,
                          src_rows, status, nullptr}, timer_name, st);
}

static AttnDims make_dims(int Hq, int Hkv, int Lt, int S, int dh, int vis_start, int n_vis, float scale) {
    AttnDims dm;
    dm.Hq = Hq; dm.Hkv = Hkv; dm.Lt = Lt; dm.S = S; dm.dh = dh; dm.vis_start = vis_start; dm.n_vis = n_vis;
    dm.rep = Hq / Hkv;
    dm.R = dm.rep * Lt;
    dm.nrt = ceil_div(dm.R, kAtTile);
    dm.tiles_n = ceil_div(S, kAtTile);
    // as many runs of key tiles as give every place on the chip one, no more: a last round would cost as much as the others
    const int most = std::max(1, std::min(kAtMaxSplits, kNumSMs * sa_ctas_per_sm(kAtPT) / (dm.nrt * Hkv)));
    dm.per = ceil_div(dm.tiles_n, most);
    dm.nsplit = ceil_div(dm.tiles_n, dm.per);
    dm.scale_log2 = scale * kLog2e;
    return dm;
}

// The tensor-core scoring path takes bf16 with head dim 64 or 128; METOK_DEBUG_FORCE_SIMT=1 in
// the environment selects the CUDA-core kernels (debugging aid).
static bool use_mma_attn(int dtype, int dh) {
    static const bool force_simt = [] { const char* e = getenv("METOK_DEBUG_FORCE_SIMT"); return e && e[0] == '1'; }();
    return !force_simt && dtype == METOK_BF16 && (dh == 64 || dh == 128);
}

struct PrefillWs {
    int32_t* status;          // device status word, first in the workspace
    float *part_m, *part_l, *part_col;
    int n_planes;
};
static PrefillWs carve_prefill(Carver& cv, const AttnDims& dm, bool mma) {
    PrefillWs w;
    w.status = cv.take<int32_t>(64);
    if (mma) {
        size_t n_ml, n_col;
        attn_mma_workspace(dm.Hq, dm.Hkv, dm.Lt, dm.S, dm.n_vis, &n_ml, &n_col, &w.n_planes);
        w.part_m = cv.take<float>(n_ml);
        w.part_l = cv.take<float>(n_ml);
        w.part_col = cv.take<float>(n_col);
    } else {
        w.part_m = cv.take<float>((size_t)dm.Hkv * dm.nsplit * dm.R);
        w.part_l = cv.take<float>((size_t)dm.Hkv * dm.nsplit * dm.R);
        w.part_col = cv.take<float>((size_t)dm.Hkv * dm.nrt * dm.n_vis);
        w.n_planes = dm.Hkv * dm.nrt;
    }
    return w;
}

// One level's scoring as run_attention_scores takes it.
struct ScoreLevel {
    const void *q_text, *k_all;
    AttnDims dm;
    PrefillWs w;                  // all levels of a call have the same status area
    float* scores;
};

template <int NL>
static int launch_score_reduce(const ScoreLevel* lv, int n, float inv_rows, const int32_t* group, int32_t* origin, cudaStream_t st) {
    ReduceArgs<NL> ra = {};
    int blocks = 0;
    for (int l = 0; l < NL; ++l) {
        ra.lv[l].block0 = l < n ? blocks : 0x7FFFFFFF;
        if (l >= n) continue;
        ra.lv[l].part_col = lv[l].w.part_col;
        ra.lv[l].scores = lv[l].scores;
        ra.lv[l].n_vis = lv[l].dm.n_vis;
        blocks += ceil_div(lv[l].dm.n_vis, 256);
    }
    ra.nparts = lv[0].w.n_planes;                             // the same heads and queries on every level
    ra.inv_rows = inv_rows;
    ra.group = group;
    ra.origin = origin;
    ra.counts = lv[0].w.status + kStatusCounts;
    {
        METOK_TIMED("attn_score_reduce_kernel", st);
        launch_chained(attn_score_reduce_kernel<NL>, dim3(blocks), dim3(256), 0, st, ra);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

template <typename T>
static int launch_attn_passes(const void* q_text, const void* k_all, const AttnDims& dm, const PrefillWs& w, int32_t* clear, cudaStream_t st) {
    dim3 grid(dm.nsplit, dm.nrt, dm.Hkv);
    {
        METOK_TIMED("attn_stats_kernel", st);
        launch_chained(attn_stats_kernel<T>, grid, dim3(kSaThreads), 0, st, reinterpret_cast<const T*>(q_text), reinterpret_cast<const T*>(k_all),
                       dm, w.part_m, w.part_l, clear);
    }
    METOK_LAUNCH_CHECK();
    {
        METOK_TIMED("attn_colsum_kernel", st);
        launch_chained(attn_colsum_kernel<T>, grid, dim3(kSaThreads), 0, st, reinterpret_cast<const T*>(q_text),
                       reinterpret_cast<const T*>(k_all), dm, w.part_m, w.part_l, w.part_col);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

}  // namespace metok

using namespace metok;

// a5 as the calls run it, for one level or several: the status word and the class counts cleared, then the two passes and
// the plane sum; scores[j] = inv_rows * (sum over this call's heads and text queries of the probabilities).  group, origin:
// see attn_score_reduce_kernel.
static int run_attention_passes(const ScoreLevel* lv, int n, int dtype, float softmax_scale, cudaStream_t st) {
    const AttnDims& dm = lv[0].dm;
    int32_t* status = lv[0].w.status;
    if (use_mma_attn(dtype, dm.dh)) {                         // (the first stats kernel does the clearing)
        AttnScoreCall calls[kMaxPruneLevels];
        for (int l = 0; l < n; ++l)
            calls[l] = {lv[l].q_text, lv[l].k_all, lv[l].dm.S, lv[l].dm.vis_start, lv[l].dm.n_vis, lv[l].w.part_m, lv[l].w.part_l,
                        lv[l].w.part_col};
        const int rc = launch_attn_scores_mma(calls, n, dm.Hq, dm.Hkv, dm.Lt, dm.dh, softmax_scale, status, st);
        if (rc != METOK_OK) return rc;
    } else {
        for (int l = 0; l < n; ++l) {
            int32_t* clear = l == 0 ? status : nullptr;
            const int rc = dtype == METOK_F32 ? launch_attn_passes<float>(lv[l].q_text, lv[l].k_all, lv[l].dm, lv[l].w, clear, st)
                                              : launch_attn_passes<__nv_bfloat16>(lv[l].q_text, lv[l].k_all, lv[l].dm, lv[l].w, clear, st);
            if (rc != METOK_OK) return rc;
        }
    }
    return METOK_OK;
}
static int run_attention_scores(const ScoreLevel* lv, int n, int dtype, float softmax_scale, float inv_rows, const int32_t* group,
                                int32_t* origin, cudaStream_t st) {
    const int rc = run_attention_passes(lv, n, dtype, softmax_scale, st);
    if (rc != METOK_OK) return rc;
    return group ? launch_score_reduce<kMaxPruneLevels>(lv, n, inv_rows, group, origin, st)
                 : launch_score_reduce<1>(lv, 1, inv_rows, nullptr, nullptr, st);
}

extern "C" size_t metok_prefill_prune_workspace_bytes(int dtype, int Hq, int Hkv, int Lt, int S, int dh, int n_vis) {
    if (Hq < 1 || Hkv < 1 || Lt < 1 || S < 1 || dh < 1 || n_vis < 1 || Hq % Hkv) return 0;
    AttnDims dm = make_dims(Hq, Hkv, Lt, S, dh, 0, n_vis, 1.f);
    Carver cv(nullptr);
    carve_prefill(cv, dm, use_mma_attn(dtype, dh));
    return cv.total();
}

// Every check of metok_prefill_prune that needs no device: arguments, shapes, alignment, workspace.
static int validate_prefill_prune(const void* q_text, const void* k_all, const void* hidden, int dtype, int Hq,
                                  int Hkv, int Lt, int S, int dh, int D, int vis_start, int n_vis,
                                  const int32_t* token_group, int G, const int32_t* group_budget,
                                  float softmax_scale, const float* scores, const int32_t* keep_idx,
                                  const int32_t* S_out, const void* hidden_out, const void* ws, size_t ws_bytes) {
    if (!q_text || !k_all || !token_group || !group_budget || !scores || !keep_idx || !S_out)
        return METOK_ERR_INVALID_ARG;
    if ((hidden == nullptr) != (hidden_out == nullptr)) return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (Hq < 1 || Hkv < 1 || Lt < 1 || S < 1 || dh < 1 || n_vis < 1 || (hidden && D < 1)) return METOK_ERR_INVALID_ARG;
    if (Hq % Hkv != 0 || Lt > S) return METOK_ERR_INVALID_ARG;
    if (vis_start < 0 || (long long)vis_start + n_vis > (long long)S - Lt) return METOK_ERR_INVALID_ARG;
    if (G < 1 || G > METOK_MAX_GROUPS) return METOK_ERR_INVALID_ARG;
    for (int g = 0; g < G; ++g)
        if (group_budget[g] < 0) return METOK_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.f)) return METOK_ERR_INVALID_ARG;
    if (!aligned16(q_text) || !aligned16(k_all) || (hidden && (!aligned16(hidden) || !aligned16(hidden_out))))
        return METOK_ERR_INVALID_ARG;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (dtype == METOK_BF16 && dh != 64 && dh != 128) return METOK_ERR_UNSUPPORTED;
    if (dtype == METOK_F32 && (dh > 128 || dh % 4 != 0)) return METOK_ERR_UNSUPPORTED;
    if (hidden && ((long long)D * eb) % 16 != 0) return METOK_ERR_UNSUPPORTED;
    const size_t need = metok_prefill_prune_workspace_bytes(dtype, Hq, Hkv, Lt, S, dh, n_vis);
    if (!ws || ws_bytes < need || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    return METOK_OK;
}

extern "C" int metok_prefill_prune(const void* q_text, const void* k_all, const void* hidden, int dtype, int Hq,
                                   int Hkv, int Lt, int S, int dh, int D, int vis_start, int n_vis,
                                   const int32_t* token_group, int G, const int32_t* group_budget,
                                   float softmax_scale, float* scores, int32_t* keep_idx, int32_t* S_out,
                                   void* hidden_out, void* ws, size_t ws_bytes, void* stream) {
    const int vrc = validate_prefill_prune(q_text, k_all, hidden, dtype, Hq, Hkv, Lt, S, dh, D, vis_start, n_vis,
                                           token_group, G, group_budget, softmax_scale, scores, keep_idx, S_out,
                                           hidden_out, ws, ws_bytes);
    if (vrc != METOK_OK) return vrc;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);

    AttnDims dm = make_dims(Hq, Hkv, Lt, S, dh, vis_start, n_vis, softmax_scale);
    Carver cv(ws);
    PrefillWs w = carve_prefill(cv, dm, use_mma_attn(dtype, dh));
    int rc = debug_arm(w.status, st);
    if (rc != METOK_OK) return rc;
    const ScoreLevel lv = {q_text, k_all, dm, w, scores};
    const float inv_rows = 1.0f / (float)(Hq * Lt);
    const CsPlan plan = cs_plan(n_vis);
    const bool inside = plan.fits && plan.items == 4 && w.n_planes <= kPlanesInside &&
                        (long long)w.n_planes * n_vis * 4 <= (long long)plan.C * kPlaneBytesInside;
    rc = inside ? run_attention_passes(&lv, 1, dtype, softmax_scale, st)
                : run_attention_scores(&lv, 1, dtype, softmax_scale, inv_rows, nullptr, nullptr, st);
    if (rc != METOK_OK) return rc;
    rc = class_topk(scores, 0, token_group, n_vis, G, group_budget, S, vis_start, keep_idx, 0, 1, S_out, nullptr, 1,
                    {w.part_col, inside ? w.n_planes : 0, inv_rows, scores}, st);
    if (rc != METOK_OK) return rc;
    if (hidden) {
        rc = launch_gather_rows_bulk(hidden, hidden_out, keep_idx, S_out, (size_t)D * eb, S, w.status, "gather_rows_kernel",
                                     st);
        if (rc != METOK_OK) return rc;
    }
    return METOK_OK;
}

extern "C" int metok_attention_scores(const void* q_text, const void* k_all, int dtype, int Hq, int Hkv, int Lt, int S,
                                      int dh, int vis_start, int n_vis, float softmax_scale, int rows_total,
                                      float* scores, void* ws, size_t ws_bytes, void* stream) {
    if (!q_text || !k_all || !scores) return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (Hq < 1 || Hkv < 1 || Lt < 1 || S < 1 || dh < 1 || n_vis < 1) return METOK_ERR_INVALID_ARG;
    if (Hq % Hkv != 0 || Lt > S) return METOK_ERR_INVALID_ARG;
    if (vis_start < 0 || (long long)vis_start + n_vis > (long long)S - Lt) return METOK_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.f) || !aligned16(q_text) || !aligned16(k_all)) return METOK_ERR_INVALID_ARG;
    if (rows_total != 0 && (long long)rows_total < (long long)Hq * Lt) return METOK_ERR_INVALID_ARG;
    if (dtype == METOK_BF16 && dh != 64 && dh != 128) return METOK_ERR_UNSUPPORTED;
    if (dtype == METOK_F32 && (dh > 128 || dh % 4 != 0)) return METOK_ERR_UNSUPPORTED;
    const size_t need = metok_prefill_prune_workspace_bytes(dtype, Hq, Hkv, Lt, S, dh, n_vis);
    if (!ws || ws_bytes < need || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    AttnDims dm = make_dims(Hq, Hkv, Lt, S, dh, vis_start, n_vis, softmax_scale);
    Carver cv(ws);
    PrefillWs w = carve_prefill(cv, dm, use_mma_attn(dtype, dh));
    const float inv_rows = 1.0f / (float)(rows_total ? rows_total : Hq * Lt);
    if (const int rc = debug_arm(w.status, reinterpret_cast<cudaStream_t>(stream))) return rc;
    const ScoreLevel lv = {q_text, k_all, dm, w, scores};
    return run_attention_scores(&lv, 1, dtype, softmax_scale, inv_rows, nullptr, nullptr, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" size_t metok_prune_by_scores_workspace_bytes(void) { return 1024; }

extern "C" int metok_prune_by_scores(const float* scores, const void* hidden, int dtype, int S, int D, int vis_start,
                                     int n_vis, const int32_t* token_group, int G, const int32_t* group_budget,
                                     int32_t* keep_idx, int32_t* S_out, void* hidden_out, void* ws, size_t ws_bytes,
                                     void* stream) {
    if (!scores || !token_group || !group_budget || !keep_idx || !S_out) return METOK_ERR_INVALID_ARG;
    if ((hidden == nullptr) != (hidden_out == nullptr)) return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (S < 1 || n_vis < 1 || (hidden && D < 1)) return METOK_ERR_INVALID_ARG;
    if (vis_start < 0 || (long long)vis_start + n_vis > (long long)S) return METOK_ERR_INVALID_ARG;
    if (G < 1 || G > METOK_MAX_GROUPS) return METOK_ERR_INVALID_ARG;
    for (int g = 0; g < G; ++g)
        if (group_budget[g] < 0) return METOK_ERR_INVALID_ARG;
    if (hidden && (!aligned16(hidden) || !aligned16(hidden_out))) return METOK_ERR_INVALID_ARG;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (hidden && ((long long)D * eb) % 16 != 0) return METOK_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < metok_prune_by_scores_workspace_bytes() || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int32_t* status = reinterpret_cast<int32_t*>(ws);
    METOK_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int32_t), st));
    int rc = debug_arm(status, st);
    if (rc != METOK_OK) return rc;
    rc = launch_class_topk(scores, 0, token_group, n_vis, G, group_budget, S, vis_start, keep_idx, 0, 1, S_out,
                               nullptr, 1, st);
    if (rc != METOK_OK) return rc;
    if (hidden)
        rc = launch_gather_rows_bulk(hidden, hidden_out, keep_idx, S_out, (size_t)D * eb, S, status, "gather_rows_kernel", st);
    return rc;
}

extern "C" int metok_retention_budgets(double alpha, double r, int stage, const int32_t* N0, int32_t* budget) {
    if (!N0 || !budget) return METOK_ERR_INVALID_ARG;
    if (!(alpha > 0.0 && alpha <= 1.0) || !(r > 0.0 && r <= 1.0)) return METOK_ERR_INVALID_ARG;
    if (stage < 0 || stage > 3 || N0[0] < 0 || N0[1] < 0) return METOK_ERR_INVALID_ARG;
    double rk, rn;
    switch (stage) {
        case 0: rk = 1.0; rn = 1.0; break;
        case 1: rk = r; rn = alpha * r; break;
        case 2: rk = r * r; rn = 0.0; break;
        default: rk = 0.0; rn = 0.0; break;
    }
    int bk = ceilq(rk * (double)N0[0]), bn = ceilq(rn * (double)N0[1]);
    budget[0] = bk < N0[0] ? bk : N0[0];
    budget[1] = bn < N0[1] ? bn : N0[1];
    return METOK_OK;
}

// --------------------------------------------------------------------------- //
// The pruning levels chained on the device.
// --------------------------------------------------------------------------- //
namespace metok {

// What a level hands to the next one and to the caller.
struct ScheduleHand {
    const int32_t *group, *origin;                    // of this level's tokens; origin null: the first level, token i is i
    int32_t *group_next, *origin_next;                // of the next level's n_next tokens; null: no next level
    int n_next;
    const int32_t* level_status;                      // the attention passes' status word and the class counts behind it
    int32_t* status;                                  // the caller's: written on the first level, later only if still 0
    bool first;
    int n0_key, n0_nonkey, n_vis;
};
__device__ __forceinline__ void schedule_check(const ScheduleHand& h) {
    if (h.first) {
        const int c0 = h.level_status[kStatusCounts], c1 = h.level_status[kStatusCounts + 1];
        *h.status = c0 == h.n0_key && c1 == h.n0_nonkey && c0 + c1 == h.n_vis ? *h.level_status : METOK_ERR_INVALID_ARG;
    } else if (*h.level_status != METOK_OK) {
        atomicCAS(h.status, METOK_OK, *h.level_status);
    }
}

// One level of a schedule: the class-wise selection of up to 81 920 items (as cs_topk_kernel), class and origin of every
// survivor for the next level, and beside it the hidden rows of the level before.  CTAs 0 .. C - 1 select; each of the others runs
// `workers` gather workers.  The selection is a chain of latencies in eight SMs or one and the gather is bound by memory.  What it
// saves is the launches, 3 us for every one that handed classes and origins on; under ncu (18 432 tokens) the second level's launch
// takes 21.6 us where its selection and the gather alone take 9 and 15, the third's 9.9 for 5 and 7.5: the gather's CTAs come in
// the selection's clusters of eight and deal the rows out by a fixed stride, so those placed late end late.
template <int IT, bool kCl>
__global__ void __launch_bounds__(IT == kCsMaxItems ? kCsMaxItemsThreads : 1024)
schedule_select_kernel(const float* __restrict__ sc, int n_vis, CsLayout lay, TopkBudgets budgets, int S, int vis_start,
                       int32_t* __restrict__ keep, int32_t* __restrict__ S_out, const __grid_constant__ ScheduleHand hand,
                       const __grid_constant__ GatherRows ga, int workers) {
    cs_enter<kCl>();
    grid_dep_wait();
    constexpr int C = kCl ? kCsMaxCluster : 1;
    __shared__ CsShared sm;
    __shared__ __align__(8) uint64_t s_bar[kGatherWorkersMax][kGbStages];
    __shared__ int s_abort[kGatherWorkersMax];
    extern __shared__ __align__(16) unsigned char sel_dyn[];
    const int tid = threadIdx.x, nthr = blockDim.x, rank = blockIdx.x;
    if (rank >= C) {
        const int w = tid >> 5;
        if (w < workers && (tid & 31) == 0)
            gather_rows_worker(ga, (long long)(rank - C) * workers + w, (long long)(gridDim.x - C) * workers,
                               ((sm100::smem_u32(sel_dyn) + 127u) & ~127u) + (uint32_t)(w * kGbWorkerBytes), s_bar[w], &s_abort[w]);
        __syncwarp();
        if constexpr (kCl) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // of cs_enter()
        return;
    }
    if (rank == 0 && tid == 0) schedule_check(hand);
    const int32_t* group = hand.group;
    const CsSlice sl = cs_slice<IT>(n_vis, rank, C);
    auto load = [&](int, int i, float& v, int& c) {
        v = sc[i];
        c = group[i];
        if (c >= 2) c = -1;
    };
    int before, kept;
    const uint32_t bits = cs_select<IT, kCl, false>(sm, sel_dyn, lay, 2, budgets.v, rank, sl.i_first, sl.i_hi, load, &before, &kept);
    const int outside = S - n_vis;
    cs_for_items<IT>(bits, before, sl.i_first, sl.i_hi, [&](int, int i, int place, bool k) {
        if (!k) return;
        keep[vis_start + place] = vis_start + i;
        if (hand.group_next && place < hand.n_next) {
            hand.group_next[place] = group[i];
            hand.origin_next[place] = hand.origin ? hand.origin[i] : i;
        }
    });
    for (int i = rank * nthr + tid; i < outside; i += C * nthr)
        keep[i < vis_start ? i : kept + i] = i < vis_start ? i : i + n_vis;
    if (hand.group_next)                                      // fewer survivors than N0 says (the status word says so)
        for (int i = kept + rank * nthr + tid; i < hand.n_next; i += C * nthr) {
            hand.group_next[i] = group[n_vis - 1];
            hand.origin_next[i] = hand.origin ? hand.origin[n_vis - 1] : n_vis - 1;
        }
    if (rank == 0 && tid == 0) *S_out = outside + kept;
}

// After a selection by select.cuh (a level of more than 81 920 tokens): class and origin of the i-th surviving visual token.
// The keep list holds every position before the visual span, so its entry vis_start + i is that token's position.
__global__ void __launch_bounds__(256)
schedule_propagate_kernel(const int32_t* __restrict__ keep_idx, int vis_start, int n_cur, const __grid_constant__ ScheduleHand hand) {
    grid_dep_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) schedule_check(hand);
    if (!hand.group_next || i >= hand.n_next) return;
    int j = keep_idx[vis_start + i] - vis_start;
    j = j < 0 ? 0 : (j >= n_cur ? n_cur - 1 : j);            // only reached with a wrong N0 (status says so)
    hand.group_next[i] = hand.group[j];
    hand.origin_next[i] = hand.origin ? hand.origin[j] : j;
}

// The selection of one level; `ga` (may be null): the gather that runs beside it.
static int launch_schedule_select(const float* scores, int n_vis, const int32_t* budget, int S, int vis_start, int32_t* keep_idx,
                                  int32_t* S_out, const ScheduleHand& hand, const GatherRows* ga, cudaStream_t st) {
    const CsPlan plan = cs_plan(n_vis);
    if (!plan.fits) {
        int rc = ga ? launch_gather(*ga, "gather_rows_kernel", st) : METOK_OK;
        if (rc == METOK_OK)
            rc = launch_class_topk(scores, 0, hand.group, n_vis, 2, budget, S, vis_start, keep_idx, 0, 1, S_out, nullptr, 1, st);
        if (rc != METOK_OK) return rc;
        METOK_TIMED("schedule_propagate_kernel", st);
        launch_chained(schedule_propagate_kernel, dim3(std::max(1, ceil_div(hand.n_next, 256))), dim3(256), 0, st, keep_idx, vis_start,
                       n_vis, hand);
        METOK_LAUNCH_CHECK();
        return METOK_OK;
    }
    TopkBudgets b = {};
    b.v[0] = budget[0];
    b.v[1] = budget[1];
    const CsLayout lay = cs_layout(2, n_vis);
    // The gather's CTAs have the selection's threads and registers: one that is alone on its SM holds six workers (the copies
    // in flight that the gather has when it is launched alone), one of two holds three.
    const int workers = std::min(plan.threads / 32, plan.threads > (plan.items == 4 ? 512 : 320) ? kGatherWorkersMax : kGatherWorkersMax / 2);
    size_t smem = lay.bytes;
    int grid = plan.C;
    GatherRows none = {};
    if (ga) {
        smem = std::max(smem, workers * kGbWorkerBytes + 128);
        const int ctas = kNumSMs * kGatherWorkersMax / workers;
        grid += (ctas - plan.C) / plan.C * plan.C;
    }
    auto launch = [&](auto kernel) -> int {
        if (smem > 32 * 1024) METOK_ALLOW_SMEM(kernel, smem);
        METOK_TIMED("schedule_select_kernel", st);
        launch_chained_clusters(plan.C, kernel, dim3(grid), dim3(plan.threads), smem, st, scores, n_vis, lay, b, S, vis_start, keep_idx,
                                S_out, hand, ga ? *ga : none, workers);
        METOK_LAUNCH_CHECK();
        return METOK_OK;
    };
    if (plan.C == 1) return launch(schedule_select_kernel<4, false>);
    if (plan.items == 4) return launch(schedule_select_kernel<4, true>);
    return launch(schedule_select_kernel<kCsMaxItems, true>);
}

// Whether the levels' scoring and selection may run ahead of the gathers before them: no array that one level writes is
// read or written by another, except hidden rows, whose gathers stay in order.
static bool schedule_levels_apart(const metok_prune_level* lv, int n, const int32_t* sizes, int S, int n_vis, int Hq, int Hkv, int Lt,
                                  int dh, int D, int eb) {
    struct Range { uintptr_t lo, hi; };
    auto range = [](const void* p, size_t bytes) { return Range{(uintptr_t)p, p ? (uintptr_t)p + bytes : (uintptr_t)p}; };
    auto meet = [](const Range& a, const Range& b) { return a.lo < b.hi && b.lo < a.hi; };
    Range w[kMaxPruneLevels][5], r[kMaxPruneLevels][4];
    for (int s = 0; s < n; ++s) {
        const size_t nv = sizes[s], rows = (size_t)(S - n_vis + sizes[s]);
        w[s][0] = range(lv[s].scores, nv * 4);
        w[s][1] = range(lv[s].keep_idx, rows * 4);
        w[s][2] = range(lv[s].S_out, 4);
        w[s][3] = range(lv[s].origin, nv * 4);
        w[s][4] = range(lv[s].token_group, nv * 4);           // (written where s > 0)
        r[s][0] = range(lv[s].q_text, (size_t)Hq * Lt * dh * eb);
        r[s][1] = range(lv[s].k_all, (size_t)Hkv * rows * dh * eb);
        r[s][2] = range(lv[s].hidden, rows * D * eb);
        r[s][3] = range(lv[s].hidden_out, rows * D * eb);
    }
    for (int a = 0; a < n; ++a)
        for (int b = 0; b < n; ++b) {
            if (a == b) continue;
            for (const Range& x : w[a]) {
                for (const Range& y : w[b]) if (meet(x, y)) return false;
                for (const Range& y : r[b]) if (meet(x, y)) return false;
            }
            if (meet(r[a][3], r[b][0]) || meet(r[a][3], r[b][1])) return false;
        }
    return true;
}

}  // namespace metok

namespace metok {
struct KvListSrc { const int32_t* keep_idx[4]; const int32_t* S_out[4]; int S_in[4]; };   // per layer group
// Layer l of group g (the pruning layers at or below it: g of them) holds the rows of level g's input;
// its list is the keep list recorded by level g + 1, or everything when no level follows.
__global__ void __launch_bounds__(256)
schedule_kv_lists_kernel(KvListSrc src, const int32_t* __restrict__ layer_group, int stride,
                         int32_t* __restrict__ kv_keep_idx, int32_t* __restrict__ kv_keep_len) {
    grid_dep_wait();
    const int layer = blockIdx.x;
    const int g = layer_group[layer];
    int32_t* out = kv_keep_idx + (size_t)layer * stride;
    const int32_t* keep = src.keep_idx[g];
    const int n = keep ? *src.S_out[g] : src.S_in[g];
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = keep ? keep[i] : i;
    if (threadIdx.x == 0) kv_keep_len[layer] = n;
}
}  // namespace metok

extern "C" int metok_prune_schedule_kv_lists(const metok_prune_level* levels, int n_levels, const int32_t* level_layer,
                                             int L, int S, int n_vis, double alpha, double r, const int32_t* N0,
                                             int32_t* kv_keep_idx, int32_t* kv_keep_len, int32_t* kv_S_cur,
                                             void* ws, size_t ws_bytes, void* stream) {
    if (!levels || !level_layer || !N0 || !kv_keep_idx || !kv_keep_len || !kv_S_cur) return METOK_ERR_INVALID_ARG;
    if (L < 1 || S < 1 || n_vis < 1 || n_vis > S) return METOK_ERR_INVALID_ARG;
    int32_t sizes[4];
    const int rc = metok_prune_schedule_sizes(n_levels, alpha, r, N0, sizes);
    if (rc != METOK_OK) return rc;
    if (sizes[0] != n_vis) return METOK_ERR_INVALID_ARG;
    for (int s = 0; s < n_levels; ++s) {
        if (!levels[s].keep_idx || !levels[s].S_out) return METOK_ERR_INVALID_ARG;
        if (level_layer[s] < 0 || (s > 0 && level_layer[s] <= level_layer[s - 1])) return METOK_ERR_INVALID_ARG;
    }
    if (!ws || ws_bytes < (size_t)L * sizeof(int32_t) || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    metok::KvListSrc src;
    for (int g = 0; g < 4; ++g) {
        src.keep_idx[g] = g < n_levels ? levels[g].keep_idx : nullptr;
        src.S_out[g] = g < n_levels ? levels[g].S_out : nullptr;
        src.S_in[g] = g <= n_levels ? S - n_vis + sizes[g] : 0;
    }
    // the group of every layer, known on the host
    int32_t group_host[1024];
    if (L > 1024) return METOK_ERR_UNSUPPORTED;
    for (int l = 0; l < L; ++l) {
        int g = 0;
        while (g < n_levels && level_layer[g] <= l) ++g;
        group_host[l] = g;
        kv_S_cur[l] = src.S_in[g];
    }
    int32_t* group_dev = reinterpret_cast<int32_t*>(ws);
    METOK_CUDA_TRY(cudaMemcpyAsync(group_dev, group_host, (size_t)L * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    {
        METOK_TIMED("schedule_kv_lists_kernel", st);
        metok::launch_chained(metok::schedule_kv_lists_kernel, dim3(L), dim3(256), 0, st, src, group_dev, S, kv_keep_idx, kv_keep_len);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

extern "C" int metok_prune_schedule_sizes(int n_levels, double alpha, double r, const int32_t* N0,
                                          int32_t* n_vis_of_level) {
    if (!N0 || !n_vis_of_level || n_levels < 1 || n_levels > 3) return METOK_ERR_INVALID_ARG;
    for (int s = 0; s <= n_levels; ++s) {
        int32_t b[2];
        const int rc = metok_retention_budgets(alpha, r, s, N0, b);
        if (rc != METOK_OK) return rc;
        n_vis_of_level[s] = b[0] + b[1];
    }
    return METOK_OK;
}

extern "C" size_t metok_prefill_prune_schedule_workspace_bytes(int n_levels, int dtype, int Hq, int Hkv, int Lt, int S,
                                                               int dh, int n_vis, double alpha, double r,
                                                               const int32_t* N0) {
    int32_t sizes[4];
    if (metok_prune_schedule_sizes(n_levels, alpha, r, N0, sizes) != METOK_OK || sizes[0] != n_vis) return 0;
    Carver cv(nullptr);
    for (int s = 0; s < n_levels; ++s) {
        const int S_s = S - n_vis + sizes[s];
        if (metok_prefill_prune_workspace_bytes(dtype, Hq, Hkv, Lt, S_s, dh, sizes[s]) == 0) return 0;
        carve_prefill(cv, make_dims(Hq, Hkv, Lt, S_s, dh, 0, sizes[s], 1.f), use_mma_attn(dtype, dh));
    }
    return cv.total();
}

extern "C" int metok_prefill_prune_schedule(const metok_prune_level* levels, int n_levels, int dtype, int Hq, int Hkv,
                                            int Lt, int S, int dh, int D, int vis_start, int n_vis, double alpha,
                                            double r, const int32_t* N0, float softmax_scale, int32_t* status,
                                            void* ws, size_t ws_bytes, void* stream) {
    if (!levels || !N0 || !status) return METOK_ERR_INVALID_ARG;
    int32_t sizes[4];
    int rc = metok_prune_schedule_sizes(n_levels, alpha, r, N0, sizes);
    if (rc != METOK_OK) return rc;
    if (sizes[0] != n_vis || n_vis < 1) return METOK_ERR_INVALID_ARG;
    for (int s = 0; s < n_levels; ++s) {
        if (sizes[s] < 1) return METOK_ERR_INVALID_ARG;
        if (!levels[s].token_group || !levels[s].origin) return METOK_ERR_INVALID_ARG;
    }
    // every level's arguments, shapes and workspace are checked before the first launch
    for (int s = 0; s < n_levels; ++s) {
        const metok_prune_level& lv = levels[s];
        int32_t budget[2];
        rc = metok_retention_budgets(alpha, r, s + 1, N0, budget);
        if (rc != METOK_OK) return rc;
        rc = validate_prefill_prune(lv.q_text, lv.k_all, lv.hidden, dtype, Hq, Hkv, Lt, S - n_vis + sizes[s], dh, D,
                                    vis_start, sizes[s], lv.token_group, 2, budget, softmax_scale, lv.scores,
                                    lv.keep_idx, lv.S_out, lv.hidden_out, ws, ws_bytes);
        if (rc != METOK_OK) return rc;
    }
    // scratch for the largest level only: the levels follow one another and use it in turn
    const bool shared = ws_bytes < metok_prefill_prune_schedule_workspace_bytes(n_levels, dtype, Hq, Hkv, Lt, S, dh, n_vis, alpha, r, N0);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int eb = dtype == METOK_F32 ? 4 : 2;
    const bool apart = !shared && schedule_levels_apart(levels, n_levels, sizes, S, n_vis, Hq, Hkv, Lt, dh, D, eb);
    ScoreLevel sl[kMaxPruneLevels];
    Carver cv(ws);
    for (int s = 0; s < n_levels; ++s) {
        const AttnDims dm = make_dims(Hq, Hkv, Lt, S - n_vis + sizes[s], dh, vis_start, sizes[s], softmax_scale);
        if (shared) cv = Carver(ws);
        sl[s] = {levels[s].q_text, levels[s].k_all, dm, carve_prefill(cv, dm, use_mma_attn(dtype, dh)), levels[s].scores};
        if (s > 0) sl[s].w.status = sl[0].w.status;
    }
    int32_t* level_status = sl[0].w.status;
    rc = debug_arm(level_status, st);
    if (rc != METOK_OK) return rc;
    // Nothing but the classes, origins and row numbers passes from level to level, so all levels are scored first, in the
    // launches of one.  Buffers that levels share make the levels follow one another.
    const float inv_rows = 1.0f / (float)(Hq * Lt);
    GatherRows pending = {};                                  // the hidden rows of the level before
    for (int s = 0; s < n_levels; ++s) {
        const metok_prune_level& lv = levels[s];
        int32_t budget[2];
        rc = metok_retention_budgets(alpha, r, s + 1, N0, budget);
        if (rc != METOK_OK) return rc;
        if (s == 0 || !apart) {
            if (pending.src) rc = launch_gather(pending, "gather_rows_kernel", st);
            pending = {};
            if (rc == METOK_OK)
                rc = run_attention_scores(sl + s, apart ? n_levels : 1, dtype, softmax_scale, inv_rows, s == 0 ? lv.token_group : nullptr,
                                          lv.origin, st);
            if (rc != METOK_OK) return rc;
        }
        const bool more = s + 1 < n_levels;
        const ScheduleHand hand = {lv.token_group, s == 0 ? nullptr : lv.origin, more ? levels[s + 1].token_group : nullptr,
                                   more ? levels[s + 1].origin : nullptr, more ? sizes[s + 1] : 0, level_status,
                                   status, s == 0, N0[0], N0[1], n_vis};
        const int S_s = S - n_vis + sizes[s];
        rc = launch_schedule_select(lv.scores, sizes[s], budget, S_s, vis_start, lv.keep_idx, lv.S_out, hand,
                                    pending.src ? &pending : nullptr, st);
        if (rc != METOK_OK) return rc;
        pending = {};
        if (lv.hidden)
            pending = {reinterpret_cast<const uint8_t*>(lv.hidden), reinterpret_cast<uint8_t*>(lv.hidden_out), lv.keep_idx, lv.S_out,
                       (uint32_t)((size_t)D * eb), S_s, level_status, status};
    }
    return pending.src ? launch_gather(pending, "gather_rows_kernel", st) : METOK_OK;
}
