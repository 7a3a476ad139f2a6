// metok_compress_vision: text relevance and key events (Eq. 5), per-event key-token
// top-k, merge-assign of the remaining tokens and averaging.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "common.cuh"
#include "select.cuh"
#include "select_cluster.cuh"
#include "simt_tile.cuh"
#include "sm100.cuh"
#include "launchers.h"

namespace metok {

// --------------------------------------------------------------------------- //
// token_score[j] = <x_j, t> / (max(|x_j|, eps) * max(|t|, eps)); also 1/max(|x_j|, eps).
// One warp per token row, 16-byte loads, eight chunks of the row in flight per lane.  The text's chunks are read
// beside them (they stay in L1), so a CTA has nothing to prepare: with the text laid out in shared memory first, a
// CTA of 64 rows x 196 tokens x 1152 spent more time on that than on its rows (11.5 us; 8.4 now).
// --------------------------------------------------------------------------- //
template <typename T>
__device__ __forceinline__ void widen_chunk(const uint4& r, float (&v)[16 / sizeof(T)]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (sizeof(T) == 4) {
            v[i] = __uint_as_float(w[i]);
        } else {
            v[2 * i]     = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
tok_score_kernel(const T* __restrict__ feats, const T* __restrict__ text, int Nv, int d,
                 float* __restrict__ token_score, float* __restrict__ inv_norm) {
    grid_dep_wait();
    constexpr int VN = Vec16<T>::N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nchunk = d / VN;
    const uint4* t4 = reinterpret_cast<const uint4*>(text);
    // rows from the last one down: the pass before this one (segmentation) streams V upwards
    // and leaves its tail in L2
    for (int rr = blockIdx.x * 8 + warp; rr < Nv; rr += gridDim.x * 8) {
        const int row = Nv - 1 - rr;
        const uint4* x4 = reinterpret_cast<const uint4*>(feats) + (size_t)row * nchunk;
        float nn = 0.f, dt = 0.f, tt = 0.f;
        constexpr int U = 8;                        // 16-byte chunks in flight per lane
        for (int c0 = 0; c0 < nchunk; c0 += 32 * U) {
            uint4 raw[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + u * 32 + lane;
                raw[u] = c < nchunk ? __ldg(x4 + c) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + u * 32 + lane;
                if (c < nchunk) {
                    float v[VN], t[VN];
                    widen_chunk<T>(raw[u], v);
                    widen_chunk<T>(__ldg(t4 + c), t);
#pragma unroll
                    for (int i = 0; i < VN; ++i) {
                        nn = fmaf(v[i], v[i], nn);
                        dt = fmaf(v[i], t[i], dt);
                        tt = fmaf(t[i], t[i], tt);
                    }
                }
            }
        }
        nn = warp_sum(nn);
        dt = warp_sum(dt);
        tt = warp_sum(tt);
        if (lane == 0) {
            const float n = fmaxf(sqrtf(nn), kEps), tn = fmaxf(sqrtf(tt), kEps);
            token_score[row] = dt / (n * tn);
            inv_norm[row] = 1.0f / n;
        }
    }
}

// Index e with off[e] <= t < off[e+1] in an ascending offset array off[0..k].
__device__ __forceinline__ int find_event(const int32_t* __restrict__ off, int k, int t) {
    int lo = 0, hi = k;                     // off[lo] <= t < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// Event scores, key events, per-event token budgets and output offsets.  One CTA; with many frames a cluster, whose
// other CTAs only average frames for it (512 frames: 13.4 us with one CTA, 6.5 with four).
// The offsets are the caller's memory: they are held to [0, Tn], and where they descend (events that overlap would want
// more outputs than the caller has room for) an offset is raised to the largest before it and the call's status word says
// METOK_ERR_INVALID_ARG.  Events of no frames are taken as they are: no key token, no output.
// The shape of a merge unit: up to `rows` tokens that are no key token x up to `cols` key tokens of an event.
struct MergeShape { int rows, cols; };
struct PlanParams {
    int Tn, N, k, n_key_events, event_agg, mode;
    // The tensor-core merge of bf16 reads shape and list only where there are more than kMmaEvents events (leaving the list out elsewhere
    // changes no time: 32 x 144 tokens in 4 events 42.3 us the path either way, 512 x 144 in 64 211).
    MergeShape shape;
    int grid, s1, s2, s1_nonkey, s2_nonkey;     // POOL: side of the token grid and the four strides
    double keep_key, keep_nonkey, beta;
    const uint8_t* key_given;                   // the caller's key events, or null
    const uint8_t* key_frames_given;            // POOL: the caller's key frames, or null
};

__global__ void __launch_bounds__(1024, 1)                      // left to itself ptxas takes 32 registers and spills: 7.3 -> 7.6 us under ncu
event_plan_kernel(const float* __restrict__ token_score, float* __restrict__ frame_score,
                  const int32_t* __restrict__ event_offsets, PlanParams pp,
                  float* __restrict__ event_score, uint8_t* __restrict__ event_is_key,
                  int32_t* __restrict__ ev_lo, int32_t* __restrict__ ev_budget, int32_t* __restrict__ ev_out_off,
                  int32_t* ev_unit_off,
                  int32_t* __restrict__ frame_ev, int32_t* __restrict__ frame_stride,
                  int32_t* __restrict__ frame_off, int32_t* __restrict__ n_out, int32_t* __restrict__ counters, int n_counters,
                  int32_t* __restrict__ status) {
    const int C = (int)gridDim.x, rank = (int)blockIdx.x;
    if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    grid_dep_wait();
    extern __shared__ float s_score[];      // [k]
    if (rank == 0 && threadIdx.x == 0) *status = 0;
    for (int i = rank * 1024 + threadIdx.x; i < n_counters; i += C * 1024) counters[i] = 0;   // what later kernels of the call count in
    __shared__ int s_scan[32];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int k = pp.k, Tn = pp.Tn;
    // frame_score[f] = mean of the frame's N token scores; eight lanes per frame (a lane's loads are
    // independent), fixed shuffle tree; the scores stay in shared memory for the event loops below
    float* s_frame = s_score + k;           // [Tn]
    int* s_off = reinterpret_cast<int*>(s_frame + Tn);      // [k + 1] event_offsets, clamped
    int* s_bud = s_off + k + 1;                              // [k] budget of the event
    int* s_units = s_bud + k;                                // [k] merge units of the event
    unsigned char* s_key = reinterpret_cast<unsigned char*>(s_units + k);   // [k]
    const int off0 = tid <= k ? event_offsets[tid] : 0;     // on its way while the frames are averaged
    float* s_frame0 = s_frame;              // the first CTA's
    if (C > 1) {
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // everybody has started
        s_frame0 = cg::this_cluster().map_shared_rank(s_frame, 0);
    }
    for (int f0 = rank * (nthr >> 3); f0 < Tn; f0 += C * (nthr >> 3)) {
        const int f = f0 + (tid >> 3), part = tid & 7;
        float s = 0.f;
        if (f < Tn) {
            constexpr int kB = 9;                           // loads in flight; the additions keep their order
            for (int p0 = part; p0 < pp.N; p0 += 8 * kB) {
                float x[kB];
#pragma unroll
                for (int u = 0; u < kB; ++u) x[u] = p0 + 8 * u < pp.N ? token_score[(size_t)f * pp.N + p0 + 8 * u] : 0.f;
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (p0 + 8 * u < pp.N) s += x[u];
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        if (f < Tn && part == 0) {
            s /= (float)pp.N;
            s_frame0[f] = s;
            frame_score[f] = s;
        }
    }
    for (int e = tid; e <= k; e += nthr) s_off[e] = min(max(e == tid ? off0 : event_offsets[e], 0), Tn);
    if (C > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank > 0) return;
    } else {
        __syncthreads();
    }
    bool descends = false;
    for (int e = tid; e < k; e += nthr) {
        const int lo = s_off[e], hi = s_off[e + 1];
        descends |= hi < lo;
        ev_lo[e] = lo;
        if (e == k - 1) ev_lo[k] = hi;
        float s;
        if (hi <= lo) {
            s = -3.0e38f;
        } else if (pp.event_agg == METOK_AGG_MEAN) {
            float a = 0.f;
#pragma unroll 8
            for (int f = lo; f < hi; ++f) a += s_frame[f];
            s = a / (float)(hi - lo);
        } else {
            float a = s_frame[lo];
#pragma unroll 8
            for (int f = lo + 1; f < hi; ++f) a = fmaxf(a, s_frame[f]);
            s = a;
        }
        s_score[e] = s;
        event_score[e] = s;
    }
    if (__syncthreads_or(descends)) {
        if (tid == 0) {
            for (int e = 1; e <= k; ++e) {
                s_off[e] = max(s_off[e], s_off[e - 1]);
                ev_lo[e] = s_off[e];
            }
            *status = METOK_ERR_INVALID_ARG;
        }
        __syncthreads();
    }
    for (int e = tid; e < k; e += nthr) {
        const float v = s_score[e];
        int rank = 0;
        for (int j = 0; j < k; ++j) {
            const float w = s_score[j];
            rank += (w > v) || (w == v && j < e);
        }
        const bool key = pp.key_given ? pp.key_given[e] != 0 : rank < pp.n_key_events;
        event_is_key[e] = (uint8_t)key;
        s_key[e] = (unsigned char)key;
    }
    __syncthreads();
    if (pp.mode == METOK_MODE_TOPK_MERGE) {
        auto units = [&](int m, int b, const MergeShape& s) {                // row tiles x key chunks
            return (m - b + s.rows - 1) / s.rows * ((b + s.cols - 1) / s.cols);
        };
        for (int e = tid; e < k; e += nthr) {
            const int m = (s_off[e + 1] - s_off[e]) * pp.N;
            const double ratio = s_key[e] ? pp.keep_key : pp.keep_nonkey;
            const double c = ratio * (double)m - 1e-9;
            long long b = (long long)c;
            if ((double)b < c) b += 1;
            if (b < 1) b = 1;
            if (b > m) b = m;
            ev_budget[e] = (int)b;
            s_bud[e] = (int)b;
            s_units[e] = units(m, (int)b, pp.shape);
        }
        __syncthreads();
        if (tid < 32) {                                     // offsets: one warp, 32 events at a time
            int slots = 0, units = 0;
            for (int e0 = 0; e0 < k; e0 += 32) {
                const int e = e0 + tid, b = e < k ? s_bud[e] : 0, u = e < k ? s_units[e] : 0;
                int bi = b, ui = u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xFFFFFFFFu, bi, o), y = __shfl_up_sync(0xFFFFFFFFu, ui, o);
                    if (tid >= o) { bi += x; ui += y; }
                }
                if (e < k) {
                    ev_out_off[e] = slots + bi - b;
                    ev_unit_off[e] = units + ui - u;
                }
                slots += __shfl_sync(0xFFFFFFFFu, bi, 31);
                units += __shfl_sync(0xFFFFFFFFu, ui, 31);
            }
            if (tid == 0) {
                ev_out_off[k] = slots;
                ev_unit_off[k] = units;
                *n_out = slots;
            }
        }
    } else {
        // Algorithm 1: key frames = the ceil(beta * len) best-scored frames of every event (ties to the
        // lower frame); a frame's stride follows from its event's and its own class; the pooled
        // frames are laid out in temporal order.
        for (int f = tid; f < Tn; f += nthr) frame_ev[f] = 0;
        __syncthreads();
        for (int e = tid; e < k; e += nthr) {
            for (int f = s_off[e]; f < s_off[e + 1]; ++f) frame_ev[f] = e;
        }
        __syncthreads();
        for (int f = tid; f < Tn; f += nthr) {
            const int e = frame_ev[f];
            const int lo = s_off[e], hi = s_off[e + 1], len = hi - lo;
            const double c = pp.beta * (double)len - 1e-9;
            long long nk = (long long)c;
            if ((double)nk < c) nk += 1;
            if (nk < 1) nk = 1;
            if (nk > len) nk = len;
            const float v = s_frame[f];
            int better = 0;
#pragma unroll 8
            for (int j = lo; j < hi; ++j) {
                const float w = s_frame[j];
                better += (w > v) || (w == v && j < f);
            }
            const bool key_frame = pp.key_frames_given ? pp.key_frames_given[f] != 0 : better < (int)nk;
            frame_stride[f] = event_is_key[e] ? (key_frame ? pp.s1 : pp.s2) : (key_frame ? pp.s1_nonkey : pp.s2_nonkey);
        }
        __syncthreads();
        // exclusive scan of the pooled sizes: contiguous ranges per thread, then a scan of the range totals
        const int per = (Tn + nthr - 1) / nthr;
        const int lo = min(Tn, tid * per), hi = min(Tn, lo + per);
        int local = 0;
        for (int f = lo; f < hi; ++f) {
            const int go = (pp.grid + frame_stride[f] - 1) / frame_stride[f];
            local += go * go;
        }
        const int lane = tid & 31, warp = tid >> 5;
        int incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_scan[warp] = incl;
        __syncthreads();
        const int wt = s_scan[lane];
        const int total = __reduce_add_sync(0xFFFFFFFFu, wt);
        int run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wt : 0) + incl - local;
        for (int f = lo; f < hi; ++f) {
            frame_off[f] = run;
            const int go = (pp.grid + frame_stride[f] - 1) / frame_stride[f];
            run += go * go;
        }
        if (tid == 0) { frame_off[Tn] = total; *n_out = total; }
    }
}

// --------------------------------------------------------------------------- //
// Adaptive pooling (Algorithm 1): an output token = one window of one frame's G x G token grid, window = stride,
// edge windows clipped to the grid.  A thread owns one 16-byte chunk of one window: the cells are added in row-major
// order in fp32, divided by their number and rounded once.  A CTA takes a share of a frame's (window, chunk) pairs, so
// the frame's stride and offset are looked up once, every load is one of consecutive 16-byte chunks, and what is in
// flight is four loads of every thread of the chip.  (A CTA per window, two rows in flight, at 128 registers: 40 us
// for 64 frames of 196 tokens of 1152; about 9 now.)
// --------------------------------------------------------------------------- //
constexpr int kPoolThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kPoolThreads)
pool_kernel(const T* __restrict__ feats, int d, int N, int G, const int32_t* __restrict__ frame_off,
            const int32_t* __restrict__ frame_stride, const int32_t* __restrict__ frame_ev, T* __restrict__ out_feats,
            int32_t* __restrict__ out_src, int32_t* __restrict__ out_event, int32_t* __restrict__ out_members,
            int32_t* __restrict__ assign) {
    grid_dep_wait();
    constexpr int VN = Vec16<T>::N;
    const int f = blockIdx.y, s = frame_stride[f], off = frame_off[f], e = frame_ev[f];
    const int go = (G + s - 1) / s, nchunk = d / VN, items = go * go * nchunk;
    const uint4* frame = reinterpret_cast<const uint4*>(feats) + (size_t)f * N * nchunk;
    for (int it = blockIdx.x * kPoolThreads + threadIdx.x; it < items; it += gridDim.x * kPoolThreads) {
        const int w = it / nchunk, c = it - w * nchunk, wy = w / go, wx = w - wy * go;
        const int r0 = wy * s, c0 = wx * s, wc = min(G, c0 + s) - c0, cells = (min(G, r0 + s) - r0) * wc;
        const int first = r0 * G + c0, o = off + w;
        float acc[VN];
        Vec16<T>::zero(acc);
        int cell = first, col = 0;                          // the next cell to load
        for (int i = 0; i < cells; i += 4) {
            uint4 raw[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                raw[u] = i + u < cells ? __ldg(frame + (size_t)cell * nchunk + c) : make_uint4(0u, 0u, 0u, 0u);
                ++cell;
                if (++col == wc) { col = 0; cell += G - wc; }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float v[VN];
                widen_chunk<T>(raw[u], v);
                if (i + u < cells) {
#pragma unroll
                    for (int q = 0; q < VN; ++q) acc[q] += v[q];
                }
            }
        }
        const float inv = 1.0f / (float)cells;
        alignas(16) T tmp[VN];
#pragma unroll
        for (int q = 0; q < VN; ++q) from_float(tmp[q], acc[q] * inv);
        reinterpret_cast<uint4*>(out_feats)[(size_t)o * nchunk + c] = *reinterpret_cast<const uint4*>(tmp);
        // the window's cells are told their output by the first of its threads
        for (int i = c; i < cells; i += nchunk) assign[(size_t)f * N + (r0 + i / wc) * G + c0 + i % wc] = o;
        if (c == 0) {
            out_src[o] = f * N + first;
            out_event[o] = e;
            out_members[o] = cells;
        }
    }
}

// --------------------------------------------------------------------------- //
// Member lists.  The kernel that chooses the key tokens starts the list of every output token with its key
// token; the merge-assign kernels add a token as soon as its output is known.  Per output: the number of members,
// the first kAvgFew of them in order of arrival, a bit per block of the event that holds a member (an output
// with more members is searched for there), and lists of the outputs with many.
// --------------------------------------------------------------------------- //
constexpr int kAvgFew = 128;       // members listed per output: 512 bytes of workspace each, whatever the output holds (see carve_vision)
constexpr int kAvgHeavy = 16;      // outputs with more members are averaged by whole CTAs,
constexpr int kAvgLong = kAvgFew;  // those with more than this in parts
struct MemberLists {
    unsigned long long* blocks;    // per output token: which blocks of its event hold a member
    int32_t* count;                // per output token: members
    int32_t* few;                  // per output token: its first kAvgFew members
    int32_t *heavy_slot, *long_slot;         // the outputs with more than kAvgHeavy (kAvgLong) members
    int32_t *heavy_counter, *long_counter;   // and how many there are
};
// An event's tokens are cut into at most 64 blocks of this many tokens.
__host__ __device__ __forceinline__ int avg_block_tokens(int m) {
    const int g = (((m + 63) / 64) + 3) & ~3;
    return g < 256 ? 256 : g;
}
// Token `row`, the i-th of its event of m tokens, is the key token of output `slot`.
__device__ __forceinline__ void members_start(const MemberLists& ml, int slot, int row, int i, int m) {
    ml.count[slot] = 1;
    ml.few[(size_t)slot * kAvgFew] = row;
    ml.blocks[slot] = 1ull << (i / avg_block_tokens(m));
}
// It joins output `slot`.  (Which place of the list or index an output gets depends on arrival order, what is computed
// from the lists does not.)
__device__ __forceinline__ void members_join(const MemberLists& ml, int slot, int row, int i, int m) {
    atomicOr(&ml.blocks[slot], 1ull << (i / avg_block_tokens(m)));
    const int pos = atomicAdd(&ml.count[slot], 1);
    if (pos < kAvgFew) ml.few[(size_t)slot * kAvgFew + pos] = row;
    if (pos == kAvgHeavy) ml.heavy_slot[atomicAdd(ml.heavy_counter, 1)] = slot;
    if (pos == kAvgLong) ml.long_slot[atomicAdd(ml.long_counter, 1)] = slot;
}
// What the kernels that choose the key tokens write per token: whether it is one, its output if so, its place in the
// list of the others if not, and the cleared scratch of its merge.
struct TokenOut {
    uint8_t* is_key;
    int32_t *out_src, *out_event, *assign;
    int32_t* rest;                 // per event, from its first token's place on: its tokens that are no key token
    unsigned long long* best64;    // packed argmax of the token's similarities
    int32_t* tile_done;            // at a row tile's first token: key chunks of the tile that are done (fp32 on the tensor cores: candidates of the token)
    unsigned long long* key_hash;  // fp32 on the tensor cores, else null: per output, hash of its key token
    MemberLists ml;
};
__device__ __forceinline__ void token_out(const TokenOut& o, int lo, int n, int i, int e, int slot0, int place, bool key) {
    o.is_key[lo + i] = key ? 1 : 0;
    o.best64[lo + i] = 0ull;
    o.tile_done[lo + i] = 0;
    if (key) {
        const int slot = slot0 + place;
        o.out_src[slot] = lo + i;
        o.out_event[slot] = e;
        o.assign[lo + i] = slot;
        if (o.key_hash) o.key_hash[slot] = 0ull;
        members_start(o.ml, slot, lo + i, i, n);
    } else {
        o.rest[lo + i - place] = lo + i;
    }
}

// Per-event key-token top-k: one cluster per event.
__global__ void __cluster_dims__(kSelCluster, 1, 1) __launch_bounds__(kSelThreads)
event_topk_kernel(const float* __restrict__ token_score, const int32_t* __restrict__ ev_lo, int N,
                  const int32_t* __restrict__ ev_budget, const int32_t* __restrict__ ev_out_off, SelectLayout lay,
                  TokenOut out) {
    grid_dep_wait();
    __shared__ SelectSmem sm;
    __shared__ int s_budget[1];
    extern __shared__ __align__(16) unsigned char sel_dyn[];
    const int e = blockIdx.x / kSelCluster;
    const int lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N;
    const int n = hi - lo;
    if (n <= 0) return;                                   // the whole cluster leaves together
    SelectCtx cx;
    cx.rank = (int)cx.cl.block_rank();
    cx.G = 1;
    cx.nb_log2 = lay.nb_log2;
    int p_lo, p_hi;
    select_slice(n, cx.rank, &p_lo, &p_hi);
    cx.item_lo = p_lo;
    cx.m = p_hi - p_lo;
    cx.cached = cx.m <= lay.cache_cap;
    cx.hist = reinterpret_cast<uint32_t*>(sel_dyn + lay.hist_off);
    cx.merged = reinterpret_cast<uint32_t*>(sel_dyn + lay.merged_off);
    cx.keys = reinterpret_cast<uint32_t*>(sel_dyn + lay.keys_off);
    cx.cls = sel_dyn + lay.cls_off;
    if (threadIdx.x == 0) s_budget[0] = ev_budget[e];
    __syncthreads();
    const float* s = token_score + lo;
    auto cls = [](int) { return 0; };
    auto val = [s](int i) { return s[i]; };
    cluster_select(cx, n, cls, val, s_budget, sm);
    const int slot0 = ev_out_off[e];
    auto flag = [&](int i) { return is_selected(sm, 0, item_at(cx, i - p_lo, cls, val).key, i); };
    auto emit = [&](int i, int rank) { token_out(out, lo, n, i, e, slot0, rank, true); };
    auto skip = [&](int i, int before) { token_out(out, lo, n, i, e, slot0, before, false); };
    cluster_compact(cx, p_lo, p_hi, flag, emit, skip, sm);
}

// The same when the largest event a segmentation can produce fits select_cluster.cuh.  It has Tn - (k - 1) frames; offsets
// with empty events can hold a longer one, which one CTA does from memory (cs_event_topk_long).
__device__ __noinline__ void cs_event_topk_long(unsigned char* dyn, const float* __restrict__ sc, int lo, int n, int e, int budget,
                                                int slot0, const TokenOut& out) {
    uint32_t* hist = reinterpret_cast<uint32_t*>(dyn);                   // [256]: the layout's two sets of buckets are at least 512 words
    uint32_t* warp_kept = hist + 256;                                    // [32]
    uint32_t* state = warp_kept + 32;                                    // the digit found, items to take inside it
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
    auto key_of = [&](int i) { return cs_key64(float_key(sc[i]), (uint32_t)i); };
    // the budget-th largest key, eight bits at a time; keys are unique
    unsigned long long thr = 0ull;
    uint32_t need = (uint32_t)budget;
    for (int shift = 56; budget < n && shift >= 0; shift -= 8) {
        for (int b = tid; b < 256; b += nthr) hist[b] = 0u;
        __syncthreads();
        for (int i = tid; i < n; i += nthr) {
            const unsigned long long key = key_of(i);
            if (((key ^ thr) >> shift) < 256ull) atomicAdd(&hist[(uint32_t)(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (tid == 0) {
            uint32_t b = 255u, left = need;
            while (b > 0u && hist[b] < left) left -= hist[b--];
            state[0] = b;
            state[1] = left;
        }
        __syncthreads();
        thr |= (unsigned long long)state[0] << shift;
        need = state[1];
    }
    uint32_t base = 0u;                                                  // kept before the round's first item
    for (int i0 = 0; i0 < n; i0 += nthr) {
        const int i = i0 + tid;
        const bool keep = i < n && key_of(i) >= thr;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
        if (lane == 0) warp_kept[warp] = (uint32_t)__popc(bal);
        __syncthreads();
        const uint32_t kept = lane < nwarps ? warp_kept[lane] : 0u;
        const uint32_t before = base + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? kept : 0u) + __popc(bal & ((1u << lane) - 1u));
        if (i < n) token_out(out, lo, n, i, e, slot0, (int)before, keep);
        base += __reduce_add_sync(0xFFFFFFFFu, kept);
        __syncthreads();
    }
}

// What a CTA reads before event_plan_kernel, the kernel before it, has completed: the caller's offsets and the token scores.
// They were complete when that kernel let this one start; its own results are read after the wait.
struct TopkEvent {
    const float* token_score;
    const int32_t *event_offsets, *ev_lo, *ev_budget, *ev_out_off;
    int Tn, N;
};

template <int IT, bool kCl>
__device__ __forceinline__ void
cs_event_topk(CsShared& sm, unsigned char* dyn, const CsLayout& lay, const TopkEvent& ev, int f_lo, int f_hi, int e, int rank, const TokenOut& out) {
    const int lo = f_lo * ev.N, n = (f_hi - f_lo) * ev.N;
    const float* sc = ev.token_score + lo;
    const CsSlice sl = cs_slice<IT>(n, rank, kCl ? kCsMaxCluster : 1);
    float score[IT];
#pragma unroll
    for (int j = 0; j < IT; ++j) score[j] = sl.i_first + 32 * j < sl.i_hi ? sc[sl.i_first + 32 * j] : 0.f;
    grid_dep_wait();
    const int budget = ev.ev_budget[e], slot0 = ev.ev_out_off[e];
    if (ev.ev_lo[e] != f_lo || ev.ev_lo[e + 1] != f_hi) {   // offsets that descend, which event_plan_kernel has raised
        const int lo2 = ev.ev_lo[e] * ev.N, n2 = ev.ev_lo[e + 1] * ev.N - lo2;
        if (rank == 0 && n2 > 0) cs_event_topk_long(dyn, ev.token_score + lo2, lo2, n2, e, budget, slot0, out);
        return;
    }
    if constexpr (kCl) cs_enter<true>();
    int before, kept;
    const uint32_t bits = cs_select<IT, kCl, true>(sm, dyn, lay, 1, &budget, rank, sl.i_first, sl.i_hi,
                                                   [&](int j, int, float& v, int& c) { v = score[j]; c = 0; }, &before, &kept);
    cs_for_items<IT>(bits, before, sl.i_first, sl.i_hi,
                     [&](int, int i, int place, bool key) { token_out(out, lo, n, i, e, slot0, place, key); });
}

constexpr int kTopkTwoThreads = 512;    // with kCsMaxItems items each; two CTAs of so many fit an SM
template <int IT, bool kCl, int kThreads>
__global__ void __launch_bounds__(kThreads, kThreads == kTopkTwoThreads ? 2 : 1)
cs_event_topk_kernel(TopkEvent ev, CsLayout lay, const __grid_constant__ TokenOut out) {
    __shared__ CsShared sm;
    extern __shared__ __align__(16) unsigned char sel_dyn[];
    constexpr int C = kCl ? kCsMaxCluster : 1;
    const int e = blockIdx.x / C, rank = blockIdx.x - e * C;
    const int f_lo = min(max(ev.event_offsets[e], 0), ev.Tn), f_hi = min(max(ev.event_offsets[e + 1], 0), ev.Tn);
    const int n = (f_hi - f_lo) * ev.N;
#define METOK_EVENT_TOPK(ITEMS, CLUSTER, RANK) cs_event_topk<ITEMS, CLUSTER>(sm, sel_dyn, lay, ev, f_lo, f_hi, e, RANK, out)
    // most events are much shorter than the longest possible one: the cluster's first CTA takes them alone
    const bool solo = !kCl || n <= min(kCsSolo, 4 * (int)blockDim.x);
    if (n <= 0 || n > IT * C * (int)blockDim.x || (solo && rank > 0)) {
        grid_dep_wait();
        const int lo = ev.ev_lo[e] * ev.N, m = ev.ev_lo[e + 1] * ev.N - lo;   // not n only where offsets descend
        if (rank == 0 && m > 0) cs_event_topk_long(sel_dyn, ev.token_score + lo, lo, m, e, ev.ev_budget[e], ev.ev_out_off[e], out);
        return;
    }
    if (solo) {
        if (IT != 8 || n <= 4 * (int)blockDim.x) METOK_EVENT_TOPK(4, false, 0);
        else METOK_EVENT_TOPK(8, false, 0);
        return;
    }
    if constexpr (kCl) {
        // (events of 18 000 in clusters of 512 threads, the call with sixteen items for all of more than four / with eight: 102.6 / 97.6 us)
        if (IT == 4 || n <= 4 * C * (int)blockDim.x) METOK_EVENT_TOPK(4, true, rank);
        else if (IT > 8 && n <= 8 * C * (int)blockDim.x) METOK_EVENT_TOPK(8, true, rank);
        else METOK_EVENT_TOPK(IT, true, rank);
    }
#undef METOK_EVENT_TOPK
}

}  // namespace metok
#include "merge_f32.cuh"
namespace metok {

// --------------------------------------------------------------------------- //
// Merge-assign on the CUDA cores (fp32 inputs; bf16 only when forced for debugging): fp32 products, added in
// the order of the row, so every dot product is one chain of fused multiply-adds.
//
// Work unit = 8 P of an event's tokens that are no key tokens x 8 P of its key tokens (P = 2 or 4: choose_simt_outputs);
// the units of all events form one list, a CTA takes its first by its number and the others from a counter; the dot
// products of a unit are SimtTile's.  Rows past a unit's end are copies of another row: nobody reads their results.
// 16 x 169 tokens in two events, d = 1156: the call takes 99 us.  Larger problems go to merge_f32.cuh.
// Units of one row meet in a 64-bit atomicMax as in the tensor-core kernel: larger value, then lower slot.
//
// kAgain: the tokens that merge_join_f32_kernel left (F3Again), none in most calls; whoever does a tile's last chunk adds its
// tokens to the member lists.
// --------------------------------------------------------------------------- //
template <typename T, int PT, bool kAgain>          // PT x PT outputs per thread
__global__ void __launch_bounds__(kSaThreads, sizeof(T) == 4 ? sa_ctas_per_sm(PT) : 4)
merge_assign_simt_kernel(const T* __restrict__ feats, int d, int N, const int32_t* __restrict__ ev_lo, int k,
                         const int32_t* __restrict__ ev_out_off, const int32_t* __restrict__ ev_unit_off,
                         const float* __restrict__ inv_norm, int32_t* __restrict__ next, TokenOut out, F3Again ag) {
    grid_dep_wait();
    const int32_t *out_src = out.out_src, *rest = out.rest;
    using Tile = SimtTile<T, PT>;
    using Count = std::conditional_t<kAgain, long long, int>;
    constexpr int kSaTile = Tile::kTile, kCopies = Tile::kCopies;
    static_assert(!kAgain || kSaTile == kF3AgainRows, "the tiles that merge_join_f32_kernel opens");
    __shared__ __align__(16) Tile tile;
    __shared__ float s_inv[kSaTile];
    __shared__ Count s_next;
    __shared__ int s_last;
    const int tid = threadIdx.x, ty = tid >> 3, tx = tid & 7;
    const unsigned long long tiles = kAgain ? *ag.tiles : 0ull;
    const Count total = kAgain ? (Count)(tiles & ((1ull << kF3UnitBits) - 1ull)) : (Count)ev_unit_off[k];
    const int row_chunks = d / Tile::CE, ksteps = Tile::steps(d);
    const uint32_t dst0 = tile.copy_dst();
    for (Count unit = blockIdx.x; unit < total; unit = s_next) {
        int e, t = 0, local;
        if constexpr (kAgain) {
            for (int n = (int)(tiles >> kF3UnitBits); n > 1;) {   // of the n tiles from t on: the last with unit0 <= unit, 32 at a time
                const int step = (n + 31) >> 5, at = (tid & 31) * step;
                const uint32_t before = __ballot_sync(0xFFFFFFFFu, at < n && ag.unit0[t + at] <= unit);
                const int skip = (31 - __clz(before)) * step;
                t += skip;
                n = min(step, n - skip);
            }
            e = ag.event[t];
            local = (int)(unit - ag.unit0[t]);
        } else {
            e = find_event(ev_unit_off, k, unit);
            local = unit - ev_unit_off[e];
        }
        const int s0 = ev_out_off[e], nk = ev_out_off[e + 1] - s0, lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N;
        const int nchunks = (nk + kSaTile - 1) / kSaTile;
        const int row_tile = kAgain ? 0 : local / nchunks, chunk = local - row_tile * nchunks;
        const int row0 = kAgain ? ag.place[t] : lo + row_tile * kSaTile;                   // places in `rest`
        const int row_end = kAgain ? min(row0 + kSaTile, lo + ag.rows[e]) : hi - nk;
        const int key0 = s0 + chunk * kSaTile, key_end = s0 + nk;
        const uint4* src[kCopies];                  // where this thread's copies of the first stage read
#pragma unroll
        for (int i = 0; i < kCopies; ++i) {
            const int r = Tile::copy_row(i);
            const int row = r < kSaTile ? rest[min(row0 + r, row_end - 1)] : out_src[min(key0 + r - kSaTile, key_end - 1)];
            src[i] = reinterpret_cast<const uint4*>(feats) + (size_t)row * row_chunks + Tile::copy_chunk();
        }
        __syncthreads();                            // the unit before is done with s_inv and both stages
        if (tid == 0) {
            s_next = total;
            if (total > (Count)gridDim.x) {
                if constexpr (kAgain) s_next = (Count)gridDim.x + (Count)atomicAdd(ag.next, 1ull);
                else s_next = (Count)gridDim.x + atomicAdd(next, 1);
            }
        }
        if (tid < kSaTile) s_inv[tid] = key0 + tid < key_end ? inv_norm[out_src[key0 + tid]] : 0.f;
        float acc[PT][PT];
        tile.dots(src, row_chunks, ksteps, dst0, acc);
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            float best_v = -3.4e38f;
            int best_s = 0x7FFFFFFF;
#pragma unroll
            for (int j = 0; j < PT; ++j) {           // ascending slots
                const int slot = key0 + tx + 8 * j;
                const float v = acc[i][j] * s_inv[tx + 8 * j];
                if (slot < key_end && v > best_v) { best_v = v; best_s = slot; }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {       // the eight column owners of the row
                const float ov = __shfl_xor_sync(0xFFFFFFFFu, best_v, o);
                const int os = __shfl_xor_sync(0xFFFFFFFFu, best_s, o);
                if (ov > best_v || (ov == best_v && os < best_s)) { best_v = ov; best_s = os; }
            }
            const int at = row0 + ty + 8 * i;
            if (tx == 0 && at < row_end && best_s != 0x7FFFFFFF)
                atomicMax(&out.best64[rest[at]], ((unsigned long long)float_key(best_v) << 32) | (unsigned long long)(~(uint32_t)best_s));
        }
        if constexpr (kAgain) {
            __threadfence();
            __syncthreads();
            if (tid == 0) s_last = atomicAdd(&ag.done[t], 1) == nchunks - 1;
            __syncthreads();
            if (s_last && row0 + tid < row_end) {
                __threadfence();
                const int row = rest[row0 + tid];
                const unsigned long long best = __ldcg(&out.best64[row]);
                f3_join(out, best ? f3_slot(best) : -1, row, lo, hi, s0, key_end);
            }
        }
    }
}

// After it, where it does all of the merge: every token that is no key token to its output.  (In the bf16 tensor-core kernel the CTA
// that does a row tile's last chunk does this; behind the chain of a unit that lengthened the launch by more than this one takes.)
__global__ void __launch_bounds__(256)
merge_join_kernel(int Nv, int N, const int32_t* __restrict__ ev_lo, int k, const int32_t* __restrict__ ev_out_off, TokenOut out) {
    grid_dep_wait();
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= Nv || out.is_key[row]) return;
    const int e = find_event(ev_lo, k, row / N);
    const int lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N, slot = (int32_t)(~(uint32_t)(out.best64[row] & 0xFFFFFFFFull));
    if (row < lo || row >= hi) return;              // a token of no event (offsets that leave frames out): its scratch is not this call's
    out.assign[row] = slot;
    if (slot >= ev_out_off[e] && slot < ev_out_off[e + 1]) members_join(out.ml, slot, row, row - lo, hi - lo);
}


// --------------------------------------------------------------------------- //
// Merge-assign on the tensor cores (bf16).
//
// Work unit = up to 256 of an event's tokens that are no key token x one chunk of the event's key tokens (up to 256
// columns; an event's keys are cut into equal chunks).  The two 128-row halves of a unit are two accumulators in TMEM
// (2 x 256 columns) that share every key tile brought into shared memory: the main loop is fed at a fixed rate per SM,
// so what counts is the work done per byte loaded -- a 256 x 256 unit needs a third fewer bytes per flop than a 128 x 256
// one.  The units of all events form one list; a persistent CTA takes every gridDim-th unit.  The
// kernel chooses the units' shape from the events' sizes (merge_launch_cost).
//   warps 9-16: producers -- both operands of a unit are rows of V scattered over the event (the key tokens and the
//              others), so the 128-byte slices of a 64-wide K step come by 16-byte asynchronous copies straight from V
//              into a ring that runs on across units, written in the 128-byte swizzle the MMA expects (eight threads per
//              row); the copies of a stage report to the stage's barrier when they have landed.  (With the token rows by
//              TMA, as boxes of consecutive rows, a fifth of the products at a keep ratio of 0.2 was spent on key tokens;
//              512 x 144 tokens of 1024 in 64 events: 138 us under ncu, 121 now);
//   warp 0   : allocates TMEM, issues tcgen05.mma (M=128, N=16..256, K=16), two per K slice (one per row half), and
//              commits to the ring / accumulator barriers;
//   warps 1-8: epilogue, four warps per accumulator -- read it with
//              tcgen05.ld, scale each column by 1/|key|, take the (value, slot) argmax of
//              the thread's row over the chunk, and add the row's token to its output's member
//              list once all chunks are known.  Units of one half take the accumulators in turn, so that the argmax of one
//              runs beside the next one's products.
// Chunks of one row tile may be handled by different CTAs: a row's result is combined
// with a 64-bit atomicMax on (order-preserving key of the value) << 32 | ~slot, which
// does not depend on the order of arrival (larger value first, then the lower slot).
// Every wait is bounded; on a timeout the CTA unwinds and writes METOK_ERR_TIMEOUT.
// --------------------------------------------------------------------------- //
constexpr int kMmaBK = 64, kMmaBN = 256, kMmaMaxStages = 6;
constexpr int kMmaThreads = 544;
constexpr int kMmaProducers = 256;                         // warps 9-16
constexpr uint32_t kMmaRingBytes = 192 * 1024;
constexpr int kMmaEvents = 512;                            // up to as many events' offsets are kept in shared memory
constexpr size_t kMmaSmemBytes = kMmaRingBytes + 1024;

// The shapes a unit may have, preferred ones first.  Large units do more per byte, but a launch lasts as long as the SM with the most
// of them, and with few events small units spread better.
constexpr int kMergeShapes = 8;
__host__ __device__ __forceinline__ MergeShape merge_shape_at(int i) {
    return {i < 5 ? 256 : 128, i < 5 ? 256 - 32 * i : i == 5 ? 256 : i == 6 ? 128 : 64};
}
__host__ __device__ __forceinline__ int merge_stages(const MergeShape& ms) {
    const int n = (int)(kMmaRingBytes / ((uint32_t)(ms.rows + ms.cols) * kMmaBK * 2));
    return n < kMmaMaxStages ? n : kMmaMaxStages;
}
// Estimated time of a unit of one or two row halves and `cols` keys, in us.  In a step of 64 elements the tensor core takes
// 0.27 ns per key and K slice of 16 for 128 rows (at least 24), the copies into the SM come at 118 KB per us, and its shared
// memory takes 128 bytes a clock (written once; 128 rows are read with all of the keys); 1.5 us for a unit's start and its argmax.
__host__ __device__ __forceinline__ float merge_unit_us(float blocks, float cols, int ksteps) {
    const float rows = 128.f * blocks + cols;
    const float mma = blocks * fmaxf(0.096f, cols * 1.09e-3f), fill = rows * (128.f / 118e3f);
    const float smem = rows * (128.f / 243e3f) + blocks * (16384.f / 243e3f + cols * (128.f / 243e3f));
    return (float)ksteps * fmaxf(mma, fmaxf(fill, smem)) + 1.5f;
}
// What a launch with one of the shapes costs, by a warp, from the events' sizes: the time it lasts, and twice the average SM's share of
// it, which is what other streams' kernels wait for.  (By the time alone, small units were taken to spread over all SMs.  70
// workloads of 4 to 512 frames, a call on its own and one of eight streams at once, relative to the time alone: with the share 1.006 and
// 0.952, with twice the share 1.004 and 0.933, with three times 1.012 and 0.914.  24 x 144 tokens of 3584 in 3 events 45.4 -> 47.4 us and
// 29.5 -> 22.1; 128 x 144 of 3584 in 16 91.5 -> 93.6 and 66.8 -> 59.6; 32 x 144 of 1024 in 4 31.6 -> 31.3 and 16.0 -> 13.2.)
constexpr float kMergeShare = 2.f / (float)kNumSMs;
__device__ __forceinline__ float merge_launch_cost(const MergeShape& ms, const int32_t* ev_lo, const int32_t* ev_out_off, int k, int N, int ksteps) {
    // (1 / 224 rounds up, and 672 keys would be four chunks: a little less gives the integer division's count up to 2.6 million keys)
    const float per_row = 1.f / (float)ms.rows, per_col = 0.9999998f / (float)ms.cols;
    float n = 0.f, all = 0.f, most = 0.f;
    for (int e = threadIdx.x & 31; e < k; e += 32) {
        const int b = ev_out_off[e + 1] - ev_out_off[e], rest = (ev_lo[e + 1] - ev_lo[e]) * N - b;
        if (rest <= 0) continue;
        const float tiles = ceilf((float)rest * per_row), chunks = ceilf((float)b * per_col);
        const float blocks = min(rest, ms.rows) > 128 ? 2.f : 1.f, cols = ceilf(__fdividef((float)b, chunks) * 0.0625f) * 16.f;
        const float us = merge_unit_us(blocks, cols, ksteps);
        n += tiles * chunks;
        all += us * (tiles * chunks);
        most = fmaxf(most, us);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n += __shfl_xor_sync(0xFFFFFFFFu, n, o);
        all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
        most = fmaxf(most, __shfl_xor_sync(0xFFFFFFFFu, most, o));
    }
    const float rounds = ceilf(n * (1.f / (float)kNumSMs));
    return (rounds <= 1.f ? most : rounds * __fdividef(all, n)) + kMergeShare * all;
}

// row_lo, row_end: the event's tokens; place0, place_end: its list of tokens that are no key token from the unit's first on;
// col0, nvalid: the unit's first key slot and its number of keys; the event's chunks and slots
struct MergeUnit { int row_lo, row_end, place0, place_end, col0, nvalid, nchunks, slot0, slot_end; };

__device__ __forceinline__ MergeUnit merge_unit(int u, const int32_t* ev_unit_off,
                                                const int32_t* ev_lo,
                                                const int32_t* ev_out_off, int k, int N, const MergeShape& ms) {
    const int e = find_event(ev_unit_off, k, u);
    const int s0 = ev_out_off[e], nk = ev_out_off[e + 1] - s0;
    const int nchunks = (nk + ms.cols - 1) / ms.cols;
    const int cols = (((nk + nchunks - 1) / nchunks) + 15) & ~15;       // equal chunks, whole MMA columns
    const int local = u - ev_unit_off[e];
    const int tile = local / nchunks, c = local - tile * nchunks;
    MergeUnit m;
    m.row_lo = ev_lo[e] * N;
    m.row_end = ev_lo[e + 1] * N;
    m.place0 = m.row_lo + tile * ms.rows;
    m.place_end = min(m.place0 + ms.rows, m.row_end - nk);
    m.col0 = s0 + c * cols;
    m.nvalid = min(cols, nk - c * cols);
    m.nchunks = nchunks;
    m.slot0 = s0;
    m.slot_end = s0 + nk;
    return m;
}

__global__ void __launch_bounds__(kMmaThreads, 1)
merge_assign_mma_kernel(const __nv_bfloat16* __restrict__ feats, int d, int N,
                        const int32_t* ev_lo, int k, const int32_t* ev_out_off,
                        const int32_t* ev_unit_off, MergeShape ms, const float* __restrict__ inv_norm,
                        TokenOut out, int32_t* __restrict__ status) {
    using namespace sm100;
    const int32_t* out_src = out.out_src;
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t full_bar[kMmaMaxStages], empty_bar[kMmaMaxStages], tfull_bar[2], tempty_bar[2], drain_bar;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort, s_last[2];
    __shared__ __align__(16) float s_keyinv[2][2][kMmaBN];    // per accumulator, alternating: a slow warp may still read the last one
    // The set-up, up to the wait, reads only what event_plan_kernel left, which was complete when the kernel after it, the choice of
    // the key tokens, let this one start.  (Tensor memory may be taken then, too: that kernel's CTAs, all of which have started,
    // need none.)
    const int ksteps = (d + kMmaBK - 1) / kMmaBK;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    // The events' offsets: every role looks a unit up, in a chain of log2(k) + 2 dependent reads that the copies of a
    // unit's first stages wait for (400 x 100 tokens of 512 in 100 events: 86.7 us the whole path with the reads from
    // global memory, 85.4 from shared memory; 127 x 174 of 1992 in 19: 193.5 and 192.6).
    // With them every CTA chooses the units' shape and counts the units, while the kernel before runs: in event_plan_kernel,
    // which everything waits for, that took 1.5 to 2 us.
    __shared__ int32_t s_off[3][kMmaEvents + 1];
    __shared__ float s_cost[kMergeShapes];
    if (k <= kMmaEvents) {
        for (int i = threadIdx.x; i <= k; i += kMmaThreads) {
            const int32_t b = ev_lo[i], c = ev_out_off[i];
            s_off[1][i] = b;
            s_off[2][i] = c;
        }
        __syncthreads();
        ev_unit_off = s_off[0];
        ev_lo = s_off[1];
        ev_out_off = s_off[2];
        if (warp < kMergeShapes) {
            const float cost = merge_launch_cost(merge_shape_at(warp), ev_lo, ev_out_off, k, N, ksteps);
            if (lane == 0) s_cost[warp] = cost;
        }
        __syncthreads();
        int best = 0;
#pragma unroll
        for (int i = 1; i < kMergeShapes; ++i)
            if (s_cost[i] < 0.97f * s_cost[best]) best = i;
        ms = merge_shape_at(best);
        if (warp == 0) {                                            // 32 events at a time
            int before = 0;
            for (int e0 = 0; e0 < k; e0 += 32) {
                const int e = e0 + lane, b = e < k ? ev_out_off[e + 1] - ev_out_off[e] : 0, rest = e < k ? (ev_lo[e + 1] - ev_lo[e]) * N - b : 0;
                const int u = (rest + ms.rows - 1) / ms.rows * ((b + ms.cols - 1) / ms.cols);
                const int incl = cs_warp_scan(u, lane);
                if (e < k) s_off[0][e] = before + incl - u;
                before += __shfl_sync(0xFFFFFFFFu, incl, 31);
            }
            if (lane == 0) s_off[0][k] = before;
        }
        __syncthreads();
    }
    const uint32_t a_bytes = (uint32_t)ms.rows * kMmaBK * 2, stage_bytes = a_bytes + (uint32_t)ms.cols * kMmaBK * 2;
    const int kMmaStages = merge_stages(ms);
    const int total_units = ev_unit_off[k];
    if ((int)blockIdx.x >= total_units) {
        grid_dep_wait();
        return;
    }
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        // a stage is full when every producer thread's copies have landed (one arrival each)
        for (int s = 0; s < kMmaStages; ++s) { mbar_init(smem_u32(&full_bar[s]), kMmaProducers); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tfull_bar[b]), 1); mbar_init(smem_u32(&tempty_bar[b]), 4); }
        mbar_init(smem_u32(&drain_bar), 1);
        s_abort = 0;
        mbar_fence_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&s_tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    grid_dep_wait();

    // Warp 0's loop runs once per K step with nothing to hide its latency: stage and phase are counted (no
    // division), addresses and descriptor words only move by adds, and the whole warp takes every step while one elected
    // thread issues, so that all of these stay in uniform registers.  (Inside a branch of lane 0 a step cost the issuing
    // thread some 1000 clocks, as long as its products: 250 for a wait that is over, 75 per product, 100 for the commit.  The
    // launch, 32 x 144 tokens of 1024 / 128 x 144 of 3584 / 512 x 144 of 1024: 20.5 / 49.5 / 138.5 us, 18.9 / 47.3 / 129.2 so.)
    const int units = __shfl_sync(0xFFFFFFFFu, total_units, 0);
    if (warp == 0) {
        int s = 0, n = 0;                                          // n: accumulators used so far
        uint32_t ph = 0;
        bool ok = true;
        const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        const uint32_t a_lo0 = desc_k128_lo(smem_base);
        const uint32_t kStageWords = stage_bytes >> 4, kBWords = a_bytes >> 4;
        constexpr uint32_t kHalfWords = (128 * kMmaBK * 2) >> 4;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const MergeUnit mu = merge_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, ms);
            const bool two = __shfl_sync(0xFFFFFFFFu, mu.place_end - mu.place0, 0) > 128;
            const uint32_t b0 = (uint32_t)n & 1u, b1 = b0 ^ 1u;
            if (!mbar_wait_warp(smem_u32(&tempty_bar[0]) + 8u * b0, ((uint32_t)(n >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            if (two && !mbar_wait_warp(smem_u32(&tempty_bar[0]) + 8u * b1, ((uint32_t)((n + 1) >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d0 = tmem + b0 * kMmaBN, d1 = tmem + b1 * kMmaBN;
            const uint32_t idesc = make_idesc_bf16(128, __shfl_sync(0xFFFFFFFFu, (mu.nvalid + 15) & ~15, 0));
            for (int ks = 0; ks < ksteps; ++ks) {
                if (!mbar_wait_warp(smem_u32(&full_bar[0]) + 8u * s, ph, abort_flag)) { ok = false; break; }
                fence_proxy_async();                             // the rows were written by ordinary (non-bulk) copies
                tc_fence_after();
                const uint32_t a_lo = a_lo0 + (uint32_t)s * kStageWords, b_lo = a_lo + kBWords;
                const uint32_t acc0 = ks != 0 ? 1u : 0u;
                if (elect_one()) {
                    if (two) {                                       // rows 128..255 of the tile: 16 KiB further on
#pragma unroll
                        for (int kk = 0; kk < kMmaBK / 16; ++kk) {
                            umma_bf16_words(d0, a_lo + 2 * kk, b_lo + 2 * kk, idesc, kk ? 1u : acc0);
                            umma_bf16_words(d1, a_lo + kHalfWords + 2 * kk, b_lo + 2 * kk, idesc, kk ? 1u : acc0);
                        }
                    } else {
#pragma unroll
                        for (int kk = 0; kk < kMmaBK / 16; ++kk)
                            umma_bf16_words(d0, a_lo + 2 * kk, b_lo + 2 * kk, idesc, kk ? 1u : acc0);
                    }
                    umma_commit(smem_u32(&empty_bar[0]) + 8u * s);   // frees the stage when these MMAs retire
                }
                __syncwarp();
                if (++s == kMmaStages) { s = 0; ph ^= 1u; }
            }
            if (ok && elect_one()) {                                // the accumulators of this unit are complete
                umma_commit(smem_u32(&tfull_bar[0]) + 8u * b0);
                if (two) umma_commit(smem_u32(&tfull_bar[0]) + 8u * b1);
            }
            __syncwarp();
            n += two ? 2 : 1;
        }
        if (!ok) {                                             // wait until whatever was issued has retired
            if (elect_one()) umma_commit(smem_u32(&drain_bar));
            __syncwarp();
            mbar_wait_warp(smem_u32(&drain_bar), 0u, abort_flag);
        }
    } else if (warp >= 9) {
        // Producers.  Thread pt copies 16-byte chunk c = pt % 8 of the rows r = pt / 8 + 32 i, i = 0..7, of the unit's tokens
        // and of its keys: eight consecutive threads read the 128 contiguous bytes of one row's K slice.  In the swizzled tile
        // row r lies at r * 128 bytes and its chunk c at position c ^ (r % 8).  Keys past the chunk's up to the next multiple
        // of 16 (the MMA's column count) are written as zeros; token rows past the unit's are not touched (what their rows of
        // the accumulator hold is not read).
        const int pt = (int)threadIdx.x - 288, c = pt & 7, rsub = pt >> 3;
        const uint32_t dst0 = smem_base + (uint32_t)rsub * 128u + (uint32_t)((c ^ (rsub & 7)) << 4);   // (r % 8) == (rsub % 8)
        const long long all = (long long)ev_lo[k] * N;
        const char* first = reinterpret_cast<const char*>(feats) + c * 16;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true, withheld = dbg_withhold(status, kDbgMergeAssign) && blockIdx.x == 0 && pt == 0;   // debug builds: one copy never reported
        for (int u = blockIdx.x; u < total_units && ok; u += gridDim.x) {
            const MergeUnit mu = merge_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, ms);
            const int rows = mu.place_end - mu.place0, npad = (mu.nvalid + 15) & ~15;
            // Where the thread's copies of the next step read.  The pointers move on after a step's copies: a copy holds its
            // address registers until it has been taken in.
            const char *row[8], *key[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = rsub + 32 * i;
                row[i] = first + (r < rows ? (size_t)dbg_bound(out.rest[mu.place0 + r], all, status) * d * 2 : 0);
                key[i] = first + (r < mu.nvalid ? (size_t)dbg_bound(out_src[mu.col0 + r], all, status) * d * 2 : 0);
            }
            for (int ks = 0; ks < ksteps; ++ks) {
                if (!mbar_wait(smem_u32(&empty_bar[0]) + 8u * s, ph ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t dst = dst0 + (uint32_t)s * stage_bytes;
                // a K slice that reaches past d (d is a multiple of 8, not of 64; the last step) reads zeros there
                const bool in_k = ks * kMmaBK + c * 8 < d;
                const uint32_t full = in_k ? 16u : 0u;
                if (!in_k) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) row[i] = key[i] = first;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (rsub + 32 * i < rows) cp_async16_zfill(dst + (uint32_t)i * 4096u, row[i], full);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = rsub + 32 * i;
                    if (r < npad) cp_async16_zfill(dst + a_bytes + (uint32_t)i * 4096u, key[i], r < mu.nvalid ? full : 0u);
                }
                if (!withheld) cp_async_arrive_noinc(smem_u32(&full_bar[0]) + 8u * s);   // arrives when this thread's copies have landed
                withheld = false;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    row[i] += kMmaBK * 2;
                    key[i] += kMmaBK * 2;
                }
                if (++s == kMmaStages) { s = 0; ph ^= 1u; }
            }
        }
        cp_async_wait_all();                                       // nothing may land after the CTA's shared memory is gone
    } else {
        const int grp = warp & 3;                                   // TMEM lanes 32*grp .. 32*grp+31
        const int buf = (warp - 1) >> 2;                            // this warp's accumulator
        const int et = ((warp - 1) & 3) * 32 + lane;                // 0..127 among the accumulator's threads
        bool ok = true;
        int n = 0, mine = 0;                                        // accumulators used so far, and of them this one
        for (int u = blockIdx.x; u < total_units; u += gridDim.x) {
            const MergeUnit mu = merge_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, ms);
            const bool two = mu.place_end - mu.place0 > 128;
            const int half = two ? (buf ^ n) & 1 : 0;               // the row half in this accumulator
            const bool has_half = two || (n & 1) == buf;
            n += two ? 2 : 1;
            if (!has_half) continue;
            const int b = mine & 1;
            const uint32_t tph = (uint32_t)mine & 1u;
            ++mine;
            for (int i = et; i < kMmaBN; i += 128) s_keyinv[buf][b][i] = i < mu.nvalid ? inv_norm[out_src[mu.col0 + i]] : 0.f;
            const int place_first = mu.place0 + half * 128, place = place_first + grp * 32 + lane;
            const bool has_row = place < mu.place_end;
            const int row = has_row ? out.rest[place] : 0;          // on its way while the products are made
            named_bar_sync(1 + buf, 128);
            if (ok && !mbar_wait(smem_u32(&tfull_bar[0]) + 8u * buf, tph, abort_flag)) ok = false;
            ok = __all_sync(0xFFFFFFFFu, ok);                      // tcgen05.ld below is warp-collective
            float best_v = -3.4e38f;
            int best_c = 0;
            if (ok) {
                tc_fence_after();
                // Row argmax.  An element costs an instruction or two: four products and their maximum, and only if
                // that beats the row's best are the four kept, so that the column is found once at the end (the
                // first column of the first group that reached the maximum, as a scan in column order finds it).
                const uint32_t t_row = tmem_base + ((uint32_t)(grp * 32) << 16) + (uint32_t)buf * kMmaBN;
                const float* keyinv = s_keyinv[buf][b];
                float b0 = 0.f, b1 = 0.f, b2 = 0.f;
                const int full = mu.nvalid & ~31;
#pragma unroll 1
                for (int c0 = 0; c0 < full; c0 += 32) {
                    uint32_t r[32];
                    tmem_ld32_issue(t_row + (uint32_t)c0, r);
                    tmem_ld32_wait(r);
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 ki = *reinterpret_cast<const float4*>(&keyinv[c0 + j]);
                        const float p0 = __uint_as_float(r[j]) * ki.x, p1 = __uint_as_float(r[j + 1]) * ki.y,
                                    p2 = __uint_as_float(r[j + 2]) * ki.z, p3 = __uint_as_float(r[j + 3]) * ki.w;
                        const float m4 = fmaxf(fmaxf(p0, p1), fmaxf(p2, p3));
                        if (m4 > best_v) { best_v = m4; best_c = c0 + j; b0 = p0; b1 = p1; b2 = p2; }
                    }
                }
                if (best_v > -3.4e38f) best_c += b0 == best_v ? 0 : b1 == best_v ? 1 : b2 == best_v ? 2 : 3;
                if (full < mu.nvalid) {
                    float v[32];
                    tmem_ld32(t_row + (uint32_t)full, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float val = v[j] * keyinv[(full + j) & (kMmaBN - 1)];
                        if (full + j < mu.nvalid && val > best_v) { best_v = val; best_c = full + j; }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[0]) + 8u * buf);
            }
            // (a warp that gave up keeps meeting the others at the named barriers)
            const bool have = ok && has_row;
            int slot = mu.col0 + best_c;
            bool last = true;
            if (mu.nchunks > 1) {
                // the chunks of a row half meet in an order-independent maximum; whoever comes last has the result
                if (have)
                    atomicMax(&out.best64[row], ((unsigned long long)float_key(best_v) << 32) | (unsigned long long)(~(uint32_t)slot));
                __threadfence();
                named_bar_sync(1 + buf, 128);
                if (et == 0) s_last[buf] = atomicAdd(&out.tile_done[place_first], 1) == mu.nchunks - 1;
                named_bar_sync(1 + buf, 128);
                last = s_last[buf];
                if (have && last) {
                    __threadfence();
                    slot = (int32_t)(~(uint32_t)(__ldcg(&out.best64[row]) & 0xFFFFFFFFull));
                }
            }
            if (have && last) {
                out.assign[row] = slot;
                // a token whose unit gave up on a wait has no maximum: it stays out of every member list (the call's
                // status word says that the results are not valid)
                if (slot >= mu.slot0 && slot < mu.slot_end) {
                    const int lo = mu.row_lo;
                    members_join(out.ml, slot, row, row - lo, mu.row_end - lo);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0 && s_abort) *status = METOK_ERR_TIMEOUT;
}

// --------------------------------------------------------------------------- //
// Averaging: a warp per (output, piece of its row).  The member rows' pieces come by 16-byte asynchronous copies into
// a ring of the warp's own, a stream that runs on from piece to piece, are added in token order in fp32, divided and
// rounded once.  No barrier wider than the warp.  What bounds it is not the memory (a warp waits for its copies a
// tenth of its time) but the fixed cost of a row and of a piece, so these are kept short and independent of each other:
// with a CTA per output, a CTA lived about 4 us for its dependent round trips (list, rows) however short the rows were,
// and 14 775 outputs of 2 KB rows shared 1184 CTA slots: 91 us between kernels of a replayed graph, 37 now; 3693 outputs
// of 7 KB rows take the 29 us they took.  The grid is what fits at once; a warp takes its first pieces by its number and
// the later ones from a counter, a piece ahead.  Rows are averaged from their last piece to their first, and outputs from
// the last down: the merge-assign pass before this one sweeps the columns of all rows together and leaves the last ones
// in L2.
//
// Outputs with many members would set the kernel's time if a warp took one late, so they come first and a CTA each: its
// warps take a quarter of the members and their sums are added in warp order.  More than kAvgLong members are not all
// listed: they are found by searching the event's blocks that hold one, in up to kAvgParts parts (a CTA each, an equal
// share of the search per warp), and the last part to finish adds the parts' sums in part order.  Such an item is a
// chain of some ten round trips, 15 to 25 us while the rest of the kernel keeps the memory busy, so its loads are
// issued together where they can be and every piece of the row is an item of its own.
// --------------------------------------------------------------------------- //
constexpr int kAvgThreads = 128;
constexpr int kAvgWarps = kAvgThreads / 32;
constexpr int kAvgCtasPerSm = 5;
constexpr int kAvgRing = 8192;         // bytes per warp
constexpr int kAvgList = 160;          // members of a long output's part listed at a time per warp: 32 kept over plus a pass of 128
constexpr int kAvgParts = 16;
constexpr int kAvgLongCapMax = 1024;   // most long outputs that get scratch for their parts' sums ...
constexpr size_t kAvgLongBytes = (size_t)32 << 20;   // ... within this much scratch
constexpr size_t kAvgSmemBytes = (size_t)kAvgWarps * kAvgRing + 128;
// long outputs that get scratch: as many as kAvgLongBytes hold (kAvgParts rows of d floats each)
__host__ __device__ inline int avg_long_cap(int d) {
    const long long c = (long long)(kAvgLongBytes / ((size_t)kAvgParts * (size_t)d * sizeof(float)));
    return (int)(c < 64 ? 64 : c > kAvgLongCapMax ? kAvgLongCapMax : c);
}
// parts of an output with `count` > kAvgLong members: about eight members per warp if they lie evenly
__host__ __device__ inline int avg_parts(int count) {
    const int p = (count + 8 * kAvgWarps - 1) / (8 * kAvgWarps);
    return p < kAvgParts ? p : kAvgParts;
}

// most pieces a row is cut into (1 KB each, of fp32 or bf16)
__host__ __device__ inline int avg_max_pieces(int d) { return (d + 255) / 256; }

struct AvgArgs {
    int d, N, Nv, nseg, seg_chunks;      // a row is cut into nseg pieces of up to seg_chunks 16-byte chunks
    const int32_t *ev_lo, *out_event, *assign;
    MemberLists ml;
    float* long_sums;
    int32_t *long_done, *next_item, *next;   // parts finished per long output and piece; the next item and piece to take
    const int32_t* n_out;
    int32_t *out_members, *status;
};

struct AvgPiece { int out, seg, n, pad; int row[kAvgHeavy]; };   // a piece of the stream: its output, piece of the row, members
constexpr int kAvgQueue = 16;            // a power of two above the R + 1 pieces that R rows can belong to

// The warp's ring of R stages, a barrier each with the parity of its next completion.
template <int R>
struct AvgRing {
    static constexpr uint32_t kStage = kAvgRing / R;
    static constexpr int kChunks = kStage / 512;             // 16-byte chunks of a row's piece per lane
    const uint8_t* mem;                  // generic address
    uint32_t mem_u32, bar_u32, phase;
    volatile int* abort_flag;
};

// Starts the copies of chunks [ch0, ch0 + nch) of V's row `row` into a stage; one arrival per lane.
template <typename T, int R>
__device__ __forceinline__ void avg_issue(AvgRing<R>& ring, int st, const T* __restrict__ feats, const AvgArgs& ar, int row,
                                          int ch0, int nch, bool withhold) {
    using namespace sm100;
    const int lane = threadIdx.x & 31;
    const uint32_t row_chunks = (uint32_t)(ar.d * (int)sizeof(T) / 16);
    const uint4* src = reinterpret_cast<const uint4*>(feats) + (size_t)dbg_bound(row, ar.Nv, ar.status) * row_chunks + ch0 + lane;
    const uint32_t dst = ring.mem_u32 + (uint32_t)st * AvgRing<R>::kStage + (uint32_t)lane * 16u;
#pragma unroll
    for (int u = 0; u < AvgRing<R>::kChunks; ++u)
        if (u * 32 + lane < nch) cp_async16_zfill(dst + u * 512u, src + u * 32, 16u);
    if (!(withhold && lane == 0)) cp_async_arrive_noinc(ring.bar_u32 + 8u * st);   // debug builds: one lane's copies never reported
}
// Waits for a stage and adds it to acc.  A lane reads only what it has copied itself.  False, for the whole warp, when a
// wait has given up: nobody may go on alone, the warp's shuffles would read lanes that have left.
template <typename T, int R>
__device__ __forceinline__ bool avg_take(AvgRing<R>& ring, int st, float (&acc)[AvgRing<R>::kChunks][16 / sizeof(T)]) {
    const int lane = threadIdx.x & 31;
    const bool ok = sm100::mbar_wait(ring.bar_u32 + 8u * st, (ring.phase >> st) & 1u, ring.abort_flag);
    ring.phase ^= 1u << st;
    if (!__all_sync(0xFFFFFFFFu, ok)) return false;
    // chunks past the piece's end add whatever the stage holds to sums that nobody stores: no branches
    const uint4* row = reinterpret_cast<const uint4*>(ring.mem + st * AvgRing<R>::kStage) + lane;
    uint4 raw[AvgRing<R>::kChunks];
#pragma unroll
    for (int u = 0; u < AvgRing<R>::kChunks; ++u) raw[u] = row[u * 32];
#pragma unroll
    for (int u = 0; u < AvgRing<R>::kChunks; ++u) {
        const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (sizeof(T) == 4) {
                acc[u][i] += __uint_as_float(w[i]);
            } else {
                acc[u][2 * i] += __uint_as_float(w[i] << 16);
                acc[u][2 * i + 1] += __uint_as_float(w[i] & 0xFFFF0000u);
            }
        }
    }
    return true;
}
// acc += all nlist rows of the list (in shared memory, the same for the whole warp), in its order.
template <typename T, int R>
__device__ __forceinline__ void avg_add_rows(AvgRing<R>& ring, const T* __restrict__ feats, const AvgArgs& ar, const int* list,
                                             int nlist, int ch0, int nch, float (&acc)[AvgRing<R>::kChunks][16 / sizeof(T)]) {
    for (int m = 0; m < nlist && m < R; ++m) avg_issue<T, R>(ring, m, feats, ar, list[m], ch0, nch, false);
    int st = 0;
    for (int m = 0; m < nlist; ++m) {
        if (!avg_take<T, R>(ring, st, acc)) break;
        if (m + R < nlist) avg_issue<T, R>(ring, st, feats, ar, list[m + R], ch0, nch, false);
        st = st + 1 == R ? 0 : st + 1;
    }
    __syncwarp();                                            // the list may be written again
}

template <typename T>
__device__ __forceinline__ void avg_store(T* out, const float* sum, float inv) {
    constexpr int VN = 16 / sizeof(T);
    alignas(16) T tmp[VN];
#pragma unroll
    for (int q = 0; q < VN; ++q) from_float(tmp[q], sum[q] * inv);
    *reinterpret_cast<uint4*>(out) = *reinterpret_cast<const uint4*>(tmp);
}

// The four warps' sums of chunks [ch0, ch0 + nch), added in warp order: handed chunk by chunk to f(chunk, sum).  They
// go through the rings' memory, into which no copy is in flight any more.
template <typename T, int CH, typename F>
__device__ __forceinline__ void avg_cta_sum(uint8_t* cta_mem, const float (&acc)[CH][16 / sizeof(T)], int nch, F f) {
    constexpr int VN = 16 / sizeof(T), kPiece = CH * 32 * VN;   // floats per warp: at most kAvgRing bytes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* sums = reinterpret_cast<float*>(cta_mem);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < CH; ++u)
#pragma unroll
        for (int q = 0; q < VN; ++q) sums[warp * kPiece + (u * 32 + lane) * VN + q] = acc[u][q];
    __syncthreads();
    for (int i = threadIdx.x; i < nch; i += kAvgThreads) {
        float t[VN];
#pragma unroll
        for (int q = 0; q < VN; ++q) {
            t[q] = sums[i * VN + q];
#pragma unroll
            for (int w = 1; w < kAvgWarps; ++w) t[q] += sums[w * kPiece + i * VN + q];
        }
        f(i, t);
    }
    __syncthreads();
}

// Output c, all of whose `count` <= kAvgFew members are listed, by the whole CTA; few: entry threadIdx.x of its list.
template <typename T, int R>
__device__ __forceinline__ void avg_heavy(AvgRing<R>& ring, const T* __restrict__ feats, T* __restrict__ out_feats, const AvgArgs& ar,
                                          int c, int count, int few, int seg, int* sorted, uint8_t* cta_mem) {
    constexpr int VN = 16 / sizeof(T), CH = AvgRing<R>::kChunks;
    const int warp = threadIdx.x >> 5;
    const int ch0 = seg * ar.seg_chunks, nch = min(ar.seg_chunks, ar.d / VN - ch0);
    // every thread ranks one member against all, every warp adds a quarter of the sorted list
    static_assert(kAvgFew == kAvgThreads, "one member per thread");
    int4* s_few = reinterpret_cast<int4*>(cta_mem);          // no copy is in flight yet
    const int tok = threadIdx.x < count ? few : 0x7FFFFFFF;  // lanes past the list hold the largest integer
    reinterpret_cast<int*>(s_few)[threadIdx.x] = tok;
    __syncthreads();
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < (count + 3) / 4; ++j) {
        const int4 x = s_few[j];
        rank += (x.x < tok) + (x.y < tok) + (x.z < tok) + (x.w < tok);
    }
    if (threadIdx.x < count) sorted[rank] = tok;
    __syncthreads();
    const int share = (count + kAvgWarps - 1) / kAvgWarps, from = min(count, warp * share), n = min(count, from + share) - from;
    float acc[CH][VN] = {};
    avg_add_rows<T, R>(ring, feats, ar, sorted + from, n, ch0, nch, acc);
    const float inv = 1.0f / (float)count;
    avg_cta_sum<T, CH>(cta_mem, acc, nch,
                            [&](int i, const float* t) { avg_store<T>(out_feats + (size_t)c * ar.d + (size_t)(ch0 + i) * VN, t, inv); });
    if (seg == 0 && threadIdx.x == 0) ar.out_members[c] = count;
}

// Part `part` of piece `seg` of output c with `count` > kAvgLong members, by the whole CTA; li: its place in the scratch of
// the parts' sums, -1: none, one part.
template <typename T, int R>
__device__ __forceinline__ void avg_long(AvgRing<R>& ring, const T* __restrict__ feats, T* __restrict__ out_feats, const AvgArgs& ar,
                                         int c, int count, int part, int nparts, int li, int seg, int* list, uint8_t* cta_mem,
                                         unsigned char* s_block, int* s_last) {
    constexpr int VN = 16 / sizeof(T), CH = AvgRing<R>::kChunks;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int e = ar.out_event[c];
    const unsigned long long blocks = ar.ml.blocks[c];
    const int lo = ar.ev_lo[e] * ar.N, hi = ar.ev_lo[e + 1] * ar.N;
    const int ch0 = seg * ar.seg_chunks, nch = min(ar.seg_chunks, ar.d / VN - ch0);
    if (tid < 64 && ((blocks >> tid) & 1ull)) s_block[__popcll(blocks & ((1ull << tid) - 1ull))] = (unsigned char)tid;
    __syncthreads();
    // the search runs over the flagged blocks' groups of four tokens (a block's first token need not start a group)
    const int bt = avg_block_tokens(hi - lo), qpb = bt / 4 + 1, total_q = __popcll(blocks) * qpb;
    const int share = (total_q + nparts * kAvgWarps - 1) / (nparts * kAvgWarps);
    const int q_begin = min(total_q, (part * kAvgWarps + warp) * share), q_end = min(total_q, q_begin + share);
    const int4* assign4 = reinterpret_cast<const int4*>(ar.assign);
    float acc[CH][VN] = {};
    int n = 0;                                               // members listed and not yet added
    for (int q0 = q_begin; q0 < q_end; q0 += 128) {
        unsigned match[4];                                   // of four rounds of 32 groups; bit i: token i of the lane's group is a member
        int first[4];
        int4 a[4];
        int j_lo[4], j_hi[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int qf = q0 + x * 32 + lane;
            a[x] = make_int4(-1, -1, -1, -1);
            first[x] = j_lo[x] = j_hi[x] = 0;
            if (qf < q_end) {
                const int bi = qf / qpb;
                j_lo[x] = lo + (int)s_block[bi] * bt;
                j_hi[x] = min(j_lo[x] + bt, hi);
                const int q = (j_lo[x] >> 2) + (qf - bi * qpb);
                first[x] = q * 4;
                if (q * 4 + 3 < ar.Nv) {
                    a[x] = assign4[q];
                } else {                                     // the array ends inside this group
                    if (q * 4 + 0 < ar.Nv) a[x].x = ar.assign[q * 4 + 0];
                    if (q * 4 + 1 < ar.Nv) a[x].y = ar.assign[q * 4 + 1];
                    if (q * 4 + 2 < ar.Nv) a[x].z = ar.assign[q * 4 + 2];
                }
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int j = first[x];
            match[x] = (unsigned)(a[x].x == c && j + 0 >= j_lo[x] && j + 0 < j_hi[x]) << 0 |
                       (unsigned)(a[x].y == c && j + 1 >= j_lo[x] && j + 1 < j_hi[x]) << 1 |
                       (unsigned)(a[x].z == c && j + 2 >= j_lo[x] && j + 2 < j_hi[x]) << 2 |
                       (unsigned)(a[x].w == c && j + 3 >= j_lo[x] && j + 3 < j_hi[x]) << 3;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int mine = __popc(match[x]);
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += v;
            }
            int r = n + incl - mine;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if ((match[x] >> i) & 1u) list[r++] = first[x] + i;
            n += __shfl_sync(0xFFFFFFFFu, incl, 31);
            __syncwarp();
            if (n > kAvgList - 128) {                        // the next round might not fit
                avg_add_rows<T, R>(ring, feats, ar, list, n, ch0, nch, acc);
                n = 0;
            }
        }
    }
    avg_add_rows<T, R>(ring, feats, ar, list, n, ch0, nch, acc);
    const float inv = 1.0f / (float)count;
    if (seg == 0 && part == 0 && tid == 0) ar.out_members[c] = count;
    if (nparts == 1) {
        avg_cta_sum<T, CH>(cta_mem, acc, nch,
                                [&](int i, const float* t) { avg_store<T>(out_feats + (size_t)c * ar.d + (size_t)(ch0 + i) * VN, t, inv); });
        return;
    }
    float* sums = ar.long_sums + (size_t)li * kAvgParts * ar.d + (size_t)ch0 * VN;
    avg_cta_sum<T, CH>(cta_mem, acc, nch, [&](int i, const float* t) {
#pragma unroll
        for (int q = 0; q < VN; q += 4)
            *reinterpret_cast<float4*>(sums + (size_t)part * ar.d + i * VN + q) = make_float4(t[q], t[q + 1], t[q + 2], t[q + 3]);
    });
    // the last part to finish adds the parts' sums in part order
    __threadfence();
    __syncthreads();
    if (tid == 0) *s_last = atomicAdd(&ar.long_done[li * ar.nseg + seg], 1) == nparts - 1;
    __syncthreads();
    if (*s_last) {
        __threadfence();
        for (int i = tid; i < nch; i += kAvgThreads) {
            float t[VN];
#pragma unroll
            for (int q = 0; q < VN; q += 4) {
                float4 v[kAvgParts];
#pragma unroll
                for (int x = 0; x < kAvgParts; ++x)
                    v[x] = x < nparts ? __ldcg(reinterpret_cast<const float4*>(sums + (size_t)x * ar.d + i * VN + q))
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
                float4 sum = v[0];
#pragma unroll
                for (int x = 1; x < kAvgParts; ++x) {
                    if (x < nparts) { sum.x += v[x].x; sum.y += v[x].y; sum.z += v[x].z; sum.w += v[x].w; }
                }
                t[q] = sum.x; t[q + 1] = sum.y; t[q + 2] = sum.z; t[q + 3] = sum.w;
            }
            avg_store<T>(out_feats + (size_t)c * ar.d + (size_t)(ch0 + i) * VN, t, inv);
        }
    }
    __syncthreads();
}

template <typename T, int R>
__global__ void __launch_bounds__(kAvgThreads, kAvgCtasPerSm)
merge_avg_kernel(const T* __restrict__ feats, T* __restrict__ out_feats, AvgArgs ar) {
    using namespace sm100;
    constexpr int VN = 16 / sizeof(T), CH = AvgRing<R>::kChunks;
    extern __shared__ uint8_t avg_dyn[];
    __shared__ __align__(8) uint64_t s_bar[kAvgWarps][R];
    __shared__ AvgPiece s_piece[kAvgWarps][kAvgQueue];
    __shared__ int s_list[kAvgWarps][kAvgList];
    __shared__ int s_abort, s_last, s_next;
    __shared__ unsigned char s_block[64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint8_t* cta_mem = avg_dyn + ((128u - (smem_u32(avg_dyn) & 127u)) & 127u);
    AvgRing<R> ring;
    ring.mem = cta_mem + warp * kAvgRing;
    ring.mem_u32 = smem_u32(ring.mem);
    ring.bar_u32 = smem_u32(&s_bar[warp][0]);
    ring.phase = 0u;
    ring.abort_flag = &s_abort;
    if (lane == 0) {
        for (int j = 0; j < R; ++j) mbar_init(ring.bar_u32 + 8u * j, 32);
        if (warp == 0) s_abort = 0;
        mbar_fence_init();
    }
    __syncthreads();
    grid_dep_wait();
    const int n_out = *ar.n_out, n_long = *ar.ml.long_counter, n_heavy = *ar.ml.heavy_counter;
    // the outputs with many members, a CTA per item: (part, output, piece), then (output, piece)
    const int per_part = n_long * ar.nseg, n_split = per_part * kAvgParts, n_items = n_split + n_heavy * ar.nseg;
    bool stop = false;                                       // a wait has given up: the same for the whole CTA
    for (int it = (int)blockIdx.x; it < n_items && !stop;) {
        if (tid == 0) s_next = n_items > (int)gridDim.x ? (int)gridDim.x + atomicAdd(ar.next_item, 1) : n_items;
        if (it < n_split) {
            const int part = it / per_part, sub = it - part * per_part, back = sub / n_long, li = sub - back * n_long;
            const int c = ar.ml.long_slot[li], count = ar.ml.count[c];
            const bool scratch = li < avg_long_cap(ar.d);
            const int nparts = scratch ? avg_parts(count) : 1;
            if (part < nparts)
                avg_long<T, R>(ring, feats, out_feats, ar, c, count, part, nparts, scratch ? li : -1, ar.nseg - 1 - back, s_list[warp],
                                 cta_mem, s_block, &s_last);
        } else {
            const int x = it - n_split, back = x / n_heavy, h = x - back * n_heavy;
            const int c = ar.ml.heavy_slot[h], count = ar.ml.count[c], few = ar.ml.few[(size_t)c * kAvgFew + tid];
            if (count <= kAvgLong) avg_heavy<T, R>(ring, feats, out_feats, ar, c, count, few, ar.nseg - 1 - back, &s_list[0][0], cta_mem);
        }
        __syncthreads();
        it = s_next;
        stop = s_abort != 0;                                 // nobody waits for copies between these two barriers
        __syncthreads();
    }
    // The others, a warp per piece: the last piece of every row first, then the one before it and so on (see above), from
    // the last output down.  A stream of rows that runs on from piece to piece: R of them are on their way while one is added, whichever
    // piece they belong to; the list of the piece after the one being issued has been fetched, and the number of the
    // one after that.  Pieces being issued or added stand in a queue in shared memory.
    const int total = n_out * ar.nseg, nchunk = ar.d / VN;
    AvgPiece* queue = s_piece[warp];
    int a_out = 0, a_seg = 0, a_n = -1, a_tok = 0;           // the piece ahead: n = 0: taken elsewhere, -1: no more pieces
    auto fetch = [&](int t) {
        a_n = -1;
        if (t < total) {
            const int back = t / n_out;
            a_seg = ar.nseg - 1 - back;
            a_out = n_out - 1 - (t - back * n_out);
            a_tok = lane < kAvgHeavy ? ar.ml.few[(size_t)a_out * kAvgFew + lane] : 0;
            a_n = ar.ml.count[a_out];
            if (a_n > kAvgHeavy) a_n = 0;
        }
    };
    // A warp's first two pieces are fixed: all warps at one counter at once would stand in line for 5 us.  A CTA that had
    // an item comes late: unless there are pieces enough for everybody, its warps take what is left, or their fixed pieces
    // would be the last to be done (4009 outputs of 208 bytes, 72 of them such items: 22 -> 16 us; with five pieces a
    // warp the two round trips to the counter cost 1 us).
    const int n_busy = total < 4 * (int)gridDim.x * kAvgWarps ? min(n_items, (int)gridDim.x) : 0, warps = ((int)gridDim.x - n_busy) * kAvgWarps;
    auto take = [&](int n) { return lane == 0 ? 2 * warps + atomicAdd(ar.next, n) : 0; };
    int ticket;
    if ((int)blockIdx.x >= n_busy) {
        const int me = ((int)blockIdx.x - n_busy) * kAvgWarps + warp;
        fetch(me);
        ticket = me + warps;
    } else {
        ticket = __shfl_sync(0xFFFFFFFFu, take(2), 0);
        fetch(ticket++);
    }
    bool withhold = dbg_withhold(ar.status, kDbgMergeAvg);   // debug builds: of every warp's first row
    int i_piece = -1, i_n = 0, i_at = 0, i_ch0 = 0, i_nch = 0;   // issued: rows [0, i_at) of piece i_piece of the stream
    auto issue_next = [&](int st) {                          // the next row of the stream; false: there is none
        if (i_at == i_n) {
            while (a_n == 0) {
                fetch(__shfl_sync(0xFFFFFFFFu, ticket, 0));
                ticket = take(1);
            }
            if (a_n < 0) return false;
            // the members into token order: rank = members before it
            AvgPiece& q = queue[++i_piece & (kAvgQueue - 1)];
            const int key = lane < a_n ? a_tok : 0x7FFFFFFF;
            int rank = 0;
            for (int j = 0; j < a_n; j += 4) {               // four at a time: lanes past the list hold the largest integer
#pragma unroll
                for (int x = 0; x < 4; ++x) rank += __shfl_sync(0xFFFFFFFFu, key, j + x) < key;
            }
            if (lane < a_n) q.row[rank] = key;
            if (lane == 0) { q.out = a_out; q.seg = a_seg; q.n = a_n; }
            __syncwarp();
            i_n = a_n;
            i_at = 0;
            i_ch0 = a_seg * ar.seg_chunks;
            i_nch = min(ar.seg_chunks, nchunk - i_ch0);
            fetch(__shfl_sync(0xFFFFFFFFu, ticket, 0));
            ticket = take(1);
        }
        avg_issue<T, R>(ring, st, feats, ar, queue[i_piece & (kAvgQueue - 1)].row[i_at], i_ch0, i_nch, withhold);
        withhold = false;
        ++i_at;
        return true;
    };
    int flying = 0;
    if (!stop)
        for (int m = 0; m < R; ++m) flying += issue_next(m) ? 1 : 0;
    int st = 0;
    for (int piece = 0; flying > 0; ++piece) {
        const AvgPiece& q = queue[piece & (kAvgQueue - 1)];
        const int out = q.out, seg = q.seg, n = q.n, ch0 = seg * ar.seg_chunks, nch = min(ar.seg_chunks, nchunk - ch0);
        float acc[CH][VN] = {};
        bool ok = true;                                      // the same for the whole warp
        for (int m = 0; m < n && ok; ++m) {
            ok = avg_take<T, R>(ring, st, acc);
            if (ok && !issue_next(st)) --flying;
            st = st + 1 == R ? 0 : st + 1;
        }
        if (!ok) break;
        const float inv = 1.0f / (float)n;
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const int ch = u * 32 + lane;
            if (ch < nch) avg_store<T>(out_feats + (size_t)out * ar.d + (size_t)(ch0 + ch) * VN, acc[u], inv);
        }
        if (seg == 0 && lane == 0) ar.out_members[out] = n;
    }
    cp_async_wait_all();                                     // nothing may land after the CTA's shared memory is gone
    if (lane == 0 && s_abort) *ar.status = METOK_ERR_TIMEOUT;
}

// --------------------------------------------------------------------------- //
// host side
// --------------------------------------------------------------------------- //
struct VisionWs {
    int32_t* status;          // device status word, first in the workspace
    float* inv_norm;
    int32_t *ev_lo, *ev_budget, *ev_out_off, *ev_unit_off;
    int32_t *frame_ev, *frame_stride, *frame_off;   // POOL mode
    uint8_t* is_key;          // the rest: merging modes (TokenOut, MemberLists, AvgArgs)
    int32_t *rest, *tile_done;
    unsigned long long* best64;
    MemberLists ml;
    float* long_sums;
    F3Planes planes;          // fp32 merge on the tensor cores; so are the candidates' lists and the hashes
    unsigned long long* cands;
    unsigned long long* key_hash;
    F3Again again;
    int32_t *suspects, *n_suspects;
    int32_t *long_done, *avg_next, *unit_next;
    int n_counters;           // the counters are cleared together: long, heavy, avg_next, unit_next and long_done, again's tiles and next, n_suspects, again's rows
};

static VisionWs carve_vision(Carver& cv, int Tn, int N, int k, int d, int cap, bool merging, bool planes) {
    VisionWs w = {};
    w.status = cv.take<int32_t>(64);
    w.inv_norm = cv.take<float>((size_t)Tn * N);
    w.ev_lo = cv.take<int32_t>((size_t)k + 1);
    w.ev_budget = cv.take<int32_t>((size_t)k + 1);
    w.ev_out_off = cv.take<int32_t>((size_t)k + 1);
    w.ev_unit_off = cv.take<int32_t>((size_t)k + 1);
    w.frame_ev = cv.take<int32_t>((size_t)Tn);
    w.frame_stride = cv.take<int32_t>((size_t)Tn);
    w.frame_off = cv.take<int32_t>((size_t)Tn + 1);
    if (merging) {
        // 528 bytes per output, most of it the member list, beside rows of usually 2 KB and more: 7.5 MB for 512 frames of
        // 144 tokens of which a fifth is kept, 300 MB for 8192 frames of which half is
        const size_t n = (size_t)cap + 64;
        w.is_key = cv.take<uint8_t>((size_t)Tn * N);
        w.rest = cv.take<int32_t>((size_t)Tn * N);
        w.tile_done = cv.take<int32_t>((size_t)Tn * N);
        w.best64 = cv.take<unsigned long long>((size_t)Tn * N);
        w.ml.blocks = cv.take<unsigned long long>(n);
        w.ml.count = cv.take<int32_t>(n);
        w.ml.few = cv.take<int32_t>(n * kAvgFew);
        w.ml.heavy_slot = cv.take<int32_t>(n);
        w.ml.long_slot = cv.take<int32_t>(n);
        const int n_avg = 5 + avg_long_cap(d) * avg_max_pieces(d), n_again = (n_avg + 1) & ~1;
        w.n_counters = planes ? n_again + 5 + k : n_avg;
        w.ml.long_counter = cv.take<int32_t>((size_t)w.n_counters);
        w.ml.heavy_counter = w.ml.long_counter + 1;
        w.avg_next = w.ml.long_counter + 2;              // two: items, pieces
        w.unit_next = w.ml.long_counter + 4;
        w.long_done = w.ml.long_counter + 5;
        w.long_sums = cv.take<float>((size_t)avg_long_cap(d) * kAvgParts * d);
        if (planes) {
            w.planes.a = cv.take<uint8_t>(f3_a_bytes((long long)Tn * N, k, d));
            w.planes.b = cv.take<uint8_t>(f3_b_bytes(cap, k, d));
            w.cands = cv.take<unsigned long long>((size_t)Tn * N * (kF3Cands + 1));
            w.key_hash = cv.take<unsigned long long>(n);
            const size_t tiles = f3_again_tiles((long long)Tn * N, k);
            w.again.unit0 = cv.take<long long>(tiles);
            w.again.event = cv.take<int32_t>(tiles);
            w.again.place = cv.take<int32_t>(tiles);
            w.again.done = cv.take<int32_t>(tiles);
            w.again.tiles = reinterpret_cast<unsigned long long*>(w.ml.long_counter + n_again);
            w.again.next = w.again.tiles + 1;
            w.n_suspects = w.ml.long_counter + n_again + 4;
            w.again.rows = w.n_suspects + 1;
            w.suspects = cv.take<int32_t>((size_t)Tn * N);
        }
    }
    return w;
}

// The shape of the units where there are more events than the merge's own choice holds.  The lengths are on the device: the estimate is
// for events of half the mean length, the mean and one and a half times it.  Shapes within 3 % of the best are told apart by the bytes
// that the ring has in flight, in the units of the mean event.  Events x tokens of each x width, keep, the call with units of 256 x 128
// whatever the events are / so: 513 x 2160 x 256, 0.1 1043 / 857 us, 0.3 1618 / 1255; 520 x 1568 x 512, 0.1 942 / 813, 0.3 1384 / 1207;
// 520 x 576 x 512, 0.3 662 / 629; 600 x 288 x 3584, 0.1 771 / 772, 0.5 1203 / 1167; 600 x 64 x 1024, 0.1 76.7 / 77.1;
// 2000 x 144 x 1024, 0.3 439 / 439.
static MergeShape choose_merge_shape(int Nv, int k, int d, double keep) {
    const int ksteps = ceil_div(d, kMmaBK);
    float us[kMergeShapes], best_us = 0.f;
    int flight[kMergeShapes];
    for (int i = 0; i < kMergeShapes; ++i) {
        const MergeShape ms = merge_shape_at(i);
        us[i] = 0.f;
        for (int half = 1; half <= 3; ++half) {
            const int m = std::max(2, (int)((long long)Nv * half / (2LL * k))), keys = std::min(m - 1, std::max(1, (int)(keep * m + 0.5))), rest = m - keys;
            const int chunks = ceil_div(keys, ms.cols), cols = ceil_div(keys, 16 * chunks) * 16;
            us[i] += (float)(ceil_div(rest, ms.rows) * chunks) * merge_unit_us(std::min(rest, ms.rows) > 128 ? 2.f : 1.f, (float)cols, ksteps);
            if (half == 2) flight[i] = merge_stages(ms) * (std::min(rest, ms.rows) + cols);
        }
        if (i == 0 || us[i] < best_us) best_us = us[i];
    }
    int best = -1;
    for (int i = 0; i < kMergeShapes; ++i)
        if (us[i] <= 1.03f * best_us && (best < 0 || flight[i] > flight[best])) best = i;
    return merge_shape_at(best);
}

// CTAs of the merge: no more than there can be units of the smallest shape where no event is empty (with more units a CTA takes several).
// A CTA has an SM to itself and chooses the shape and counts the units before it knows whether it has one, so that in small calls
// idle CTAs kept other streams from the SMs.  With 148 CTAs always / so, a call of eight streams at once and on its own: 9 frames x 39
// tokens 4.5 -> 3.2 us, 18.8 -> 19.1; 32 x 21 in 11 events 5.0 -> 3.7, 19.7 -> 20.2; 6 x 147 x 1096 7.3 -> 5.9, 26.8 -> 26.9.
static int merge_ctas(int Tn, int N, int k, const metok_vision_params* p) {
    const double keep = std::max(p->keep_key, p->keep_nonkey), Nv = (double)Tn * N, longest = (double)(Tn - (k - 1)) * N;
    // sum of ceil(x) ceil(y) <= sum of x y + x + y + 1, x = tokens / 128, y = keys / 64
    const double tiles = Nv / 128, chunks = (keep * Nv + k) / 64, both = tiles * (keep * longest + 1) / 64;
    return (int)std::min<double>(kNumSMs, both + tiles + chunks + k + 1);
}

// The tensor-core merge path needs bf16 rows of whole 16-byte pieces;
// METOK_DEBUG_FORCE_SIMT=1 in the environment selects the CUDA-core kernels (debugging aid).
static bool force_simt() {
    static const bool force = [] { const char* e = getenv("METOK_DEBUG_FORCE_SIMT"); return e && e[0] == '1'; }();
    return force;
}
static bool use_mma_path(int d) { return !force_simt() && d % 8 == 0; }

// Outputs per thread (a side of the square) of the CUDA-core kernel, from the number of 64 x 64 units of the mean event.
// Few of them leave SMs idle and last as long as one unit's chain of d steps: 16 x 16 units are then the fastest.  The whole
// call with 16 x 16 / 32 x 32, at that many units: 169 tokens of 1156, 34 units 42 / 48 us, 57: 51 / 49, 103: 82 / 70; 100 tokens
// of 512, 36: 29 / 32, 75: 39 / 42, 98: 48 / 44.  Units of 64 x 64 wherever 740 to 888 of them fill a round of CTAs, in a launch of
// their own that finds none elsewhere, matter only for rows so narrow that fp32 stays here however many units there are; the call
// with that launch / without: rows of 20 floats, 612 such units 39.0 / 37.0 us, 735: 41.0 / 39.0; of 56, 740: 43.3 / 43.0, 888: 46.4 /
// 49.2, 891: 50.7 / 49.2; of 32, 888: 39.8 / 41.2.  So there is none.
static int choose_simt_outputs(int Nv, int k, double keep) {
    const double m = (double)Nv / k, keys = std::max(1.0, keep * m), units = ((m - keys) / 64 + 0.5) * (keys / 64 + 0.5) * k;
    return units < kNumSMs / 2 ? 2 : 4;
}

// The fp32 merge: on the tensor cores (keys per unit; see merge_f32.cuh) or 0, on the CUDA cores.  Both times are estimated for
// the mean event.  Tensor cores: the planes read and written at 5.2 TB/s, then rounds of units, a step of which takes what its
// tensor instructions or its shared-memory traffic take, then the chains of the near ties; the events' lengths are not known
// here, so that units are counted as 1.3 times the estimate where fewer keys per unit would just fit a round.  CUDA cores: 64 us
// per 10^9 multiply-adds (and 3 us in favour of what needs no planes).  The whole call on the CUDA cores / on the tensor cores,
// frames x tokens x width in events, keep: 24 x 100 x 512 in 3, 0.3: 56 / 58 us; 40 x 100 x 512 in 4: 67 / 61; 64 x 100 x 512 in 7: 104 / 66;
// 20 x 64 x 2048 in 2: 80 / 95; 50 x 64 x 2048 in 4: 140 / 122; 14 x 144 x 3584 in 2, 0.2: 174 / 175; 20 x 144 x 3584 in 2: 225 / 183;
// 128 x 64 x 128 in 6: 61 / 54; 61 x 169 x 1156 in 7, 0.25: 265 / 133.
// The planes take one and a half times the memory of the features, and the share of the key tokens as much again, so beyond kF3MaxBytes
// the CUDA cores do it.
constexpr size_t kF3MaxBytes = (size_t)1 << 30;
static bool f3_fits(long long Nv, int k, int d, int cap) {
    return d >= kF3MinD && f3_a_bytes(Nv, k, d) + f3_b_bytes(cap, k, d) <= kF3MaxBytes;
}
static int choose_f3(int Nv, int k, int d, int cap, double keep) {
    if (!f3_fits(Nv, k, d, cap)) return 0;
    const double m = (double)Nv / k, keys = std::max(1.0, keep * m), rest = m - keys;
    double best = 0.0;
    int best_bn = 0;
    for (const int bn : {256, 128, 64}) {
        const double units = k * (rest / kF3BM + 0.5) * (keys / bn + 0.5) * (bn < 256 ? 1.3 : 1.0);
        const double cols = std::min(256.0, std::ceil(keys / std::ceil(keys / bn) / 16) * 16);
        const double mma = 12 * std::max(0.024, cols * 0.272e-3), smem = ((kF3BM + cols) * kF3RowBytes + 12 * (4096 + 32 * cols)) / 243e3;
        const double us = std::ceil(units / kNumSMs) * (f3_steps(d) * std::max(mma, smem) + 3.0);
        if (!best_bn || us < 0.9 * best) { best_bn = bn; best = us; }
    }
    best += 11.0 + 0.004 * d + (double)Nv * d * 10.0 / 5.2e6;
    return best < 3.0 + 64e-9 * k * rest * keys * d ? best_bn : 0;
}

static bool ratio_ok(double r) { return r > 0.0 && r <= 1.0; }

static size_t vision_ws_bytes(int Tn, int N, int k, int d, int cap, bool merging, bool planes) {
    Carver cv(nullptr);
    carve_vision(cv, Tn, N, k, d, cap, merging, planes);
    return cv.total();
}

template <typename T>
static int launch_vision(const void* feats_, int Tn, int N, int d, const int32_t* event_offsets, int k,
                         const void* text_, const metok_vision_params* p, void* out_feats_, int32_t* out_src,
                         int32_t* out_event, int32_t* out_members, int32_t* assign, float* token_score,
                         float* frame_score, float* event_score, uint8_t* event_is_key, int32_t* n_out, int cap,
                         void* ws, size_t ws_bytes, cudaStream_t st) {
    const T* feats = reinterpret_cast<const T*>(feats_);
    const T* text = reinterpret_cast<const T*>(text_);
    T* out_feats = reinterpret_cast<T*>(out_feats_);
    const int Nv = Tn * N;
    constexpr bool kBf16 = sizeof(T) == 2;
    const bool mma = kBf16 && use_mma_path(d) && p->mode == METOK_MODE_TOPK_MERGE;
    Carver cv(ws);
    const double keep = p->alpha * p->keep_key + (1.0 - p->alpha) * p->keep_nonkey;
    int f3_bn = kBf16 || p->mode != METOK_MODE_TOPK_MERGE || force_simt() ? 0 : choose_f3(Nv, k, d, cap, keep);
    // a workspace sized for other ratios, for which there were no planes: the CUDA cores do it (with the same assignment as far as f3_margin holds)
    if (f3_bn && ws_bytes < vision_ws_bytes(Tn, N, k, d, cap, true, true)) f3_bn = 0;
    VisionWs w = carve_vision(cv, Tn, N, k, d, cap, p->mode == METOK_MODE_TOPK_MERGE, f3_bn > 0);
    // (the status word and the scratch that must start cleared are written by event_plan_kernel)
    if (const int rc = debug_arm(w.status, st)) return rc;

    // Eq. 5 per token, unless the caller brings the scores and norms from metok_segment_score_events
    const float* inv_norm = p->token_inv_norm ? p->token_inv_norm : w.inv_norm;
    if (!p->token_inv_norm) {
        {
            METOK_TIMED("tok_score_kernel", st);
            launch_chained(tok_score_kernel<T>, dim3(min(ceil_div(Nv, 8), kNumSMs * 32)), dim3(256), 0, st, feats, text, Nv, d,
                           token_score, w.inv_norm);
        }
        METOK_LAUNCH_CHECK();
    }
    const int simt = choose_simt_outputs(Nv, k, keep);
    PlanParams pp;
    pp.Tn = Tn; pp.N = N; pp.k = k;
    pp.n_key_events = min(k, ceilq(p->alpha * (double)k));
    pp.event_agg = p->event_agg; pp.mode = p->mode;
    if (mma) pp.shape = k > kMmaEvents ? choose_merge_shape(Nv, k, d, keep) : MergeShape{256, 128};
    else pp.shape = f3_bn ? MergeShape{kF3BM, f3_bn} : MergeShape{8 * simt, 8 * simt};
    pp.keep_key = p->keep_key; pp.keep_nonkey = p->keep_nonkey; pp.beta = p->beta;
    pp.key_given = p->key_events_given;
    pp.key_frames_given = p->key_frames_given;
    pp.grid = 1;
    while (pp.grid * pp.grid < N) ++pp.grid;
    pp.s1 = p->s1; pp.s2 = p->s2; pp.s1_nonkey = p->s1_nonkey; pp.s2_nonkey = p->s2_nonkey;
    const size_t plan_smem = (size_t)(k + Tn) * sizeof(float) + (size_t)k * (3 * sizeof(int) + 1) + sizeof(int);
    // more CTAs than one as soon as one would need more than two rounds for the frames
    const int plan_ctas = Tn <= 256 ? 1 : Tn <= 512 ? 4 : 8;
    if (plan_smem > 40 * 1024)
        METOK_ALLOW_SMEM(event_plan_kernel, plan_smem);
    {
        METOK_TIMED("event_plan_kernel", st);
        launch_chained_clusters(plan_ctas, event_plan_kernel, dim3(plan_ctas), dim3(1024), plan_smem, st, token_score, frame_score, event_offsets, pp, event_score,
                       event_is_key, w.ev_lo, w.ev_budget, w.ev_out_off, w.ev_unit_off, w.frame_ev, w.frame_stride, w.frame_off,
                       n_out, w.ml.long_counter, w.n_counters, w.status);
    }
    METOK_LAUNCH_CHECK();

    if (p->mode == METOK_MODE_POOL) {
        {
            METOK_TIMED("pool_kernel", st);
            // about sixteen CTAs per SM, but no more per frame than its largest number of pairs fills
            const int smin = std::min(std::min(p->s1, p->s2), std::min(p->s1_nonkey, p->s2_nonkey));
            const int side = ceil_div(pp.grid, smin);
            const int most = (int)std::min<long long>(ceil_div(kNumSMs * 16, Tn),
                                                      ((long long)side * side * (d * (int)sizeof(T) / 16) + kPoolThreads - 1) / kPoolThreads);
            launch_chained(pool_kernel<T>, dim3(std::max(1, most), Tn), dim3(kPoolThreads), 0, st, feats, d, N, pp.grid, w.frame_off,
                           w.frame_stride, w.frame_ev, out_feats, out_src, out_event, out_members, assign);
        }
        METOK_LAUNCH_CHECK();
        return METOK_OK;
    }

    const TokenOut to = {w.is_key, out_src, out_event, assign, w.rest, w.best64, w.tile_done, w.key_hash, w.ml};
    const F3Cands cands = {w.cands, w.tile_done, w.key_hash, w.suspects, w.n_suspects};
    {
        // an event has at most Tn - (k - 1) frames if none is empty; cs_event_topk_long takes one that has more
        const long long longest = (long long)(Tn - (k - 1)) * N;
        const CsPlan plan = cs_plan(longest);
        // Between event_plan_kernel and the merge nothing may be launched that writes scores or offsets, or that takes tensor memory:
        // cs_event_topk_kernel reads the former, and merge_assign_mma_kernel event_plan_kernel's offsets, before their waits.
        if (plan.fits) {
            const CsLayout lay = cs_layout(1, std::max(Nv / k, 2048));          // buckets for the mean event
            const TopkEvent ev = {token_score, event_offsets, w.ev_lo, w.ev_budget, w.ev_out_off, Tn, N};
            METOK_TIMED("event_topk_kernel", st);
            auto launch = [&](auto kernel, int C, int threads) {
                launch_chained_clusters(C, kernel, dim3(k * C), dim3(threads), lay.bytes, st, ev, lay, to);
            };
            // One CTA per event where that holds the longest one there can be.  Clusters, most of which come down to
            // their first CTA, cost nothing while all of them are resident at once; with more events (61 of them: 488
            // CTAs of 1024 threads, 9 us against 6) a CTA with eight items per thread is preferred as long as it can.
            if (plan.C == 1) launch(cs_event_topk_kernel<4, false, 1024>, 1, plan.threads);
            else if (longest <= 2 * kCsSolo && k * plan.C > kNumSMs) launch(cs_event_topk_kernel<8, false, 1024>, 1, 1024);
            else if (plan.items == 4) launch(cs_event_topk_kernel<4, true, 1024>, plan.C, kCsSolo / 4);
            // With so many registers a CTA has an SM to itself, and the clusters of more than some fifteen events (a cluster's CTAs
            // lie in one group of SMs) take several rounds; up to 65 536 tokens in the longest event the registers of two CTAs per SM
            // do.  One per SM / two, frames x tokens of 8, the call: 200 x 196 in 2 events 125.7 / 134.5 us, 512 x 120 in 12
            // 77.5 / 77.4, in 15 75.1 / 75.3, in 16 72.2 / 66.1, in 48 53.5 / 50.2; 512 x 144 of 1024 in 64 the path 218.4 / 217.1.
            else if (k * plan.C > kNumSMs * 2 / 3 && longest <= (long long)kCsMaxItems * kCsMaxCluster * kTopkTwoThreads)
                launch(cs_event_topk_kernel<kCsMaxItems, true, kTopkTwoThreads>, plan.C, kTopkTwoThreads);
            else launch(cs_event_topk_kernel<kCsMaxItems, true, kCsMaxItemsThreads>, plan.C, kCsMaxItemsThreads);
        } else {
            // the cache is sized for the longest event there can be, the thread count for twice the mean
            const SelectLayout lay = select_layout(1, select_items_per_cta((long long)(Tn - (k - 1)) * N));
            const int nthreads = select_threads(select_items_per_cta(2LL * Nv / k));
            if (lay.bytes > 32 * 1024)                    // static + dynamic beyond 48 KiB needs the opt-in
                METOK_ALLOW_SMEM(event_topk_kernel, lay.bytes);
            METOK_TIMED("event_topk_kernel", st);
            launch_chained(event_topk_kernel, dim3(k * kSelCluster), dim3(nthreads), lay.bytes, st,
                token_score, w.ev_lo, N, w.ev_budget, w.ev_out_off, lay, to);
        }
        METOK_LAUNCH_CHECK();
    }

    if (mma) {
        METOK_ALLOW_SMEM(merge_assign_mma_kernel, kMmaSmemBytes);
        {
            METOK_TIMED("merge_assign_mma_kernel", st);
            launch_chained(merge_assign_mma_kernel, dim3(merge_ctas(Tn, N, k, p)), dim3(kMmaThreads), kMmaSmemBytes, st,
                reinterpret_cast<const __nv_bfloat16*>(feats), d, N, w.ev_lo, k, w.ev_out_off, w.ev_unit_off, pp.shape, inv_norm,
                to, w.status);
        }
        METOK_LAUNCH_CHECK();
    } else {
        if constexpr (!kBf16) {
            if (f3_bn) {
                // the planes: about eight CTAs per SM, rows in shares of their steps where there are few
                const int steps = f3_steps(d), shares = std::min(steps, std::max(1, kNumSMs * 8 * 32 / Nv)), per = ceil_div(steps, shares);
                {
                    METOK_TIMED("merge_planes_kernel", st);
                    launch_chained(merge_planes_kernel, dim3(ceil_div(Nv, 32), ceil_div(steps, per)), dim3(256), 0, st, feats, Nv, d, N,
                                   w.ev_lo, k, w.ev_out_off, inv_norm, to, w.planes, cands, f3_bn, per, w.status);
                }
                METOK_LAUNCH_CHECK();
                METOK_ALLOW_SMEM(merge_assign_f32_mma_kernel, kF3SmemBytes);
                {
                    METOK_TIMED("merge_assign_f32_mma_kernel", st);
                    launch_chained(merge_assign_f32_mma_kernel, dim3(kNumSMs), dim3(kF3Threads), kF3SmemBytes, st, d, N, w.ev_lo, k,
                                   w.ev_out_off, w.ev_unit_off, inv_norm, to, w.planes, cands, f3_bn, w.status);
                }
                METOK_LAUNCH_CHECK();
                {
                    METOK_TIMED("merge_join_f32_kernel", st);
                    const int per = kF3JoinWarps * 32, suspect_ctas = std::min(kNumSMs * 4, ceil_div(Nv, kF3JoinWarps));
                    launch_chained(merge_join_f32_kernel, dim3(suspect_ctas + ceil_div(Nv, per)), dim3(per), 0, st, feats, Nv, d, N, w.ev_lo, k,
                                   w.ev_out_off, inv_norm, to, cands, w.again, suspect_ctas);
                }
                METOK_LAUNCH_CHECK();
                {
                    METOK_TIMED("merge_again_kernel", st);
                    launch_chained(merge_assign_simt_kernel<float, 4, true>, dim3(kNumSMs * sa_ctas_per_sm(4)), dim3(kSaThreads), 0, st, feats,
                                   d, N, w.ev_lo, k, w.ev_out_off, w.ev_unit_off, inv_norm, w.unit_next, to, w.again);
                }
                METOK_LAUNCH_CHECK();
            }
        }
        if (!f3_bn) {
            {
                METOK_TIMED("merge_assign_simt_kernel", st);
                auto assign_units = [&](auto kernel) {
                    launch_chained(kernel, dim3(kNumSMs * sa_ctas_per_sm(simt)), dim3(kSaThreads), 0, st, feats, d, N, w.ev_lo, k,
                                   w.ev_out_off, w.ev_unit_off, inv_norm, w.unit_next, to, w.again);
                };
                if (simt == 2) assign_units(merge_assign_simt_kernel<T, 2, false>);
                else assign_units(merge_assign_simt_kernel<T, 4, false>);
            }
            METOK_LAUNCH_CHECK();
            {
                METOK_TIMED("merge_join_kernel", st);
                launch_chained(merge_join_kernel, dim3(ceil_div(Nv, 256)), dim3(256), 0, st, Nv, N, w.ev_lo, k, w.ev_out_off, to);
            }
            METOK_LAUNCH_CHECK();
        }
    }

    // Pieces of up to 2 KB, or of 1 KB (so that twice as many copies of a row list are in flight per warp) when the rows
    // are that short or 2 KB pieces would leave half of the warps without one.
    AvgArgs ar = {};
    const int nchunk = d * (int)sizeof(T) / 16;
    const int warps = kNumSMs * kAvgCtasPerSm * kAvgWarps;
    const bool small = nchunk <= 64 || (long long)cap * ceil_div(nchunk, 128) < warps / 2;
    ar.nseg = ceil_div(nchunk, small ? 64 : 128);
    ar.seg_chunks = ceil_div(nchunk, ar.nseg);
    ar.d = d; ar.N = N; ar.Nv = Nv;
    ar.ev_lo = w.ev_lo; ar.out_event = out_event; ar.assign = assign;
    ar.ml = w.ml;
    ar.long_sums = w.long_sums; ar.long_done = w.long_done; ar.next_item = w.avg_next; ar.next = w.avg_next + 1;
    ar.n_out = n_out; ar.out_members = out_members; ar.status = w.status;
    // a warp per piece, and CTAs for the outputs with many members, which there may be Nv / (kAvgHeavy + 1) of
    const long long pieces = (long long)cap * ar.nseg, heavy = std::min<long long>(kNumSMs, (long long)Nv / (kAvgHeavy + 1) * ar.nseg);
    const int grid = (int)std::min<long long>(kNumSMs * kAvgCtasPerSm, (pieces + kAvgWarps - 1) / kAvgWarps + heavy);
    auto launch = [&](auto kernel) -> int {
        METOK_ALLOW_SMEM(kernel, kAvgSmemBytes);
        {
            METOK_TIMED("merge_avg_kernel", st);
            launch_chained(kernel, dim3(grid), dim3(kAvgThreads), kAvgSmemBytes, st, feats, out_feats, ar);
        }
        METOK_LAUNCH_CHECK();
        return METOK_OK;
    };
    return small ? launch(merge_avg_kernel<T, 8>) : launch(merge_avg_kernel<T, 4>);
}

}  // namespace metok

using namespace metok;

static int vision_params_ok(const metok_vision_params* p, int N) {
    if (!p) return 0;
    if (!ratio_ok(p->alpha)) return 0;
    if (p->event_agg != METOK_AGG_MEAN && p->event_agg != METOK_AGG_MAX) return 0;
    if (p->mode == METOK_MODE_TOPK_MERGE) return ratio_ok(p->keep_key) && ratio_ok(p->keep_nonkey);
    if (p->mode == METOK_MODE_POOL) {
        if (!ratio_ok(p->beta)) return 0;
        if (p->s1 < 1 || p->s2 < 1 || p->s1_nonkey < 1 || p->s2_nonkey < 1) return 0;
        int g = 1;
        while (g * g < N) ++g;
        return g * g == N;
    }
    return 0;
}

extern "C" int metok_compress_vision_bound(int T, int N, int k, const metok_vision_params* p) {
    if (T < 1 || N < 1 || k < 1 || k > T || !vision_params_ok(p, N)) return METOK_ERR_INVALID_ARG;
    const long long Nv = (long long)T * N;
    if (p->mode == METOK_MODE_TOPK_MERGE) {
        const double r = p->keep_key > p->keep_nonkey ? p->keep_key : p->keep_nonkey;
        long long b = (long long)ceilq(r * (double)Nv) + k;     // sum of per-event ceilings
        if (b > Nv) b = Nv;
        return (int)b;
    }
    int smin = p->s1;
    if (p->s2 < smin) smin = p->s2;
    if (p->s1_nonkey < smin) smin = p->s1_nonkey;
    if (p->s2_nonkey < smin) smin = p->s2_nonkey;
    int g = 1;
    while (g * g < N) ++g;
    const int go = (g + smin - 1) / smin;
    return T * go * go;
}

extern "C" size_t metok_compress_vision_workspace_bytes(int dtype, int T, int N, int d, int k, int cap,
                                                        const metok_vision_params* p) {
    if (T < 1 || N < 1 || k < 1 || d < 1 || cap < 0) return 0;
    const bool merging = !(p && p->mode == METOK_MODE_POOL);
    bool planes = merging && dtype == METOK_F32 && !force_simt() && (long long)T * N <= 0x7FFFFFFFLL / 2;
    if (planes && p) planes = choose_f3(T * N, k, d, cap, p->alpha * p->keep_key + (1.0 - p->alpha) * p->keep_nonkey) > 0;
    else if (planes) planes = f3_fits((long long)T * N, k, d, cap);
    return vision_ws_bytes(T, N, k, d, cap, merging, planes);
}

extern "C" int metok_compress_vision(const void* feats, int dtype, int T, int N, int d,
                                     const int32_t* event_offsets, int k, const void* text_emb,
                                     const metok_vision_params* p, void* out_feats, int32_t* out_src,
                                     int32_t* out_event, int32_t* out_members, int32_t* assign,
                                     float* token_score, float* frame_score, float* event_score,
                                     uint8_t* event_is_key, int32_t* n_out, int cap, void* ws, size_t ws_bytes,
                                     void* stream) {
    if (!feats || !event_offsets || !text_emb || !p || !out_feats || !out_src || !out_event || !out_members ||
        !assign || !token_score || !frame_score || !event_score || !event_is_key || !n_out)
        return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (T < 1 || N < 1 || d < 1 || k < 1 || k > T) return METOK_ERR_INVALID_ARG;
    if ((long long)T * N > 0x7FFFFFFFLL / 2) return METOK_ERR_INVALID_ARG;
    if (!vision_params_ok(p, N)) return METOK_ERR_INVALID_ARG;
    if (!aligned16(feats) || !aligned16(text_emb) || !aligned16(out_feats)) return METOK_ERR_INVALID_ARG;
    const int bound = metok_compress_vision_bound(T, N, k, p);
    if (bound < 0 || cap < bound) return METOK_ERR_INVALID_ARG;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (((long long)d * eb) % 16 != 0 || T > 8192) return METOK_ERR_UNSUPPORTED;
    const size_t need = vision_ws_bytes(T, N, k, d, cap, p->mode != METOK_MODE_POOL, false);
    if (!ws || ws_bytes < need || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (dtype == METOK_F32)
        return launch_vision<float>(feats, T, N, d, event_offsets, k, text_emb, p, out_feats, out_src, out_event,
                                    out_members, assign, token_score, frame_score, event_score, event_is_key,
                                    n_out, cap, ws, ws_bytes, st);
    return launch_vision<__nv_bfloat16>(feats, T, N, d, event_offsets, k, text_emb, p, out_feats, out_src,
                                        out_event, out_members, assign, token_score, frame_score, event_score,
                                        event_is_key, n_out, cap, ws, ws_bytes, st);
}
