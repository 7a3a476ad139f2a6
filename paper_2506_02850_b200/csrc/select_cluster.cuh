// Exact multi-class top-k of up to 81 920 scored items by one CTA or one cluster of eight, with the items in
// registers.  Used by the class-wise top-k of the pruning levels, the K/V lists and the per-event key-token
// selection; select.cuh takes the larger problems.
//
// Every item gets a 64-bit key (score key << 32 | ~index): unique, and larger <=> ranks higher (higher score,
// lower index on equal scores).  A CTA owns a contiguous slice of the items, a warp a contiguous run of it, a lane
// every 32nd item, so that kept items are counted and placed by ballots.
//   1  load, keys, [min, max] of the score keys                                       -> barrier
//   2  histogram of (key - min) >> shift per class, and the sums of every 32 buckets  -> barrier
//   3  one warp per class finds the bucket of the n-th best: sums first, then the 32
//      buckets behind one sum; it also learns how many items lower CTAs keep
//   4  items above the bucket are kept, the few inside it (at most kCsCand) are listed
//      in every CTA                                                                   -> barrier
//   5  every CTA ranks the listed items and so knows the threshold and the place of its own
// What bounds it is this chain: a step costs a barrier, a round trip to shared memory (a neighbour's costs about
// 600 clocks), and its instructions, which every warp executes whatever it holds.  So what the others need to know is
// written into their shared memory before a barrier instead of being fetched after it (only the 32 buckets are
// fetched), and the steps keep to a few instructions per item.
// A bucket with more than kCsCand items (many equal or nearly equal scores) is narrowed by further passes over
// the 64-bit keys, which are unique, so this ends.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace metok {

namespace cg = cooperative_groups;

constexpr int kCsCand = 128;           // most items ranked by counting
constexpr int kCsMaxCluster = 8;
constexpr int kCsMaxItems = 16;        // items per thread at most ...
constexpr int kCsMaxItemsThreads = 640;   // ... and threads of a CTA then (registers)
constexpr int kCsNone = 1 << 30;

struct CsShared {
    unsigned long long lo[METOK_MAX_GROUPS], hi[METOK_MAX_GROUPS];   // key range of the search, finally of the listed items
    unsigned long long thr[METOK_MAX_GROUPS];                        // a listed item is kept if its key is at least this
    int bucket[METOK_MAX_GROUPS + 1];                                // first pass: the bucket; -1 keep all, kCsNone keep none (last entry: no class)
    int shift[METOK_MAX_GROUPS];                                     // bucket width = 1 << shift
    int need[METOK_MAX_GROUPS];                                      // items to take inside [lo, hi]
    int total[METOK_MAX_GROUPS];                                     // items of the class
    int cand_n[METOK_MAX_GROUPS];                                    // items listed
    int cand_low[METOK_MAX_GROUPS], cand_from[METOK_MAX_GROUPS];     // those of lower CTAs; where this CTA's next one goes
    unsigned char state[METOK_MAX_GROUPS];                           // 0 decided, 1 narrowing, 2 listing
    uint32_t red_min[32], red_max[32];                               // per warp
    int warp_tot[32];                                                // kept items per warp
    uint2 x_range[kCsMaxCluster];                                    // per CTA of the cluster, written by it
    int before, kept;                                                // items kept by lower CTAs; by all
    int busy;
};

struct CsLayout {
    int nb_log2;
    uint32_t coarse_off, cand_off, bytes;
};
// Buckets: 2048 as long as they fit; fewer for small problems, which would only clear and add up empty ones.
inline CsLayout cs_layout(int G, long long n) {
    CsLayout L;
    L.nb_log2 = G <= 4 ? 11 : G <= 16 ? 10 : G <= 32 ? 9 : 7;
    while (L.nb_log2 > 8 && (1LL << (L.nb_log2 + 1)) > n) --L.nb_log2;
    const uint32_t hist = ((uint32_t)G << L.nb_log2) * 4u;
    L.coarse_off = 2 * hist;                                         // histograms alternate between passes,
    L.cand_off = L.coarse_off + 2 * kCsMaxCluster * (hist / 32);     // so do the sums, which there is a set of per CTA
    L.bytes = L.cand_off + (uint32_t)G * kCsCand * 8u;
    return L;
}

__device__ __forceinline__ unsigned long long cs_key64(uint32_t key, uint32_t i) {
    return ((unsigned long long)key << 32) | (unsigned long long)(~i);
}

// The same shared-memory variable in CTA `rank` of the cluster.
template <bool kCl, typename T>
__device__ __forceinline__ T* cs_at(T* p, int rank) {
    if constexpr (kCl) return cg::this_cluster().map_shared_rank(p, rank);
    return p;
}
template <bool kCl>
__device__ __forceinline__ void cs_barrier() {
    if constexpr (kCl) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}
// First statement of a cluster's CTA: nobody writes into a CTA that has not started.  (Nor does anybody touch one that
// has ended: cs_select ends with a barrier after the last access to other CTAs' memory.)
template <bool kCl>
__device__ __forceinline__ void cs_enter() {
    if constexpr (kCl) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}

__device__ __forceinline__ int cs_warp_scan(int v, int lane) {       // inclusive
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += a;
    }
    return v;
}

// One warp per searching class: the bucket that holds the need-th best, counted from the top.  `coarse` holds the
// sums of every CTA of the cluster, `hist` this CTA's buckets.
template <bool kCl>
__device__ __forceinline__ void cs_walk(CsShared& sm, uint32_t* hist, const uint32_t* coarse, int G, int nb_log2, int rank,
                                        bool first, const int* __restrict__ budgets) {
    constexpr int C = kCl ? kCsMaxCluster : 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int NC = 1 << (nb_log2 - 5);                               // 32-bucket sums per class: 4 .. 64
    for (int g = warp; g < G; g += nwarps) {
        if (sm.state[g] != 1) continue;
        // lane l: the sums NC - 1 - 2 l and NC - 2 - 2 l; l0 and l1 are the parts of CTAs before this one
        const int i0 = NC - 1 - 2 * lane;
        int s0 = 0, s1 = 0, l0 = 0, l1 = 0;
        if (i0 > 0) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const uint32_t* x = coarse + c * (G * NC) + g * NC + i0;
                const int a = (int)x[0], b = (int)x[-1];
                if (kCl && c == rank) { l0 = s0; l1 = s1; }
                s0 += a;
                s1 += b;
            }
        }
        const int incl = cs_warp_scan(s0 + s1, lane), excl = incl - s0 - s1;
        const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        int need = sm.need[g];
        if (first) {
            int b = budgets[g];
            b = b < total ? b : total;                               // a budget above the population keeps everything
            if (lane == 0) {
                sm.total[g] = total;
                if (b > 0) atomicAdd(&sm.kept, b);
            }
            if (b <= 0 || b >= total) {
                const int lower = kCl ? (int)__reduce_add_sync(0xFFFFFFFFu, l0 + l1) : 0;
                if (lane == 0) {                                     // every key is above 0, none is above the largest integer
                    sm.state[g] = 0;
                    sm.bucket[g] = b <= 0 ? kCsNone : -1;
                    sm.hi[g] = b <= 0 ? ~0ull : 0ull;
                    if (b > 0 && lower) atomicAdd(&sm.before, lower);
                }
                continue;
            }
            need = b;
        }
        const bool in0 = excl < need && need <= excl + s0, in1 = excl + s0 < need && need <= incl;
        const int hl = __ffs(__ballot_sync(0xFFFFFFFFu, in0 || in1)) - 1;   // exactly one lane
        const int group = __shfl_sync(0xFFFFFFFFu, in0 ? i0 : i0 - 1, hl);
        const int above = __shfl_sync(0xFFFFFFFFu, in0 ? excl : excl + s0, hl);
        int v = 0, from = 0;                                         // lane l: bucket 31 - l of the group
        uint32_t* h = &hist[(g << nb_log2) + group * 32 + 31 - lane];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (kCl && c == rank) from = v;
            v += (int)*cs_at<kCl>(h, c);
        }
        const int pv = cs_warp_scan(v, lane);
        const int want = need - above;
        const bool hit = pv - v < want && want <= pv;                // exactly one lane
        if constexpr (kCl) {
            const int hb = __ffs(__ballot_sync(0xFFFFFFFFu, hit)) - 1;
            const int lower = __reduce_add_sync(0xFFFFFFFFu, (lane < hl ? l0 + l1 : lane == hl && !in0 ? l0 : 0) + (lane < hb ? from : 0));
            if (lane == 0 && lower) atomicAdd(&sm.before, lower);
        }
        if (hit) {
            const int bucket = group * 32 + 31 - lane, sh = sm.shift[g];
            const unsigned long long lo = sm.lo[g] + ((unsigned long long)bucket << sh), top = sm.hi[g];
            const unsigned long long span = sh ? ((1ull << sh) - 1ull) : 0ull;
            const unsigned long long hi = top - lo < span ? top : lo + span;
            sm.lo[g] = lo;
            sm.hi[g] = hi;
            sm.need[g] = want - (pv - v);
            if (v <= kCsCand) {
                sm.state[g] = 2;
                sm.bucket[g] = bucket;
                sm.cand_n[g] = v;
                sm.cand_low[g] = from;
                sm.cand_from[g] = from;
            } else {
                const unsigned long long width = hi - lo;
                const int bits = width ? 64 - __clzll((long long)width) : 0;
                sm.shift[g] = bits > nb_log2 ? bits - nb_log2 : 0;
                sm.busy = 1;
            }
        }
    }
}

// Sums of 32 buckets, eight lanes per sum; in a cluster lane c of the eight gives it to CTA c.
template <bool kCl>
__device__ __forceinline__ void cs_sums(const uint32_t* hist, uint32_t* coarse, int buckets, int rank) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < buckets / 4; i += blockDim.x) {    // a multiple of 32: whole warps
        const uint4 h = reinterpret_cast<const uint4*>(hist)[i];
        uint32_t s = h.x + h.y + h.z + h.w;
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 4);
        if constexpr (kCl) *cs_at<true>(&coarse[rank * (buckets / 32) + (i >> 3)], lane & 7) = s;
        else if ((lane & 7) == 0) coarse[i >> 3] = s;
    }
}

// Decides which items are kept.  Item j of this thread is i = i_first + 32 j, j < IT, if i < i_hi; `load(j, i, v, c)`
// gives its score and class (c < 0: it takes no part).  On return bit j of the result says whether it is kept;
// *before is the number of items kept before this warp's first one in the whole problem, *kept the number of all;
// sm.total[g] is the number of items of class g.  All threads of the cluster (or CTA) call it, after cs_enter().
template <int IT, bool kCl, bool kOne, typename LoadF>
__device__ __forceinline__ uint32_t cs_select(CsShared& sm, unsigned char* dyn, const CsLayout& lay, int G,
                                              const int* __restrict__ budgets, int rank, int i_first, int i_hi, LoadF load,
                                              int* before, int* kept) {
    constexpr int C = kCl ? kCsMaxCluster : 1;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
    const int nb_log2 = lay.nb_log2, buckets = G << nb_log2;
    uint32_t* hist = reinterpret_cast<uint32_t*>(dyn);               // two of `buckets`, for alternating passes
    uint32_t* coarse = reinterpret_cast<uint32_t*>(dyn + lay.coarse_off);
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(dyn + lay.cand_off);

    // 1: the items, and the range of their keys
    uint32_t key[IT];
    int cls[IT];
    {
        float v[IT];
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            cls[j] = -1;
            v[j] = 0.f;
            if (i_first + 32 * j < i_hi) load(j, i_first + 32 * j, v[j], cls[j]);
        }
        for (int b = tid; b < buckets / 4; b += nthr) reinterpret_cast<uint4*>(hist)[b] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) { sm.busy = 0; sm.before = 0; sm.kept = 0; }
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            key[j] = float_key(v[j]);
            if (cls[j] >= 0) {
                mn = key[j] < mn ? key[j] : mn;
                mx = key[j] > mx ? key[j] : mx;
            }
        }
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (lane == 0) { sm.red_min[warp] = mn; sm.red_max[warp] = mx; }
    }
    __syncthreads();
    uint32_t mn = lane < nwarps ? sm.red_min[lane] : 0xFFFFFFFFu, mx = lane < nwarps ? sm.red_max[lane] : 0u;
    mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if constexpr (kCl) {
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // of cs_enter(): everybody has started
        if (warp == 0 && lane < C) *cs_at<kCl>(&sm.x_range[rank], lane) = make_uint2(mn, mx);
        cs_barrier<kCl>();
        const uint2 r = sm.x_range[lane & (kCsMaxCluster - 1)];
        mn = __reduce_min_sync(0xFFFFFFFFu, r.x);
        mx = __reduce_max_sync(0xFFFFFFFFu, r.y);
    }
    const bool empty = mn > mx;                                      // no item takes part at all
    const int sh0 = empty || mx == mn ? 0 : max(0, 32 - __clz(mx - mn) - nb_log2);
    for (int g = tid; g < G; g += nthr) {
        sm.lo[g] = (unsigned long long)mn << 32;
        sm.hi[g] = empty ? ~0ull : ((unsigned long long)mx << 32) | 0xFFFFFFFFull;
        sm.shift[g] = sh0 + 32;
        sm.bucket[g] = kCsNone;
        sm.need[g] = 0;
        sm.total[g] = 0;
        sm.thr[g] = 0ull;
        sm.state[g] = empty ? 0 : 1;
    }
    if (tid == 0) sm.bucket[METOK_MAX_GROUPS] = kCsNone;

    // 2 and 3: histogram and walk
    bool wide = false;                                               // ranges narrower than a bucket of the first pass
    if (!empty) {
#pragma unroll
        for (int j = 0; j < IT; ++j)
            if (cls[j] >= 0) atomicAdd(&hist[((kOne ? 0 : cls[j]) << nb_log2) + ((key[j] - mn) >> sh0)], 1u);
        __syncthreads();
        cs_sums<kCl>(hist, coarse, buckets, rank);
        cs_barrier<kCl>();
        cs_walk<kCl>(sm, hist, coarse, G, nb_log2, rank, true, budgets);
        __syncthreads();
        wide = sm.busy != 0;
        for (int pass = 1; pass < 16 && sm.busy; ++pass) {
            uint32_t* h = hist + (size_t)(pass & 1) * buckets;
            uint32_t* c = coarse + (size_t)(pass & 1) * C * (buckets / 32);
            for (int b = tid; b < buckets / 4; b += nthr) reinterpret_cast<uint4*>(h)[b] = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
            if (tid == 0) sm.busy = 0;
#pragma unroll
            for (int j = 0; j < IT; ++j) {
                if (cls[j] < 0) continue;
                const int g = kOne ? 0 : cls[j];
                const unsigned long long k64 = cs_key64(key[j], (uint32_t)(i_first + 32 * j)), lo = sm.lo[g];
                if (sm.state[g] == 1 && k64 >= lo && k64 <= sm.hi[g])
                    atomicAdd(&h[(g << nb_log2) + (uint32_t)((k64 - lo) >> sm.shift[g])], 1u);
            }
            __syncthreads();
            cs_sums<kCl>(h, c, buckets, rank);
            cs_barrier<kCl>();
            cs_walk<kCl>(sm, h, c, G, nb_log2, rank, false, budgets);
            __syncthreads();
        }
    } else {
        __syncthreads();
    }

    // 4: kept above the bucket, listed inside it
    uint32_t keep = 0u, open = 0u;
    if (!wide) {
        const int cut0 = sm.bucket[0];
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            const int cut = kOne ? (cls[j] >= 0 ? cut0 : kCsNone) : sm.bucket[cls[j] >= 0 ? cls[j] : METOK_MAX_GROUPS];
            const int b = cls[j] >= 0 ? (int)((key[j] - mn) >> sh0) : 0;
            keep |= (b > cut ? 1u : 0u) << j;
            open |= (b == cut ? 1u : 0u) << j;
        }
    } else {
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            const int g = kOne ? 0 : max(cls[j], 0);
            const unsigned long long k64 = cs_key64(key[j], (uint32_t)(i_first + 32 * j));
            const bool up = cls[j] >= 0 && k64 > sm.hi[g];
            keep |= (up ? 1u : 0u) << j;
            open |= (cls[j] >= 0 && !up && sm.state[g] == 2 && k64 >= sm.lo[g] ? 1u : 0u) << j;
        }
    }
    if (open) {
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            if ((open >> j) & 1u) {
                const int g = kOne ? 0 : cls[j];
                unsigned long long* at = &cand[g * kCsCand + atomicAdd(&sm.cand_from[g], 1)];
                const unsigned long long k64 = cs_key64(key[j], (uint32_t)(i_first + 32 * j));
#pragma unroll
                for (int c = 0; c < C; ++c) *cs_at<kCl>(at, c) = k64;
            }
        }
    }
    cs_barrier<kCl>();

    // 5: the listed items ranked, 32 of a class per warp
    constexpr int kParts = kCsCand / 32;
    for (int t = warp; t < G * kParts; t += nwarps) {
        const int g = t / kParts, i0 = (t - g * kParts) * 32, i = i0 + lane;
        if (sm.state[g] != 2) continue;
        const unsigned long long* a = cand + g * kCsCand;
        const int m = sm.cand_n[g];
        if (i0 < m) {
            const int need = sm.need[g];
            const unsigned long long c = i < m ? a[i] : ~0ull;
            int better = 0;
#pragma unroll 8
            for (int x = 0; x < m; ++x) better += a[x] > c;
            if (i < m && better == need - 1) sm.thr[g] = c;
            if constexpr (kCl) {                                     // those of them that lower CTAs keep
                const int lower = __popc(__ballot_sync(0xFFFFFFFFu, i < sm.cand_low[g] && better < need));
                if (lane == 0 && lower) atomicAdd(&sm.before, lower);
            }
        }
    }
    __syncthreads();
    int mine = __reduce_add_sync(0xFFFFFFFFu, __popc(keep));
    if (__any_sync(0xFFFFFFFFu, open != 0u)) {
#pragma unroll
        for (int j = 0; j < IT; ++j) {
            const bool take = ((open >> j) & 1u) && cs_key64(key[j], (uint32_t)(i_first + 32 * j)) >= sm.thr[kOne ? 0 : cls[j]];
            keep |= (take ? 1u : 0u) << j;
        }
        mine = __reduce_add_sync(0xFFFFFFFFu, __popc(keep));
    }
    if (lane == 0) sm.warp_tot[warp] = mine;
    __syncthreads();
    *before = sm.before + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? sm.warp_tot[lane] : 0);
    *kept = sm.kept;
    return keep;
}

// Calls f(j, i, place, is_kept) for this thread's items; place = number of kept items before it in the problem.
template <int IT, typename F>
__device__ __forceinline__ void cs_for_items(uint32_t keep, int before, int i_first, int i_hi, F f) {
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
#pragma unroll
    for (int j = 0; j < IT; ++j) {
        const bool k = (keep >> j) & 1u;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, k);
        const int i = i_first + 32 * j;
        if (i < i_hi) f(j, i, before + __popc(bal & lt), k);
        before += __popc(bal);
    }
}

// Items of a problem of n items: CTA `rank` of C owns a contiguous slice, warp w the w-th run of 32 * IT of it.
struct CsSlice { int i_first, i_hi; };
template <int IT>
__device__ __forceinline__ CsSlice cs_slice(int n, int rank, int C) {
    const int per = (n + C - 1) / C, lo = min(n, rank * per), hi = min(n, lo + per);
    const int first = lo + (int)(threadIdx.x >> 5) * 32 * IT;
    CsSlice s;
    s.i_first = first + (int)(threadIdx.x & 31);
    s.i_hi = min(hi, first + 32 * IT);
    return s;
}

// How a problem of at most n items is cut up: one CTA up to kCsSolo items (a cluster's barriers cost more than its
// SMs save there), else a cluster of eight.  Four items per thread: every step costs each warp some fifty
// instructions whatever it holds and about ten per item, so fewer, fuller warps are faster.
constexpr int kCsSolo = 4096;
struct CsPlan { int C, threads, items; bool fits; };
inline CsPlan cs_plan(long long n) {
    CsPlan p;
    p.C = n <= kCsSolo ? 1 : kCsMaxCluster;
    const long long per = (n + p.C - 1) / p.C;
    p.items = per <= 4096 ? 4 : kCsMaxItems;
    p.fits = per <= kCsMaxItemsThreads * (long long)kCsMaxItems;
    const long long t = (per + p.items - 1) / p.items;
    p.threads = (int)(t <= 64 ? 64 : t >= 1024 ? 1024 : (t + 31) / 32 * 32);
    return p;
}

}  // namespace metok
