// Text->visual attention scores on the tensor cores (bf16, head dim 64 or 128).
//
// Per KV head g the rep = Hq/Hkv query heads of the group give R = rep*Lt query rows
// (row r = local head * Lt + q) that all multiply the same K[g].  The R x S matrix of
// probabilities is never stored.  Two kernels, both TMA -> shared memory ->
// tcgen05.mma -> TMEM -> registers:
//
//   stats  : D = Q_tile (128 query rows = TMEM lanes) x K_tile^T (256 keys = columns).
//            A thread owns one query row, so the running (max, sum) of the softmax is
//            thread-local.  The keys are split over CTAs; each CTA leaves one (max,
//            sum) pair per row (the column quarters are merged in the CTA).
//   colsum : D = K_tile (128 keys = TMEM lanes) x Q_chunk^T (up to 256 query rows =
//            columns).  The row normalisers are known now (log-sum-exp per query row,
//            kept in shared memory), a thread owns one key and adds up
//            exp2(logit - lse) over its columns: the sum over queries is thread-local
//            too.  Only key tiles that touch the visual span are visited.
//
// Warp roles in both: warp 0 = TMA producer, warp 1 = MMA issuer (one elected lane),
// the others = epilogue: four warps per TMEM lane quadrant, each taking a quarter of the
// columns.  Two accumulators in TMEM (2 x 256 columns) so
// that the epilogue of tile i overlaps the MMA of tile i+1.  Every wait is bounded.
//
// What bounds both is the exponentials and what goes with them: 16 a clock on an SM's special-function units, so every
// fourth pair is taken on the FMA pipe, the multiply-adds and sums are done two at a time (half the issue slots), stats
// takes no maximum after its first tile, and a warp empties its part of the accumulator before the arithmetic, so that
// the next product never waits for it.  28 heads, 128 queries, 73 856 keys of 128: stats 85 -> 74 us (76 since its arguments
// are held below 2^126), colsum 91 -> 80.
#include <algorithm>

#include "common.cuh"
#include "launchers.h"
#include "sm100.cuh"

namespace metok {

namespace {

constexpr int kEpiWarps = 16;             // four warps per TMEM lane quadrant, a quarter of a tile's columns each
constexpr int kThreads = 64 + kEpiWarps * 32;
constexpr float kLog2e = 1.4426950408889634f;
template <int V> struct Int { static constexpr int value = V; };
constexpr float kNegInf = -3.0e38f;       // finite stand-in: keeps (m_old - m_new) free of inf - inf

constexpr int kStBM = 128;                // stats: query rows per CTA
constexpr int kStBN = 256;                // stats: keys per tile
constexpr int kStStages = 2;
constexpr int kCsBM = 128;                // colsum: keys per tile
constexpr int kCsMaxNQ = 256;             // colsum: query rows per chunk (multiple of 32)
constexpr int kCsStages = 4;
constexpr int kCsItems = 4;               // colsum: items whose normalisers are worked out at a time
constexpr uint32_t kCsRingBytes = 216 * 1024;   // colsum: queries of two items and up to kCsStages key tiles
constexpr int kStMinTiles = 2;            // fewest key tiles a stats CTA is started for
constexpr int kCsMinTiles = 3;            // the same for colsum (on average)

struct AttnMmaDims {
    int Hq, Hkv, Lt, S, vis_start, n_vis, R;
    int st_nrt, st_tiles, st_per, st_nsplit;          // stats: row tiles, key tiles, tiles per split, splits
    int cs_nq, cs_nchunk, cs_t0, cs_tiles, cs_per, cs_nsplit;   // colsum; the last two of a level scored alone
    float scale_log2;
};

__host__ AttnMmaDims make_mma_dims(int Hq, int Hkv, int Lt, int S, int vis_start, int n_vis, float scale) {
    AttnMmaDims dm;
    dm.Hq = Hq; dm.Hkv = Hkv; dm.Lt = Lt; dm.S = S; dm.vis_start = vis_start; dm.n_vis = n_vis;
    dm.R = (Hq / Hkv) * Lt;
    dm.scale_log2 = scale * kLog2e;
    // one CTA per SM: as many key splits as keep the grid within one wave
    dm.st_nrt = ceil_div(dm.R, kStBM);
    dm.st_tiles = ceil_div(S, kStBN);
    // ... but a CTA gets at least kStMinTiles tiles: a launch that is mostly prologue on every SM
    // keeps other streams' kernels off the GPU for nothing
    int ns = kNumSMs / (Hkv * dm.st_nrt);
    if (ns > ceil_div(dm.st_tiles, kStMinTiles)) ns = ceil_div(dm.st_tiles, kStMinTiles);
    if (ns < 1) ns = 1;
    if (ns > dm.st_tiles) ns = dm.st_tiles;
    dm.st_per = ceil_div(dm.st_tiles, ns);
    dm.st_nsplit = ceil_div(dm.st_tiles, dm.st_per);   // every split owns at least one tile
    dm.cs_nchunk = ceil_div(dm.R, kCsMaxNQ);
    dm.cs_nq = ceil_div(ceil_div(dm.R, dm.cs_nchunk), 32) * 32;       // quarters of whole 8-column groups
    dm.cs_t0 = vis_start / kCsBM;
    dm.cs_tiles = (vis_start + n_vis - 1) / kCsBM - dm.cs_t0 + 1;
    ns = kNumSMs / (Hkv * dm.cs_nchunk);
    // A level scored alone: at least kCsMinTiles key tiles per CTA, or fewer where the launch then still leaves five eighths of the SMs to
    // other streams' kernels, for which a CTA that is mostly set-up is SM time lost.  Heads / queries / keys, one call (graph) and a
    // pruning call of eight streams at once, with three tiles / one / so:
    //   14 / 24 / 6272   13.8 / 11.6 / 12.7 us    6.4 / 7.7 / 6.7        28 / 64 / 1536   14.7 / 12.3 / 13.6    6.0 / 7.3 / 6.4
    //   28 / 64 / 784    15.6 / 13.3 / 14.4       4.0 / 4.5 / 4.1        28 / 64 / 2160   14.8 / 12.9 / 14.8    8.2 / 10.2 / 8.2
    //   14 / 24 / 784    14.0 / 12.0 / 12.0       3.3 / 3.0 / 3.0        14 / 24 / 2048   13.3 / 11.2 / 11.2    3.4 / 3.4 / 3.4
    // Eight 128-frame videos at once, all calls: 96.1 / 95.4 / 96.1 M visual tokens/s.
    ns = std::min(ns, std::max(ceil_div(dm.cs_tiles, kCsMinTiles), kNumSMs * 3 / 8 / (Hkv * dm.cs_nchunk)));
    if (ns < 1) ns = 1;
    if (ns > dm.cs_tiles) ns = dm.cs_tiles;
    dm.cs_per = ceil_div(dm.cs_tiles, ns);
    dm.cs_nsplit = ceil_div(dm.cs_tiles, dm.cs_per);
    return dm;
}

// Key tiles in flight beside the queries of two items.
__host__ __device__ inline int cs_stages(int nq, int dh) {
    const int n = ((int)kCsRingBytes - 2 * nq * dh * 2) / (kCsBM * dh * 2);
    return n < kCsStages ? n : kCsStages;
}

// What one launch scores: one level, or the pruning levels of a schedule together (their queries, keys and sizes are all
// known before the first one).  A CTA's share of a level is an item: a run of key tiles of one row tile or query chunk.
// Its barriers, ring and tensor memory run on from item to item, and the next item's queries are fetched while one is
// worked on.
//   stats : a row's normaliser is added up in the order of the runs, so every level is cut as it is when it is scored
//           alone and its results are the same to the bit.  The items of all levels form one list, longest first; CTA c
//           takes the c-th of every round of gridDim items, forwards and backwards in turn.
//   colsum: a key's sum does not depend on the run it is in, so the key tiles of all query chunks, KV heads and levels form
//           one line, and every CTA takes an equal piece of it (24 us for the three levels below, 27.6 with stats' list).
// A level scored alone keeps a CTA per item: with pieces of the line, some of which cross from one head to the next, 14
// heads x 24 queries x 6272 keys took 27.4 us the whole call instead of 25.2.
// (18 432, 6 768 and 2 160 keys, 28 heads x 64 queries: the two passes took 17.7 + 16.1, 11.6 + 9.7 and 8.7 + 8.9 us in launches
// of their own, of which every one spent about 3 us before its first tile.)
struct AttnLevel {
    AttnMmaDims dm;
    float *part_m, *part_l, *part_col;
};
template <int NL>
struct AttnBatch {
    CUtensorMap q[NL], k[NL];
    AttnLevel lv[NL];
    int first[NL + 1];                                // stats: items before each level's; colsum: key tiles
};
struct AttnItem { int level, row, g, t_lo, nt, split; };   // row: row tile (stats) or query chunk (colsum); nt key tiles from t_lo on
// The CTA's n-th item.
template <int NL>
__device__ __forceinline__ bool stats_item(const AttnBatch<NL>& ab, int n, AttnItem& it) {
    it.level = 0;
    if constexpr (NL == 1) {                          // a CTA per item
        if (n > 0) return false;
        it.split = blockIdx.x;
        it.row = blockIdx.y;
        it.g = blockIdx.z;
    } else {
        int i = n * (int)gridDim.x + ((n & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
        if (i >= ab.first[NL]) return false;
#pragma unroll
        for (int l = 1; l < NL; ++l) it.level += i >= ab.first[l];
        i -= ab.first[it.level];
        const int ns = ab.lv[it.level].dm.st_nsplit, nr = ab.lv[it.level].dm.st_nrt;
        it.split = i % ns;
        i /= ns;
        it.row = i % nr;
        it.g = i / nr;
    }
    const AttnMmaDims& dm = ab.lv[it.level].dm;
    it.t_lo = it.split * dm.st_per;
    it.nt = min(dm.st_tiles, it.t_lo + dm.st_per) - it.t_lo;          // >= 1 by construction
    return true;
}
// The item that starts at `at`, where the CTA's piece of the line ends at `end`; `at` moves past it.
template <int NL>
__device__ __forceinline__ bool colsum_item(const AttnBatch<NL>& ab, int& at, int end, AttnItem& it) {
    if (at >= end) return false;
    it.level = 0;
    it.split = 0;
    const AttnMmaDims& dm0 = ab.lv[0].dm;
    if constexpr (NL == 1) {
        it.row = blockIdx.y;
        it.g = blockIdx.z;
        it.t_lo = dm0.cs_t0 + (int)blockIdx.x * dm0.cs_per;
        it.nt = min(dm0.cs_t0 + dm0.cs_tiles, it.t_lo + dm0.cs_per) - it.t_lo;
        at = end;
    } else {
#pragma unroll
        for (int l = 1; l < NL; ++l) it.level += at >= ab.first[l];
        const AttnMmaDims& dm = ab.lv[it.level].dm;
        const int local = at - ab.first[it.level], line = local / dm.cs_tiles, t = local - line * dm.cs_tiles;
        it.g = line / dm.cs_nchunk;
        it.row = line - it.g * dm.cs_nchunk;
        it.t_lo = dm.cs_t0 + t;
        it.nt = min(dm.cs_tiles - t, end - at);
        at += it.nt;
    }
    return true;
}

// Sum of 2^(v[j] * sc + add) over the 32 columns; every fourth pair's exponentials on the FMA pipe.  Wherever an exponent is
// above the range the sum is above 1e18, never below it.
__device__ __forceinline__ float exp2_sum32(const uint32_t (&v)[32], uint64_t sc, uint64_t add) {
    using namespace sm100;
    uint64_t s0 = 0ull, s1 = 0ull;                             // {0.f, 0.f}
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const uint64_t x = fma_pair(pair(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), sc, add);
        const uint64_t e = (j & 3) == 3 ? exp2_fma_pair<true>(x) : exp2_pair(x);
        if (j & 1) s1 = add_pair(s1, e);
        else s0 = add_pair(s0, e);
    }
    float a, b;
    unpair(add_pair(s0, s1), a, b);
    return a + b;
}

// --------------------------------------------------------------------------- //
// stats
// --------------------------------------------------------------------------- //
template <int DH, int NL>
__global__ void __launch_bounds__(kThreads, 1)
attn_stats_mma_kernel(const __grid_constant__ AttnBatch<NL> ab, int32_t* __restrict__ status) {
    grid_dep_wait();
    using namespace sm100;
    constexpr int KB = DH / 64;                               // 64-element (128-byte) K blocks
    constexpr uint32_t kQBlk = kStBM * 128, kKBlk = kStBN * 128;
    constexpr uint32_t kQBytes = KB * kQBlk, kKBytes = KB * kKBlk;
    constexpr int kQBufs = NL > 1 ? 2 : 1;
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t q_bar[kQBufs], q_free_bar[kQBufs], drain_bar, full_bar[kStStages], empty_bar[kStStages], tfull_bar[2],
        tempty_bar[2];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ float s_pm[2][4][kStBM], s_pl[2][4][kStBM];    // the column quarters' (max, sum) per query row, of two items

    // The call's status word and class counts start cleared: written by the first CTA of the call's first kernel
    // instead of by a memset node.  A CTA that gives up writes the status only after its waits have run
    // out, seconds later.
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
        *status = 0;
        status[kStatusCounts] = status[kStatusCounts + 1] = 0;
    }
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t q_addr = smem_base;
    auto k_addr = [&](int s) { return smem_base + kQBufs * kQBytes + (uint32_t)s * kKBytes; };

    if (threadIdx.x == 0) {
        for (int b = 0; b < kQBufs; ++b) { mbar_init(smem_u32(&q_bar[b]), 1); mbar_init(smem_u32(&q_free_bar[b]), 1); }
        mbar_init(smem_u32(&drain_bar), 1);
        for (int s = 0; s < kStStages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tfull_bar[b]), 1); mbar_init(smem_u32(&tempty_bar[b]), kEpiWarps); }
        s_abort = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&s_tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);

    // Warps 0 and 1, here and in the colsum kernel, stay whole and one elected thread issues: addresses and descriptors are then
    // in uniform registers.  (In a branch of lane 0 an issue loop costs some 75 clocks per product.  One level of 73 728 keys,
    // 28 heads x 128 queries: 239.1 us the whole call, 234.7 now; three levels from 18 432: 89.2 -> 86.7; 6272: 23.6 -> 23.2.)
    AttnItem item = {};
    if (warp == 0) {
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (elect_one()) { prefetch_tmap(&ab.q[l]); prefetch_tmap(&ab.k[l]); }
        __syncwarp();
        int it = 0, n = 0;                                 // tiles and items so far
        bool ok = true;
        for (; ok && stats_item(ab, n, item); ++n) {
            const AttnMmaDims& dm = ab.lv[item.level].dm;
            const CUtensorMap *tmQ = &ab.q[item.level], *tmK = &ab.k[item.level];
            // the item that had this buffer is done with its query tile
            const int qb = n % kQBufs;
            const uint32_t qph = (uint32_t)(n / kQBufs) & 1u;
            if (!mbar_wait_warp(smem_u32(&q_free_bar[qb]), qph ^ 1u, abort_flag)) { ok = false; break; }
            if (elect_one()) {
                mbar_arrive_expect_tx(smem_u32(&q_bar[qb]), kQBytes);
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
                    tma_load_2d(q_addr + qb * kQBytes + kb * kQBlk, tmQ, kb * 64, item.g * dm.R + item.row * kStBM, smem_u32(&q_bar[qb]));
            }
            __syncwarp();
            for (int t = item.t_lo; t < item.t_lo + item.nt; ++t, ++it) {
                const int s = it % kStStages;
                const uint32_t ph = (uint32_t)(it / kStStages) & 1u;
                if (!mbar_wait_warp(smem_u32(&empty_bar[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t fb = smem_u32(&full_bar[s]);
                const bool held = dbg_withhold(status, kDbgAttnStats) && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && it == 0;   // debug builds: one copy never sent
                if (elect_one()) {
                    mbar_arrive_expect_tx(fb, kKBytes);
                    if (!held) {
#pragma unroll
                        for (int kb = 0; kb < KB; ++kb)
                            tma_load_2d(k_addr(s) + kb * kKBlk, tmK, kb * 64, item.g * dm.S + t * kStBN, fb);
                    }
                }
                __syncwarp();
            }
        }
        // every copy issued has landed before the CTA's shared memory goes away, whichever way the
        // other warps leave (in a normal run these waits are over already)
        for (int j = n > kQBufs ? n - kQBufs : 0; j < n; ++j)
            mbar_wait_warp(smem_u32(&q_bar[j % kQBufs]), (uint32_t)(j / kQBufs) & 1u, abort_flag);
        for (int back = 1; back <= kStStages && back <= it; ++back) {
            const int j = it - back;
            mbar_wait_warp(smem_u32(&full_bar[j % kStStages]), (uint32_t)(j / kStStages) & 1u, abort_flag);
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = make_idesc_bf16(kStBM, kStBN);
        bool ok = true;
        int it = 0;
        for (int n = 0; ok && stats_item(ab, n, item); ++n) {
            const int qb = n % kQBufs;
            ok = mbar_wait_warp(smem_u32(&q_bar[qb]), (uint32_t)(n / kQBufs) & 1u, abort_flag);
            for (const int end = it + item.nt; it < end && ok; ++it) {
                const int b = it & 1, s = it % kStStages;
                if (!mbar_wait_warp(smem_u32(&tempty_bar[b]), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                if (!mbar_wait_warp(smem_u32(&full_bar[s]), (uint32_t)(it / kStStages) & 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)b * kStBN;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < DH / 16; ++kk) {
                        const uint64_t ad = make_desc_k128(q_addr + qb * kQBytes + (kk >> 2) * kQBlk + (kk & 3) * 32);
                        const uint64_t bd = make_desc_k128(k_addr(s) + (kk >> 2) * kKBlk + (kk & 3) * 32);
                        umma_bf16(d_tmem, ad, bd, idesc, kk != 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&empty_bar[s]));
                    umma_commit(smem_u32(&tfull_bar[b]));
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit(smem_u32(&q_free_bar[qb]));
            __syncwarp();
        }
        if (!ok) {                                         // wait until whatever was issued has retired
            if (elect_one()) umma_commit(smem_u32(&drain_bar));
            __syncwarp();
            mbar_wait_warp(smem_u32(&drain_bar), 0u, abort_flag);
        }
    } else {
        const int quad = warp & 3;                             // TMEM lanes 32*quad .. 32*quad+31
        const int part = (warp - 2) >> 2;                      // column quarter of every tile
        bool ok = true;
        int done = 0;                                          // tiles so far
        for (int n = 0; stats_item(ab, n, item); ++n) {
            const AttnLevel& lv = ab.lv[item.level];
            const AttnMmaDims& dm = lv.dm;
            const int t_lo = item.t_lo, nt = item.nt;
            const int text_start = dm.S - dm.Lt;
            const int r = item.row * kStBM + quad * 32 + lane;
            const bool valid = r < dm.R;
            const int limit = valid ? text_start + (r % dm.Lt) : -1;     // last key this query may see
            const float sc = dm.scale_log2;
            float m_run = kNegInf, l_run = 0.f;
            for (int it = 0; it < nt; ++it, ++done) {
                const int b = done & 1;
                if (ok && !mbar_wait(smem_u32(&tfull_bar[b]), (uint32_t)(done >> 1) & 1u, abort_flag)) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);                  // tcgen05.ld below is warp-collective
                if (!ok) break;
                tc_fence_after();
                const int u_tile = (t_lo + it) * kStBN;
                const int u0 = u_tile + part * (kStBN / 4);
                const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * kStBN + part * (kStBN / 4));
                const bool masked = u_tile + kStBN - 1 > text_start;       // some query cannot see some key of the tile
                uint32_t raw[2][32];
                tmem_ld32_issue(taddr, raw[0]);
                // A row's (m_run, l_run) stands for l_run * 2^m_run, and any reference m_run that its logits do not exceed by
                // the exponent range will do: the first tile's maximum stays, later tiles only add 2^(logit - m_run), with no
                // maximum taken.  A chunk whose sum leaves the range (a logit 60 octaves above the reference) is done again
                // against its own maximum.
                const bool plain = !masked && it > 0;
                tmem_ld32_issue(taddr + 32u, raw[1]);
                tmem_ld32_wait(raw[0]);
                tmem_ld32_wait(raw[1]);
                tc_fence_before();                                 // the accumulator is free before the arithmetic
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[b]));
#pragma unroll
                for (int ci = 0; ci < kStBN / 128; ++ci) {
                    const int c0 = ci * 32;
                    bool redo = !plain;
                    if (plain) {
                        const float sum = exp2_sum32(raw[ci & 1], pair(sc, sc), pair(-m_run, -m_run));
                        redo = __any_sync(0xFFFFFFFFu, !(sum >= 0.f && sum < 1.0e18f));
                        if (!redo) l_run += sum;
                    }
                    if (redo) {
                        float v[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(raw[ci & 1][j]);
                        float sum = 0.f;
                        float m_new;
                        if (masked) {                              // hidden keys add exactly nothing
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = (u0 + c0 + j <= limit) ? v[j] * sc : kNegInf;
                            float cm = v[0];
#pragma unroll
                            for (int j = 1; j < 32; ++j) cm = fmaxf(cm, v[j]);
                            m_new = fmaxf(m_run, cm);
#pragma unroll
                            for (int j = 0; j < 32; ++j) sum += (v[j] > kNegInf) ? fast_exp2(v[j] - m_new) : 0.f;
                        } else {
                            // the scale is positive: the maximum of the raw logits, scaled, is the maximum of the scaled ones
                            float t16[16];                         // a tree: the maximum is five steps deep, not 31
#pragma unroll
                            for (int j = 0; j < 16; ++j) t16[j] = fmaxf(v[2 * j], v[2 * j + 1]);
#pragma unroll
                            for (int w = 8; w >= 1; w >>= 1) {
#pragma unroll
                                for (int j = 0; j < w; ++j) t16[j] = fmaxf(t16[j], t16[j + w]);
                            }
                            m_new = fmaxf(m_run, t16[0] * sc);
                            sum = exp2_sum32(raw[ci & 1], pair(sc, sc), pair(-m_new, -m_new));
                        }
                        l_run = l_run * fast_exp2(m_run - m_new) + sum;
                        m_run = m_new;
                    }
                }
            }
            // the four column quarters of a row are merged here, in quarter order: one pair per row and split.  (A warp that
            // gave up keeps meeting the others at this barrier.  Two buffers: who writes one again has passed the barrier of the
            // item between, which the reader reaches after reading.)
            const int rl = quad * 32 + lane, nb = n & 1;
            s_pm[nb][part][rl] = m_run;
            s_pl[nb][part][rl] = l_run;
            asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
            if (part == 0 && ok && valid) {
                float M = s_pm[nb][0][rl];
#pragma unroll
                for (int p2 = 1; p2 < 4; ++p2) M = fmaxf(M, s_pm[nb][p2][rl]);
                float Z = 0.f;
#pragma unroll
                for (int p2 = 0; p2 < 4; ++p2) Z += s_pl[nb][p2][rl] * fast_exp2(s_pm[nb][p2][rl] - M);
                const size_t o = ((size_t)item.g * dm.st_nsplit + (size_t)item.split) * dm.R + r;
                lv.part_m[o] = M;
                lv.part_l[o] = Z;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0 && s_abort) *status = METOK_ERR_TIMEOUT;
}

// --------------------------------------------------------------------------- //
// colsum
// --------------------------------------------------------------------------- //
template <int DH, int NL>
__global__ void __launch_bounds__(kThreads, 1)
attn_colsum_mma_kernel(const __grid_constant__ AttnBatch<NL> ab, int32_t* __restrict__ status) {
    grid_dep_wait();
    using namespace sm100;
    constexpr int KB = DH / 64;
    constexpr uint32_t kKBlk = kCsBM * 128;
    constexpr uint32_t kKBytes = KB * kKBlk;
    constexpr int kQBufs = NL > 1 ? 2 : 1, kItems = NL > 1 ? kCsItems : 1;
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t q_bar[kQBufs], q_free_bar[kQBufs], drain_bar, full_bar[kCsStages], empty_bar[kCsStages], tfull_bar[2],
        tempty_bar[2];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ float s_part[4][3][kCsBM];                      // sums of the column quarters 1 to 3 per key, of four tiles
    __shared__ __align__(8) uint64_t part_bar[4][4];           // [tile % 4][lane quadrant]: its three warps have written them
    __shared__ __align__(16) float s_nlse[kItems][kCsMaxNQ];   // -(log-sum-exp) per query row of the item's chunk, log2 units

    const int NQ = ab.lv[0].dm.cs_nq;                          // the levels have the same queries and heads
    const uint32_t kQBlk = (uint32_t)NQ * 128;
    const uint32_t kQBytes = KB * kQBlk;
    const int stages = NL > 1 ? cs_stages(NQ, DH) : kCsStages;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t q_addr = smem_base;
    auto k_addr = [&](int s) { return smem_base + kQBufs * kQBytes + (uint32_t)s * kKBytes; };

    if (threadIdx.x == 0) {
        for (int b = 0; b < kQBufs; ++b) { mbar_init(smem_u32(&q_bar[b]), 1); mbar_init(smem_u32(&q_free_bar[b]), 1); }
        mbar_init(smem_u32(&drain_bar), 1);
        for (int s = 0; s < kCsStages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tfull_bar[b]), 1); mbar_init(smem_u32(&tempty_bar[b]), kEpiWarps); }
        s_abort = 0;
        mbar_fence_init();
    }
    if (warp == 2 && lane < 16) {
        mbar_init(smem_u32(&part_bar[lane >> 2][lane & 3]), 3);
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&s_tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);

    AttnItem item = {};
    int at = 0, at_end = 1;
    if constexpr (NL > 1) {                                    // the CTA's piece of the line of key tiles
        at = (int)((long long)ab.first[NL] * blockIdx.x / gridDim.x);
        at_end = (int)((long long)ab.first[NL] * (blockIdx.x + 1) / gridDim.x);
    }
    if (warp == 0) {
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (elect_one()) { prefetch_tmap(&ab.q[l]); prefetch_tmap(&ab.k[l]); }
        __syncwarp();
        int it = 0, n = 0;                                 // as in the stats kernel
        bool ok = true;
        for (; ok && colsum_item(ab, at, at_end, item); ++n) {
            const AttnMmaDims& dm = ab.lv[item.level].dm;
            const CUtensorMap *tmQ = &ab.q[item.level], *tmK = &ab.k[item.level];
            const int qb = n % kQBufs;
            const uint32_t qph = (uint32_t)(n / kQBufs) & 1u;
            if (!mbar_wait_warp(smem_u32(&q_free_bar[qb]), qph ^ 1u, abort_flag)) { ok = false; break; }
            if (elect_one()) {
                mbar_arrive_expect_tx(smem_u32(&q_bar[qb]), kQBytes);
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
                    tma_load_2d(q_addr + qb * kQBytes + kb * kQBlk, tmQ, kb * 64, item.g * dm.R + item.row * NQ, smem_u32(&q_bar[qb]));
            }
            __syncwarp();
            for (int t = item.t_lo; t < item.t_lo + item.nt; ++t, ++it) {
                const int s = it % stages;
                const uint32_t ph = (uint32_t)(it / stages) & 1u;
                if (!mbar_wait_warp(smem_u32(&empty_bar[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t fb = smem_u32(&full_bar[s]);
                const bool held = dbg_withhold(status, kDbgAttnColsum) && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && it == 0;   // debug builds: one copy never sent
                if (elect_one()) {
                    mbar_arrive_expect_tx(fb, kKBytes);
                    if (!held) {
#pragma unroll
                        for (int kb = 0; kb < KB; ++kb)
                            tma_load_2d(k_addr(s) + kb * kKBlk, tmK, kb * 64, item.g * dm.S + t * kCsBM, fb);
                    }
                }
                __syncwarp();
            }
        }
        for (int j = n > kQBufs ? n - kQBufs : 0; j < n; ++j)
            mbar_wait_warp(smem_u32(&q_bar[j % kQBufs]), (uint32_t)(j / kQBufs) & 1u, abort_flag);
        for (int back = 1; back <= stages && back <= it; ++back) {
            const int j = it - back;
            mbar_wait_warp(smem_u32(&full_bar[j % stages]), (uint32_t)(j / stages) & 1u, abort_flag);
        }
    } else if (warp == 1) {
        const uint32_t idesc = make_idesc_bf16(kCsBM, NQ);
        bool ok = true;
        int it = 0;
        for (int n = 0; ok && colsum_item(ab, at, at_end, item); ++n) {
            const int qb = n % kQBufs;
            ok = mbar_wait_warp(smem_u32(&q_bar[qb]), (uint32_t)(n / kQBufs) & 1u, abort_flag);
            for (const int end = it + item.nt; it < end && ok; ++it) {
                const int b = it & 1, s = it % stages;
                if (!mbar_wait_warp(smem_u32(&tempty_bar[b]), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                if (!mbar_wait_warp(smem_u32(&full_bar[s]), (uint32_t)(it / stages) & 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)b * kCsMaxNQ;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < DH / 16; ++kk) {
                        const uint64_t ad = make_desc_k128(k_addr(s) + (kk >> 2) * kKBlk + (kk & 3) * 32);
                        const uint64_t bd = make_desc_k128(q_addr + qb * kQBytes + (kk >> 2) * kQBlk + (kk & 3) * 32);
                        umma_bf16(d_tmem, ad, bd, idesc, kk != 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&empty_bar[s]));
                    umma_commit(smem_u32(&tfull_bar[b]));
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit(smem_u32(&q_free_bar[qb]));
            __syncwarp();
        }
        if (!ok) {
            if (elect_one()) umma_commit(smem_u32(&drain_bar));
            __syncwarp();
            mbar_wait_warp(smem_u32(&drain_bar), 0u, abort_flag);
        }
    } else {
        // The epilogue warps first turn the key-split partials into the log-sum-exp of the chunk's
        // query rows, two threads per row, while the producer's first copies and the first MMA are
        // already under way; nobody else reads s_nlse, so a barrier among these threads is enough.
        // (Of all the CTA's items at once: between items nothing else would hide it.)
        auto normalisers = [&](int at) {
            static_assert(kEpiWarps * 32 == 2 * kCsMaxNQ, "two threads per row");
            AttnItem x = {};
            for (int n = 0; n < kItems && colsum_item(ab, at, at_end, x); ++n) {
                const AttnLevel& lv = ab.lv[x.level];
                const AttnMmaDims& dm = lv.dm;
                const int c = (threadIdx.x - 64) >> 1, odd = threadIdx.x & 1;   // two threads per row: its even and its odd splits
                const int r = x.row * NQ + c;
                const bool row = c < NQ && r < dm.R;
                const int ns2 = row ? dm.st_nsplit : 0;            // one (max, sum) pair per key split
                const float* pm = lv.part_m + (size_t)x.g * dm.st_nsplit * dm.R + r;
                const float* pl = lv.part_l + (size_t)x.g * dm.st_nsplit * dm.R + r;
                float M = kNegInf, Z = 0.f;                        // running maximum and sum, partials in order
                for (int s0 = odd; s0 < ns2; s0 += 16) {
                    float m8[8], l8[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const bool in = s0 + 2 * u < ns2;
                        m8[u] = in ? pm[(size_t)(s0 + 2 * u) * dm.R] : kNegInf;
                        l8[u] = in ? pl[(size_t)(s0 + 2 * u) * dm.R] : 0.f;
                    }
                    float Mn = M;
#pragma unroll
                    for (int u = 0; u < 8; ++u) Mn = fmaxf(Mn, m8[u]);
                    Z *= exp2f(M - Mn);
#pragma unroll
                    for (int u = 0; u < 8; ++u) Z += l8[u] * exp2f(m8[u] - Mn);
                    M = Mn;
                }
                const float Mo = __shfl_xor_sync(0xFFFFFFFFu, M, 1), Zo = __shfl_xor_sync(0xFFFFFFFFu, Z, 1);
                const float Mn = fmaxf(M, Mo);
                const float ze = odd ? Zo : Z, me = odd ? Mo : M, zo = odd ? Z : Zo, mo = odd ? M : Mo;
                Z = ze * exp2f(me - Mn) + zo * exp2f(mo - Mn);
                // rows past R contribute exp2(x - 3e38) = 0
                if (!odd) s_nlse[n][c] = row ? -(Mn + log2f(Z)) : kNegInf;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
        };
        bool ok = true;
        int done = 0;                                          // tiles so far
        for (int n = 0; colsum_item(ab, at, at_end, item); ++n) {
            const AttnLevel& lv = ab.lv[item.level];
            const AttnMmaDims& dm = lv.dm;
            const int chunk = item.row, g = item.g, t_lo = item.t_lo, nt = item.nt;
            if (n % kItems == 0) {
                if (n > 0) asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");   // nobody reads the ones before any more
                normalisers(NL > 1 ? at - nt : 0);
            }
            const int quad = warp & 3;
            const int part = (warp - 2) >> 2;                      // column quarter
            const int width = NQ >> 2, c_lo = part * width;        // 8 .. 64 columns
            const float sc = dm.scale_log2;
            const uint64_t sc2 = pair(sc, sc);
            const int vis_end = dm.vis_start + dm.n_vis;
            float* plane = lv.part_col + (size_t)(g * dm.cs_nchunk + chunk) * dm.n_vis;
            for (int it = 0; it < nt; ++it, ++done) {
                const int b = done & 1;
                if (ok && !mbar_wait(smem_u32(&tfull_bar[b]), (uint32_t)(done >> 1) & 1u, abort_flag)) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                float sum;
                {
                    tc_fence_after();
                    // the whole quarter into registers, so that the accumulator is free before the arithmetic (columns past
                    // the quarter are loaded too, and not used)
                    const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * kCsMaxNQ + c_lo);
                    uint32_t raw[2][32];
                    tmem_ld32_issue(taddr, raw[0]);
                    if (width > 32) tmem_ld32_issue(taddr + 32u, raw[1]);
                    tmem_ld32_wait(raw[0]);
                    tmem_ld32_wait(raw[1]);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[b]));
                    uint64_t s0 = 0ull, s1 = 0ull;                 // {0.f, 0.f}
                    const float* nlse = &s_nlse[n % kItems][c_lo];
                    // the quarter's n columns, a constant in each case: no branch between them, so that their exponentials overlap
                    auto fold = [&](auto n_) {
                        constexpr int n = decltype(n_)::value;
#pragma unroll
                        for (int c = 0; c < n; c += 4) {
                            const uint32_t* r = &raw[c >> 5][c & 31];
                            const ulonglong2 nl = *reinterpret_cast<const ulonglong2*>(nlse + c);
                            const uint64_t x0 = fma_pair(pair(__uint_as_float(r[0]), __uint_as_float(r[1])), sc2, nl.x);
                            const uint64_t x1 = fma_pair(pair(__uint_as_float(r[2]), __uint_as_float(r[3])), sc2, nl.y);
                            s0 = add_pair(s0, exp2_pair(x0));
                            s1 = add_pair(s1, (c & 4) ? exp2_fma_pair<false>(x1) : exp2_pair(x1));   // every fourth pair on the FMA pipe; no logit is above the row's log-sum-exp
                        }
                    };
                    switch (width >> 3) {
                        case 1: fold(Int<8>()); break;
                        case 2: fold(Int<16>()); break;
                        case 3: fold(Int<24>()); break;
                        case 4: fold(Int<32>()); break;
                        case 5: fold(Int<40>()); break;
                        case 6: fold(Int<48>()); break;
                        case 7: fold(Int<56>()); break;
                        default: fold(Int<64>()); break;
                    }
                    float a0, a1;
                    unpair(add_pair(s0, s1), a0, a1);
                    sum = a0 + a1;
                }
                // The four quarters meet at the first one's warp, in quarter order.  Four buffers: whoever is at tile it + 4 has
                // its accumulator from the first quarter's warps, which gave it back at tile it + 2, after tile it.  (A
                // barrier of all 16 warps per tile put their loads and their arithmetic in step: 92 us at 73 728 keys.)
                const int slot = done & 3, col = quad * 32 + lane;
                const uint32_t pb = smem_u32(&part_bar[slot][quad]);
                if (part > 0) {
                    s_part[slot][part - 1][col] = sum;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(pb);
                } else {
                    if (ok && !mbar_wait(pb, (uint32_t)(done >> 2) & 1u, abort_flag)) ok = false;
                    const int u = (t_lo + it) * kCsBM + col;
                    if (ok && u >= dm.vis_start && u < vis_end)
                        plane[u - dm.vis_start] = ((sum + s_part[slot][0][col]) + s_part[slot][1][col]) + s_part[slot][2][col];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0 && s_abort) *status = METOK_ERR_TIMEOUT;
}

template <int DH, int NL>
int launch_levels(const AttnScoreCall* calls, int n, int Hq, int Hkv, int Lt, float scale, int32_t* status, cudaStream_t st) {
    AttnBatch<NL> stats, colsum;
    const uint64_t qrows = (uint64_t)Hq * Lt;
    int n_st = 0, n_cs = 0, rc;
    for (int l = 0; l < NL; ++l) {
        const AttnScoreCall& c = calls[l < n ? l : 0];            // a level that is not there has no items
        const AttnMmaDims dm = make_mma_dims(Hq, Hkv, Lt, c.S, c.vis_start, c.n_vis, scale);
        const uint64_t krows = (uint64_t)Hkv * c.S;
        if ((rc = make_tmap_bf16_2d(&stats.q[l], c.q_text, qrows, DH, kStBM)) != METOK_OK) return rc;
        if ((rc = make_tmap_bf16_2d(&stats.k[l], c.k_all, krows, DH, kStBN)) != METOK_OK) return rc;
        if ((rc = make_tmap_bf16_2d(&colsum.q[l], c.q_text, qrows, DH, (uint32_t)dm.cs_nq)) != METOK_OK) return rc;
        if ((rc = make_tmap_bf16_2d(&colsum.k[l], c.k_all, krows, DH, kCsBM)) != METOK_OK) return rc;
        stats.lv[l] = colsum.lv[l] = {dm, c.part_m, c.part_l, c.part_col};
        stats.first[l] = n_st;
        colsum.first[l] = n_cs;
        if (l < n) {
            n_st += dm.st_nsplit * dm.st_nrt * Hkv;
            n_cs += dm.cs_tiles * dm.cs_nchunk * Hkv;
        }
    }
    stats.first[NL] = n_st;
    colsum.first[NL] = n_cs;
    constexpr int KB = DH / 64;
    const int cs_nq = colsum.lv[0].dm.cs_nq;
    const size_t smem_st = (size_t)KB * ((NL > 1 ? 2 : 1) * kStBM + kStStages * kStBN) * 128 + 1024;
    const size_t smem_cs = (size_t)KB * (NL > 1 ? 2 * cs_nq + cs_stages(cs_nq, DH) * kCsBM : cs_nq + kCsStages * kCsBM) * 128 + 1024;
    METOK_ALLOW_SMEM((attn_stats_mma_kernel<DH, NL>), smem_st);
    METOK_ALLOW_SMEM((attn_colsum_mma_kernel<DH, NL>), smem_cs);
    {
        METOK_TIMED("attn_stats_mma_kernel", st);
        const AttnMmaDims& dm = stats.lv[0].dm;
        const dim3 grid = NL == 1 ? dim3(dm.st_nsplit, dm.st_nrt, Hkv) : dim3(std::min(n_st, kNumSMs));
        launch_chained(attn_stats_mma_kernel<DH, NL>, grid, dim3(kThreads), smem_st, st, stats, status);
    }
    METOK_LAUNCH_CHECK();
    {
        METOK_TIMED("attn_colsum_mma_kernel", st);
        const AttnMmaDims& dm = colsum.lv[0].dm;
        const dim3 grid = NL == 1 ? dim3(dm.cs_nsplit, dm.cs_nchunk, Hkv) : dim3(std::min(ceil_div(n_cs, kCsMinTiles), kNumSMs));
        launch_chained(attn_colsum_mma_kernel<DH, NL>, grid, dim3(kThreads), smem_cs, st, colsum, status);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

}  // namespace

void attn_mma_workspace(int Hq, int Hkv, int Lt, int S, int n_vis, size_t* n_part_ml, size_t* n_part_col,
                        int* n_planes) {
    const AttnMmaDims dm = make_mma_dims(Hq, Hkv, Lt, S, 0, n_vis, 1.f);
    *n_part_ml = (size_t)Hkv * dm.st_nsplit * dm.R;
    *n_planes = Hkv * dm.cs_nchunk;
    *n_part_col = (size_t)(*n_planes) * n_vis;
}

int launch_attn_scores_mma(const AttnScoreCall* calls, int n, int Hq, int Hkv, int Lt, int dh, float scale, int32_t* status,
                           cudaStream_t st) {
    if (n < 1 || n > kMaxPruneLevels) return METOK_ERR_INVALID_ARG;
    if (dh == 128)
        return n == 1 ? launch_levels<128, 1>(calls, n, Hq, Hkv, Lt, scale, status, st)
                      : launch_levels<128, kMaxPruneLevels>(calls, n, Hq, Hkv, Lt, scale, status, st);
    if (dh == 64)
        return n == 1 ? launch_levels<64, 1>(calls, n, Hq, Hkv, Lt, scale, status, st)
                      : launch_levels<64, kMaxPruneLevels>(calls, n, Hq, Hkv, Lt, scale, status, st);
    return METOK_ERR_UNSUPPORTED;
}

}  // namespace metok
