// Merge-assign of fp32 features on the tensor cores.  Included by vision.cu after the member lists.
//
// A float is the sum of three bf16 numbers, its leading, middle and trailing eight significant bits (x = h + m + l exactly,
// by truncation), so a product of two floats is the sum of nine products of bf16 numbers, each exact in the tensor core's
// fp32.  Six are made: hh, hm, mh, mm, hl, lh; the three left out (ml, lm, ll) are below 2^-21 of the product, 2^-24.5 of it on
// average, and have its sign: similarities near one are 4e-8 too low, all of them.  What would lose precision is the
// accumulator, which the tensor core cuts off instead of rounding: the sums of hh are therefore taken out of tensor memory after
// every two steps, four additions, and added up in registers with rounding, and the other five, 2^-8 of the whole, have an
// accumulator of their own.
//
// Which of several key tokens that are nearly alike is the most similar is decided by the fp32 chain all the same.  The tensor cores
// find, for every token, the key with the largest similarity and the others that are within f3_margin of it; where there are any
// (a few per cent of the tokens where frames differ by a tenth, nearly all in still video), these products are made again as one
// chain of fused multiply-adds and the largest is taken, by merge_join_f32_kernel, or for tokens with too many of them by
// merge_assign_simt_kernel, which has the same chains.
//
// merge_planes_kernel writes the three planes of every token into the workspace, the tokens that are no key tokens and the key
// tokens of an event apart, in the order and the swizzle in which a step's tiles lie in shared memory;
// merge_assign_f32_mma_kernel then brings a step of a unit in with two bulk copies.  (Splitting the rows inside the second kernel,
// where they were needed, was bound by the latency of the scattered loads: 95 us at 61 x 169 tokens of 1156.)
#pragma once

namespace metok {

constexpr int kF3BM = 128, kF3BN = 256, kF3BK = 32;           // most tokens and keys of a unit; elements per step
constexpr int kF3MaxStages = 8;
constexpr int kF3MinD = 60;                                   // narrowest rows that this has been compared with 64 bits at
// Steps whose hh add up in tensor memory.  A row of few steps has little else to round: one, or its error would be above that
// of the CUDA cores' chain.  Relative error of the cosines against 64 bits, root mean square (largest), chain / here: width
// 60: 5.5e-8 (6.3e-7) / 4.6e-8 (2.8e-7); 96: 6.1e-8 / 5.2e-8; 512: 7.7e-8 (1.3e-6) / 4.3e-8 (3.6e-7); 1156: 1.5e-7 (1.6e-6) / 8.3e-8
// (5.7e-7); 2048: 1.8e-7 / 1.1e-7; 3580: 2.3e-7 (2.9e-6) / 1.7e-7 (9.6e-7).  One step everywhere costs 2.5 us at 61 x 169 x 1156.
__device__ __forceinline__ int f3_segment(int d) { return d < 96 ? 1 : 2; }
constexpr int kF3EpiWarps = 16, kF3Threads = kF3EpiWarps * 32 + 64;
constexpr uint32_t kF3RowBytes = 3 * kF3BK * 2;               // a row's share of a step: three planes
constexpr uint32_t kF3ABytes = kF3BM * kF3RowBytes, kF3RingBytes = 3 * (kF3ABytes + kF3BN * kF3RowBytes);
constexpr size_t kF3SmemBytes = kF3RingBytes + 1024;
constexpr int kF3Events = 512;                                // up to as many events' offsets are kept in shared memory

// Where the planes of an event lie.  Tokens that are no key tokens: tiles of 128 rows, the event's first at f3_tile0; a tile is
// [step][plane][128 rows][64 bytes].  Key tokens: groups of 16 rows, the first at f3_group0; a unit's keys are whole groups,
// [step][plane][rows][64 bytes].  Both are rounded down from the rows before the event, plus one per event before, so that
// events never overlap whatever their sizes.
__host__ __device__ inline long long f3_tile0(long long rest_before, int e) { return rest_before / kF3BM + e; }
__host__ __device__ inline long long f3_group0(long long keys_before, int e) { return keys_before / 16 + e; }
__host__ __device__ inline int f3_steps(int d) { return (d + kF3BK - 1) / kF3BK; }
__host__ __device__ inline size_t f3_a_bytes(long long Nv, int k, int d) { return (size_t)(f3_tile0(Nv, k) + 1) * kF3ABytes * f3_steps(d); }
__host__ __device__ inline size_t f3_b_bytes(long long cap, int k, int d) { return (size_t)(f3_group0(cap, k) + 1) * 16 * kF3RowBytes * f3_steps(d); }
struct F3Planes { uint8_t *a, *b; };

// The chain's error and the tensor cores' together, twice (for the two keys that are compared), and something to spare.  Measured, not
// proven: the largest errors of a cosine against 64 bits are, chain + here, for Gaussian rows of very different size 6.3e-7 + 2.8e-7 at
// width 60 (margin 4.1e-6), 1.6e-6 + 5.7e-7 at 1156 (3.8e-5), 2.9e-6 + 9.6e-7 at 3580 (1.2e-4), for uniform and rectified ones no
// more; in rows of nearly equal elements all additions of a chain round one way and it is off by up to 9.1e-7, 1.7e-5 and 5.3e-5 (1.5e-8
// times the width), which is what the second term is for.  (Without it such rows took other keys than on the CUDA cores; it costs
// 0.3 us of 111 at 61 x 169 x 1156, 2.4 of 155 at 24 x 144 x 3584.)
__device__ __forceinline__ float f3_margin(int d) { return 1.0e-6f + fmaxf(4.0e-7f * sqrtf((float)d), 3.2e-8f * (float)d); }
// A token's candidates beside the best one so far (best64, whose packing they share): at most kF3Cands are listed, and a
// count of kF3All or more stands for all keys of the event (a norm that is no finite number).  Key tokens that are copies
// of one another (frames that repeat) would fill the lists: of those with the same similarity and the same hash the first counts.
// The hash is a sum over a row's 16-byte pieces, each multiplied with keys of its place: a sum of the bits alone, whatever their
// weights, is the same for rows of few significant bits that differ (any even number of flipped signs), and such rows tie.
constexpr int kF3Cands = 31, kF3All = 1 << 30, kF3NonZero = 1 << 29;
// Inverse norms from here on are those of rows at or below the norms' lower clamp: zeros, mostly, for which all keys are alike.
// Where such a row is none of zeros, merge_planes_kernel adds kF3NonZero to its count.
constexpr float kF3TinyInv = 9.9e7f;
struct F3Cands {
    unsigned long long* list;                                 // [token][kF3Cands + 1]
    int32_t* count;                                           // [token], cleared with the merge's scratch
    unsigned long long* hash;                                 // [slot] of the key token's row and the inverse of its norm
    int32_t *suspects, *n_suspects;                           // the tokens whose count is not zero
};
// A piece's share: two products of pairs of words, each word with a key of its own that depends on the place.  A thread's sum of
// them is mixed once, so that the sums of different threads do not cancel.
__device__ __forceinline__ unsigned long long f3_piece(const uint4& x, uint32_t place) {
    uint32_t m = (place + 1u) * 0x6A09E667u;                  // odd constants: leading fractional bits of square roots
    m = (m ^ (m >> 15)) * 0xBB67AE85u;
    return (unsigned long long)(x.x + m * 0x3C6EF373u) * (x.y + m * 0xA54FF53Bu) +
           (unsigned long long)(x.z + m * 0x510E527Fu) * (x.w + m * 0x9B05688Du);
}
__device__ __forceinline__ unsigned long long f3_mix(unsigned long long z) {
    z = (z ^ (z >> 32)) * 0x1F83D9ABFB41BD6Bull;
    return z ^ (z >> 29);
}
__device__ __forceinline__ unsigned long long f3_pack(float v, int slot) {
    return ((unsigned long long)float_key(v) << 32) | (unsigned long long)(~(uint32_t)slot);
}
__device__ __forceinline__ float f3_value(unsigned long long p) {
    const uint32_t k = (uint32_t)(p >> 32);
    return __uint_as_float(k & 0x80000000u ? k & 0x7FFFFFFFu : ~k);
}
__device__ __forceinline__ int f3_slot(unsigned long long p) { return (int)~(uint32_t)p; }
__device__ __forceinline__ bool f3_push(const F3Cands& ca, int row, unsigned long long p, bool& fresh) {   // false: the list is full
    const int at = atomicAdd(&ca.count[row], 1);
    fresh |= at == 0;
    if (at >= kF3Cands) return false;
    ca.list[(size_t)row * (kF3Cands + 1) + at] = p;
    return true;
}

// What merge_join_f32_kernel leaves to merge_assign_simt_kernel: tokens to be done with all keys of their event, in `rest` (nobody
// reads what was there any more) from the event's first place on, in tiles of kF3AgainRows that are opened as they come.
constexpr int kF3AgainRows = 32, kF3UnitBits = 40;
struct F3Again {
    int32_t* rows;                                            // [event]: tokens in tiles
    unsigned long long* tiles;                                // tiles << kF3UnitBits | units (tile x chunk of kF3AgainRows keys)
    unsigned long long* next;                                 // units taken beyond the first of every CTA
    long long* unit0;                                         // [tile]: units before it
    int32_t *event, *place, *done;                            // [tile]: its event, its first row's place in `rest`, chunks done
};
__host__ __device__ inline size_t f3_again_tiles(long long Nv, int k) { return (size_t)(Nv / kF3AgainRows + k); }

// An event's key tokens in equal chunks of whole sixteens.
__device__ __forceinline__ int f3_chunk(int nk, int nchunks) { return ((nk + nchunks - 1) / nchunks + 15) & ~15; }
struct F3Unit {
    int at, rows, col0, cols;                                 // rest[at .. at + rows), slots [col0, col0 + cols)
    long long tile, group;                                    // its rows' tile, its keys' first group
};
__device__ __forceinline__ F3Unit f3_unit(int u, const int32_t* ev_unit_off, const int32_t* ev_lo, const int32_t* ev_out_off, int k, int N, int bn) {
    const int e = find_event(ev_unit_off, k, u);
    const int s0 = ev_out_off[e], nk = ev_out_off[e + 1] - s0, lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N;
    const int nchunks = (nk + bn - 1) / bn, size = f3_chunk(nk, nchunks);
    const int local = u - ev_unit_off[e], tile = local / nchunks, c = local - tile * nchunks;
    F3Unit x;
    x.at = lo + tile * kF3BM;
    x.rows = min(kF3BM, hi - nk - x.at);
    x.col0 = s0 + c * size;
    x.cols = min(size, nk - c * size);
    x.tile = f3_tile0(lo - s0, e) + tile;
    x.group = f3_group0(s0, e) + c * (size / 16);
    return x;
}

// A 64-byte-swizzled K-major tile: rows of 64 bytes, groups of eight rows 512 bytes apart.
__device__ __forceinline__ constexpr uint32_t desc_k64_hi() { return (uint32_t)(512 >> 4) | (1u << 14) | (4u << 29); }
__device__ __forceinline__ void umma_bf16_k64(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc, uint32_t accumulate) {
    const uint32_t a_lo = sm100::desc_k128_lo(a_addr), b_lo = sm100::desc_k128_lo(b_addr);
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_k64_hi()), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The three planes' four elements of x: two words each.
__device__ __forceinline__ void f3_split(const uint4& x, uint2& h, uint2& m, uint2& l) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
    uint32_t r1[4], r2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float a = __uint_as_float(w[i]) - __uint_as_float(w[i] & 0xFFFF0000u);
        r1[i] = __float_as_uint(a);
        r2[i] = __float_as_uint(a - __uint_as_float(r1[i] & 0xFFFF0000u));
    }
    h = make_uint2(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632));
    m = make_uint2(__byte_perm(r1[0], r1[1], 0x7632), __byte_perm(r1[2], r1[3], 0x7632));
    l = make_uint2(__byte_perm(r2[0], r2[1], 0x7632), __byte_perm(r2[2], r2[3], 0x7632));
}

// The planes of all tokens.  Four rows per warp, eight threads and 128 bytes of a row each, so that 256 bytes of a plane leave
// together; kF3Ahead steps of loads in flight per thread.  blockIdx.y: a share of the steps.  In a plane row r lies at
// r * 64 bytes and its 16-byte piece p at position p ^ (r / 2 % 4).
constexpr int kF3Ahead = 6;
__global__ void __launch_bounds__(256)
merge_planes_kernel(const float* __restrict__ feats, int Nv, int d, int N, const int32_t* ev_lo, int k, const int32_t* ev_out_off,
                    const float* __restrict__ inv_norm, TokenOut out, F3Planes pl, F3Cands ca, int bn, int steps_per_cta,
                    int32_t* __restrict__ status) {
    grid_dep_wait();
    __shared__ int32_t s_lo[kF3Events + 1], s_out[kF3Events + 1];
    const long long all = (long long)ev_lo[k] * N, first = (long long)ev_lo[0] * N;
    if (k <= kF3Events) {
        for (int i = threadIdx.x; i <= k; i += blockDim.x) {
            s_lo[i] = ev_lo[i];
            s_out[i] = ev_out_off[i];
        }
        __syncthreads();
        ev_lo = s_lo;
        ev_out_off = s_out;
    }
    const long long i = (long long)blockIdx.x * 32 + (threadIdx.x >> 3);   // a place: an event's other tokens, then its key tokens
    if (i < first || i >= all) return;
    const int e = find_event(ev_lo, k, (int)(i / N));
    const int s0 = ev_out_off[e], nk = ev_out_off[e + 1] - s0, lo = ev_lo[e] * N, nr = ev_lo[e + 1] * N - lo - nk, x = (int)i - lo;
    uint8_t* dst;
    uint32_t plane;                                           // bytes of a plane; three of them are a step
    int r, row, slot = -1;
    if (x < nr) {
        r = x % kF3BM;
        row = out.rest[lo + x];
        dst = pl.a + (size_t)(f3_tile0(lo - s0, e) + x / kF3BM) * kF3ABytes * f3_steps(d);
        plane = kF3BM * 64;
    } else {
        const int j = x - nr, nchunks = (nk + bn - 1) / bn, size = f3_chunk(nk, nchunks), c = j / size;
        r = j - c * size;
        slot = s0 + j;
        row = out.out_src[slot];
        dst = pl.b + (size_t)(f3_group0(s0, e) + c * (size / 16)) * 16 * kF3RowBytes * f3_steps(d);
        plane = (uint32_t)((min(size, nk - c * size) + 15) & ~15) * 64u;
    }
    row = (int)dbg_bound(row, all, status);
    const int c = threadIdx.x & 7;
    dst += (uint32_t)r * 64u + (uint32_t)(((c >> 1) ^ ((r >> 1) & 3)) << 4) + (uint32_t)(c & 1) * 8u;
    const float* src = feats + (size_t)row * d + c * 4;
    const int k_lo = (int)blockIdx.y * steps_per_cta, k_hi = min(f3_steps(d), k_lo + steps_per_cta);
    unsigned long long hash = 0;
    const float inv = inv_norm[row];
    uint32_t bits = 0u;                                       // of all elements, without their signs
    for (int k0 = k_lo; k0 < k_hi; k0 += kF3Ahead) {
        uint4 v[kF3Ahead];
#pragma unroll
        for (int u = 0; u < kF3Ahead; ++u) {                  // the last step may reach past d (a multiple of 4): zeros there
            const int at = (k0 + u) * kF3BK;
            v[u] = k0 + u < k_hi && at + c * 4 < d ? __ldg(reinterpret_cast<const uint4*>(src + at)) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kF3Ahead; ++u) {
            if (k0 + u >= k_hi) continue;
            if (slot >= 0) hash += f3_piece(v[u], (uint32_t)((k0 + u) * 8 + c));
            bits |= (v[u].x | v[u].y | v[u].z | v[u].w) << 1;
            uint2 h, m, l;
            f3_split(v[u], h, m, l);
            uint8_t* o = dst + (size_t)(k0 + u) * 3 * plane;
            *reinterpret_cast<uint2*>(o) = h;
            *reinterpret_cast<uint2*>(o + plane) = m;
            *reinterpret_cast<uint2*>(o + 2 * plane) = l;
        }
    }
    if (slot >= 0) {                                          // (the eight threads of a row are in one case)
        const uint32_t row_lanes = 0xFFu << (threadIdx.x & 24);
        hash = f3_mix(hash + (c == 0 && k_lo == 0 ? __float_as_uint(inv) : 0u));
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) hash += __shfl_xor_sync(row_lanes, hash, o);
        if (c == 0) atomicAdd(&ca.hash[slot], hash);
    }
    if (inv >= kF3TinyInv && bits) atomicOr(&ca.count[row], kF3NonZero);
}

// Work unit = up to 128 of an event's tokens that are no key tokens x up to 256 of its key tokens (equal chunks of its keys);
// a persistent CTA takes every gridDim-th unit of the list of all events.
//   warp 16    : brings a step's tiles in, one bulk copy for the tokens and one for the keys;
//   warp 17    : issues tcgen05.mma (M = 128, N = the chunk's keys, K = 16), twelve per step of 32 elements: hh last, so that its
//                accumulator may still be read while the others of the next step are made;
//   warps 0-15 : epilogue, four TMEM lane quadrants x four quarters of the columns: a thread adds up 64 columns of its row, scales
//                them by 1/|key| and takes their (value, slot) argmax; the quarters and the chunks of a row meet in a 64-bit atomicMax
//                (larger value, then lower slot), and whichever of two falls behind there, or beside it in the quarter, by less
//                than the margin is listed.
// Shared memory bounds it: a step of 128 x 256 writes 72 KB and its products read 144 KB, 0.89 us at 128 bytes a clock beside 0.84
// us of tensor time.  Every wait is bounded; on a timeout the CTA unwinds and writes METOK_ERR_TIMEOUT.
__global__ void __launch_bounds__(kF3Threads, 1)
merge_assign_f32_mma_kernel(int d, int N, const int32_t* ev_lo, int k, const int32_t* ev_out_off,
                            const int32_t* ev_unit_off, const float* __restrict__ inv_norm, TokenOut out, F3Planes pl, F3Cands ca, int bn,
                            int32_t* __restrict__ status) {
    grid_dep_wait();
    using namespace sm100;
    const int32_t *out_src = out.out_src, *rest = out.rest;
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t full_bar[kF3MaxStages], empty_bar[kF3MaxStages], hfull_bar, hempty_bar, sfull_bar, sempty_bar, drain_bar;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ __align__(16) float s_keyinv[2][kF3BN];
    const int total_units = ev_unit_off[k];
    if ((int)blockIdx.x >= total_units) return;
    const int ksteps = f3_steps(d), segment = f3_segment(d), nseg = (ksteps + segment - 1) / segment;
    const uint32_t stage_bytes = kF3ABytes + (uint32_t)bn * kF3RowBytes;
    const int stages = min(kF3MaxStages, (int)(kF3RingBytes / stage_bytes));
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        mbar_init(smem_u32(&hfull_bar), 1);
        mbar_init(smem_u32(&hempty_bar), kF3EpiWarps);
        mbar_init(smem_u32(&sfull_bar), 1);
        mbar_init(smem_u32(&sempty_bar), kF3EpiWarps);
        mbar_init(smem_u32(&drain_bar), 1);
        s_abort = 0;
        mbar_fence_init();
    }
    if (warp == kF3EpiWarps + 1) {
        tmem_alloc(smem_u32(&s_tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;                   // columns 0 ..: the sums of hh, 256 ..: the others'
    volatile int* abort_flag = &s_abort;

    // The loops of these two warps: the whole warp takes every step and one elected thread issues, so that stage, addresses and
    // descriptors stay in uniform registers (see merge_assign_mma_kernel; 61 x 169 tokens of 1156: 140.0 -> 136.5 us the whole path).
    const int units = __shfl_sync(0xFFFFFFFFu, total_units, 0);
    if (warp == kF3EpiWarps) {
        int s = 0, issued = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const F3Unit un = f3_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, bn);
            const uint32_t b_bytes = (uint32_t)((un.cols + 15) & ~15) * kF3RowBytes;
            const uint8_t* a = pl.a + (size_t)un.tile * kF3ABytes * ksteps;
            const uint8_t* b = pl.b + (size_t)un.group * 16 * kF3RowBytes * ksteps;
            for (int ks = 0; ks < ksteps; ++ks, a += kF3ABytes, b += b_bytes) {
                if (!mbar_wait_warp(smem_u32(&empty_bar[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t fb = smem_u32(&full_bar[s]), dst = smem_base + (uint32_t)s * stage_bytes;
                if (elect_one()) {
                    mbar_arrive_expect_tx(fb, kF3ABytes + b_bytes);
                    bulk_load(dst, a, kF3ABytes, fb);
                    if (!(dbg_withhold(status, kDbgMergeAssign) && blockIdx.x == 0 && issued == 0))   // debug builds: one copy never sent
                        bulk_load(dst + kF3ABytes, b, b_bytes, fb);
                }
                __syncwarp();
                ++issued;
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
        }
        // every copy has landed before the CTA's shared memory goes away
        for (int back = 1; back <= stages && back <= issued; ++back) {
            const int j = issued - back;
            mbar_wait_warp(smem_u32(&full_bar[j % stages]), (uint32_t)(j / stages) & 1u, abort_flag);
        }
    } else if (warp == kF3EpiWarps + 1) {
        int s = 0, n = 0, seg = 0;                            // stage; units and segments so far
        uint32_t ph = 0;
        bool ok = true;
        const uint32_t d_hh = __shfl_sync(0xFFFFFFFFu, tmem_base, 0), d_small = d_hh + kF3BN;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++n) {
            const F3Unit un = f3_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, bn);
            const uint32_t cols = __shfl_sync(0xFFFFFFFFu, (uint32_t)(un.cols + 15) & ~15u, 0), idesc = make_idesc_bf16(kF3BM, (int)cols);
            constexpr uint32_t kA = kF3BM * 64;               // a plane of the tokens, and of the keys
            const uint32_t kB = cols * 64;
            for (int ks = 0; ks < ksteps; ++ks) {
                if (!mbar_wait_warp(smem_u32(&full_bar[s]), ph, abort_flag)) { ok = false; break; }
                if (ks == 0 && !mbar_wait_warp(smem_u32(&sempty_bar), ((uint32_t)n & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a = smem_base + (uint32_t)s * stage_bytes, b = a + kF3ABytes;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kF3BK / 16; ++kk) {
                        const uint32_t ah = a + 32u * kk, bh = b + 32u * kk;
                        umma_bf16_k64(d_small, ah + kA, bh + kB, idesc, ks > 0 || kk > 0 ? 1u : 0u);
                        umma_bf16_k64(d_small, ah, bh + 2 * kB, idesc, 1u);
                        umma_bf16_k64(d_small, ah + 2 * kA, bh, idesc, 1u);
                        umma_bf16_k64(d_small, ah, bh + kB, idesc, 1u);
                        umma_bf16_k64(d_small, ah + kA, bh, idesc, 1u);
                    }
                }
                __syncwarp();
                const bool opens = (ks & (segment - 1)) == 0;
                if (opens) {
                    if (!mbar_wait_warp(smem_u32(&hempty_bar), ((uint32_t)seg & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                }
                const bool closes = (ks & (segment - 1)) == segment - 1 || ks == ksteps - 1;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kF3BK / 16; ++kk) umma_bf16_k64(d_hh, a + 32u * kk, b + 32u * kk, idesc, !opens || kk > 0 ? 1u : 0u);
                    umma_commit(smem_u32(&empty_bar[s]));
                    if (closes) umma_commit(smem_u32(&hfull_bar));
                }
                __syncwarp();
                if (++s == stages) { s = 0; ph ^= 1u; }
                if (closes) ++seg;
            }
            if (ok && elect_one()) umma_commit(smem_u32(&sfull_bar));
            __syncwarp();
        }
        if (!ok) {                                            // wait until whatever was issued has retired
            if (elect_one()) umma_commit(smem_u32(&drain_bar));
            __syncwarp();
            mbar_wait_warp(smem_u32(&drain_bar), 0u, abort_flag);
        }
    } else {
        const int quad = warp & 3, part = warp >> 2;          // TMEM lanes 32 * quad ..., columns 64 * part ...
        const int et = threadIdx.x, c0 = 64 * part;
        bool ok = true;
        int n = 0, seg = 0;
        const float margin = f3_margin(d);
        for (int u = blockIdx.x; u < total_units; u += gridDim.x, ++n) {
            const F3Unit un = f3_unit(u, ev_unit_off, ev_lo, ev_out_off, k, N, bn);
            float* keyinv = s_keyinv[n & 1];                  // alternates: a slow warp may still read the last one
            if (et < kF3BN) keyinv[et] = et < un.cols ? inv_norm[out_src[un.col0 + et]] : 1.f;
            const int r = quad * 32 + lane;
            const int row = r < un.rows ? rest[un.at + r] : -1;
            const float rinv = row >= 0 ? inv_norm[row] : 1.f;
            named_bar_sync(1, kF3EpiWarps * 32);
            const bool mine = c0 < un.cols;                   // the same for the whole warp
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
            float sum[64];
#pragma unroll
            for (int j = 0; j < 64; ++j) sum[j] = 0.f;
            auto take = [&](uint32_t col, uint32_t bar, uint32_t parity, uint32_t free_bar) {
                if (ok && !mbar_wait(bar, parity, abort_flag)) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);             // tcgen05.ld below is warp-collective
                if (!ok) return;
                if (mine) {
                    tc_fence_after();
#pragma unroll
                    for (int x = 0; x < 64; x += 16) {
                        float v[16];
                        tmem_ld16(t_row + col + (uint32_t)x, v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) sum[x + j] += v[j];
                    }
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(free_bar);
            };
            for (int i = 0; i < nseg; ++i, ++seg) take(0u, smem_u32(&hfull_bar), (uint32_t)seg & 1u, smem_u32(&hempty_bar));
            take(kF3BN, smem_u32(&sfull_bar), (uint32_t)n & 1u, smem_u32(&sempty_bar));
            bool fresh = false;                               // the first to find something beside the best key of its token
            if (ok && mine && row >= 0) {
                float best_v = -3.4e38f, least = rinv;        // zero: a norm beyond the largest float, of the token or of a key
                int best_c = -1;
#pragma unroll
                for (int j = 0; j < 64; ++j) {
                    const float ki = keyinv[c0 + j], v = c0 + j < un.cols ? sum[j] * ki : -3.4e38f;
                    least = fminf(least, ki);
                    sum[j] = v;
                    if (v > best_v) { best_v = v; best_c = c0 + j; }
                }
                const bool whole = least == 0.f || rinv >= kF3TinyInv;
                if (whole) fresh = (atomicOr(&ca.count[row], kF3All) & ~kF3NonZero) == 0;
                if (best_c >= 0) {
                    const unsigned long long me = f3_pack(best_v, un.col0 + best_c), old = atomicMax(&out.best64[row], me);
                    const float old_v = old ? f3_value(old) : -3.4e38f, from = fmaxf(best_v, old_v) - margin / rinv;
                    bool room = !whole;
                    if (room && best_v >= from && old_v >= from && !(old_v == best_v && ca.hash[f3_slot(old)] == ca.hash[f3_slot(me)]))
                        room = f3_push(ca, row, old > me ? me : old, fresh);
                    uint32_t close[2] = {0u, 0u};             // the others of these columns
#pragma unroll
                    for (int j = 0; j < 64; ++j)
                        if (sum[j] >= from) close[j >> 5] |= 1u << (j & 31);
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
#pragma unroll 1
                        for (uint32_t left = close[w]; left && room; left &= left - 1) {
                            const int c = c0 + 32 * w + __ffs(left) - 1;
                            float v = 0.f;
#pragma unroll
                            for (int j = 32 * w; j < 32 * w + 32; ++j) v = c0 + j == c ? sum[j] : v;
                            if (c != best_c && c < un.cols && !(v == best_v && ca.hash[un.col0 + c] == ca.hash[f3_slot(me)]))
                                room = f3_push(ca, row, f3_pack(v, un.col0 + c), fresh);
                        }
                    }
                }
            }
            const uint32_t f = __ballot_sync(0xFFFFFFFFu, fresh);
            if (f) {
                int at = lane == 0 ? atomicAdd(ca.n_suspects, __popc(f)) : 0;
                at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(f & ((1u << lane) - 1u));
                if (fresh) ca.suspects[at] = row;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kF3EpiWarps + 1) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0 && s_abort) *status = METOK_ERR_TIMEOUT;
}

// A warp and its candidates' rows: lane j < nc <= G runs the chain of row `row` with row `key`.  Pieces of 16 float4s of the nc + 1
// rows come by 16-byte asynchronous copies into a ring of the warp's own, at a pitch that puts the candidates into different banks.
constexpr int kF3Piece = 16, kF3RingFloat4s = 4 * 9 * (kF3Piece + 1);   // four stages of 8 candidates, or two of 16
template <int G>
__device__ __forceinline__ float f3_chains(const float* __restrict__ feats, int d, int row, int key, int nc, float4* ring) {
    constexpr int kPitch = kF3Piece + 1, kStage = (G + 1) * kPitch, S = G == 8 ? 4 : 2, kCopies = G / 2 + 1;
    static_assert(S * kStage <= kF3RingFloat4s, "");
    const int lane = threadIdx.x & 31, half = lane >> 4, col = lane & 15, n4 = d >> 2, pieces = (n4 + kF3Piece - 1) / kF3Piece;
    const float4* src[kCopies];                               // rows half, half + 2, ...; row 0 is the token
#pragma unroll
    for (int i = 0; i < kCopies; ++i) {
        const int r = half + 2 * i, other = __shfl_sync(0xFFFFFFFFu, key, max(r, 1) - 1);
        src[i] = reinterpret_cast<const float4*>(feats + (size_t)(r == 0 ? row : other) * d) + col;
    }
    const uint32_t dst0 = sm100::smem_u32(ring + half * kPitch + col);
    auto issue = [&](int p, int stage) {
        if (p < pieces) {
            const uint32_t bytes = p * kF3Piece + col < n4 ? 16u : 0u;   // past the row's end: zeros, which change nothing
#pragma unroll
            for (int i = 0; i < kCopies; ++i)
                if (half + 2 * i <= nc)
                    sm100::cp_async16_zfill(dst0 + (uint32_t)(stage * kStage + 2 * i * kPitch) * 16u, bytes ? src[i] + p * kF3Piece : src[i], bytes);
        }
        sm100::cp_async_commit();
    };
    __syncwarp();                                             // the ring is free
#pragma unroll
    for (int p = 0; p < S; ++p) issue(p, p);
    float a = 0.f;
    int stage = 0;
    for (int p = 0; p < pieces; ++p) {
        sm100::cp_async_wait<S - 1>();
        __syncwarp();
        if (lane < nc) {
            const float4 *x = ring + stage * kStage, *y = x + (lane + 1) * kPitch;
#pragma unroll
            for (int i = 0; i < kF3Piece; ++i) {
                const float4 u = x[i], v = y[i];
                a = fmaf(u.w, v.w, fmaf(u.z, v.z, fmaf(u.y, v.y, fmaf(u.x, v.x, a))));
            }
        }
        __syncwarp();
        issue(p + S, stage);
        stage = stage + 1 == S ? 0 : stage + 1;
    }
    sm100::cp_async_wait<0>();
    return a;
}
// Every token to its key, and into that output's member list.  The last CTAs take the tokens without any candidate beside the
// best key, a thread each; the first ones take the others, a warp each: the candidates that are still within the margin of the best,
// and if there are several, their chains.  What bounds it is latency, five dependent loads and a chain of d multiply-adds, and with
// many candidates the reading of their rows, which tokens do not share.  A tile of merge_assign_simt_kernel reads all keys of the
// event, but for 32 tokens, and a key per token costs kF3KeysPerCand times less there (61 x 169 x 1156 in seven events, all
// tokens: nine candidates each 57 us, all 368 keys 205; 64 x 100 x 512: ten 23, all 250 keys 55); so a token with more than kF3Few
// candidates is left to it if that outweighs the keys that are none.  So are those whose list is full, and those with a norm
// that is no finite number.
// The call with frames of an event that differ by 0.1 / 0.01 / 0.001 / 0.0001, with a third of the tokens zero and with tokens
// that are all alike but for 0.001: 61 x 169 x 1156 in one event 271 / 337 / 446 / 1560 / 285 / 1578 us, on the CUDA cores 1346
// whatever they are; in seven 118 / 129 / 167 / 177 / 122 / 326, on the CUDA cores 257.  What is left above the CUDA cores is the
// planes and the products that decided nothing.
constexpr int kF3JoinWarps = 4, kF3Few = 8, kF3KeysPerCand = 12;
__device__ __forceinline__ void f3_join(const TokenOut& out, int slot, int row, int lo, int hi, int s0, int s1) {
    out.assign[row] = slot;
    if (slot >= s0 && slot < s1) members_join(out.ml, slot, row, row - lo, hi - lo);
}
__global__ void __launch_bounds__(kF3JoinWarps * 32, 4)
merge_join_f32_kernel(const float* __restrict__ feats, int Nv, int d, int N, const int32_t* ev_lo, int k, const int32_t* ev_out_off,
                      const float* __restrict__ inv_norm, TokenOut out, F3Cands ca, F3Again ag, int n_suspect_ctas) {
    grid_dep_wait();
    __shared__ int32_t s_lo[kF3Events + 1], s_out[kF3Events + 1];
    __shared__ float4 s_ring[kF3JoinWarps][kF3RingFloat4s];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool certain = (int)blockIdx.x >= n_suspect_ctas;
    const int first = certain ? ((int)blockIdx.x - n_suspect_ctas) * (kF3JoinWarps * 32) + (int)threadIdx.x
                              : (int)blockIdx.x + warp * n_suspect_ctas;   // token, or place among the suspects
    bool todo = first < Nv;
    int row = first, count = 0, total = 0;
    unsigned long long best = 0;
    if (certain) {
        if (todo) {                                           // (a key token's are not used)
            count = ca.count[row];
            best = out.best64[row];
            todo = !out.is_key[row];
        }
        todo = todo && (count & ~kF3NonZero) == 0;
    } else {
        total = *ca.n_suspects;
        row = todo ? ca.suspects[first] : 0;                  // with the total, which says whether it is one
    }
    if (k <= kF3Events) {
        for (int i = threadIdx.x; i <= k; i += kF3JoinWarps * 32) {
            s_lo[i] = ev_lo[i];
            s_out[i] = ev_out_off[i];
        }
        __syncthreads();
        ev_lo = s_lo;
        ev_out_off = s_out;
    }
    if (certain) {
        if (!todo) return;
        const int e = find_event(ev_lo, k, row / N), lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N;
        if (row >= lo && row < hi)                            // else a token of no event: its scratch is not this call's
            f3_join(out, best ? f3_slot(best) : -1, row, lo, hi, ev_out_off[e], ev_out_off[e + 1]);
        return;
    }
    float4* ring = s_ring[warp];
    for (int t = first; t < total; t += n_suspect_ctas * kF3JoinWarps) {
        if (t != first) row = ca.suspects[t];
        count = ca.count[row];
        const float inv = inv_norm[row];
        best = out.best64[row];
        unsigned long long x = ca.list[(size_t)row * (kF3Cands + 1) + lane];   // beyond the count: whatever was there
        const int e = find_event(ev_lo, k, row / N), lo = ev_lo[e] * N, hi = ev_lo[e + 1] * N, s0 = ev_out_off[e], s1 = ev_out_off[e + 1];
        // a row of zeros: its products are zeros, and best64 has the first key with one
        const bool zeros = inv >= kF3TinyInv && !(count & kF3NonZero), all = count > kF3Cands && !zeros;
        if (all || zeros || lane > count) x = 0ull;
        if (lane == (all || zeros ? 0 : count)) x = best;     // behind the candidates
        const bool near = x && f3_value(x) >= f3_value(best) - f3_margin(d) / inv;
        const uint32_t set = zeros ? 1u : __ballot_sync(0xFFFFFFFFu, near);
        const int n = __popc(set);
        if (all || (n > kF3Few && s1 - s0 < kF3KeysPerCand * n)) {
            if (lane == 0) {
                const int i = atomicAdd(&ag.rows[e], 1);
                out.rest[lo + i] = row;
                out.best64[row] = 0ull;
                if (i % kF3AgainRows == 0) {
                    const unsigned long long units = (unsigned long long)((s1 - s0 + kF3AgainRows - 1) / kF3AgainRows);
                    const unsigned long long was = atomicAdd(ag.tiles, (1ull << kF3UnitBits) + units);
                    const int at = (int)(was >> kF3UnitBits);
                    ag.unit0[at] = (long long)(was & ((1ull << kF3UnitBits) - 1ull));
                    ag.event[at] = e;
                    ag.place[at] = lo + i;
                    ag.done[at] = 0;
                }
            }
            continue;
        }
        if (n <= 1) {
            if (lane == 0) f3_join(out, best ? f3_slot(best) : -1, row, lo, hi, s0, s1);
            continue;
        }
        int* slots = reinterpret_cast<int*>(ring);            // the candidates to the first lanes
        __syncwarp();
        if (near) slots[__popc(set & ((1u << lane) - 1u))] = f3_slot(x);
        __syncwarp();
        const int slot = lane < n ? slots[lane] : 0, key = lane < n ? out.out_src[slot] : row;
        const float key_inv = inv_norm[key];
        unsigned long long won = 0;
        for (int c = 0; c < n;) {
            const bool few = n - c <= 8;
            const int nc = min(few ? 8 : 16, n - c), other = __shfl_sync(0xFFFFFFFFu, key, (c + lane) & 31);
            const float a = few ? f3_chains<8>(feats, d, row, other, nc, ring) : f3_chains<16>(feats, d, row, other, nc, ring);
            const float v = __shfl_sync(0xFFFFFFFFu, a, (lane - c) & 31) * key_inv;
            if (lane >= c && lane < c + nc && v > -3.4e38f) won = f3_pack(v, slot);
            c += nc;
        }
        const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(won >> 32));
        const uint32_t low = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(won >> 32) == top ? (uint32_t)won : 0u);
        if (lane == 0) f3_join(out, top ? (int)~low : -1, row, lo, hi, s0, s1);
    }
}

}  // namespace metok
