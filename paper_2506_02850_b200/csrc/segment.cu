// metok_segment_events: adjacent-frame cosine similarity (Eq. 4) and the split at
// the k-1 lowest similarities.
//
// FLATTEN mode is one streaming pass over V.  The flattened frame vector (N*d
// elements) is cut into slabs of 256 threads x 4 x 16 bytes; a CTA walks a run of
// consecutive frames of one slab, keeps the previous frame's chunks in registers
// and accumulates <v_f, v_f> and <v_f, v_{f+1}> in fp32.  Per-(slab, frame)
// partial sums go to the workspace and are added in a fixed order by the finishing
// kernel, so the result does not depend on scheduling.
#include <cooperative_groups.h>

#include "common.cuh"
#include "sm100.cuh"

namespace metok {

namespace cg = cooperative_groups;

constexpr int kSegThreads = 256;
constexpr int kSegUnroll = 4;     // 16-byte chunks per thread per frame
constexpr int kMaxFrames = 8192;

// Raw 16-byte chunk of either dtype, widened on use.
template <typename T>
__device__ __forceinline__ void widen16(const uint4& r, float (&v)[16 / sizeof(T)]) {
    if constexpr (sizeof(T) == 4) {
        v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y);
        v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    } else {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i]     = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
}

constexpr int kSegMaxRun = 16;    // frames per CTA at most
constexpr int kSegCtasPerSm = 4;  // by its registers

template <typename T>
__global__ void __launch_bounds__(kSegThreads, kSegCtasPerSm)
seg_partial_kernel(const T* __restrict__ feats, int Tn, long long chunks_per_frame, int frames_per_cta,
                   float* __restrict__ part_dot, float* __restrict__ part_nrm) {
    grid_dep_wait();
    constexpr int VN = Vec16<T>::N;
    constexpr int NW = kSegThreads / 32;
    __shared__ float s_nn[kSegMaxRun + 1][NW], s_dp[kSegMaxRun + 1][NW];
    const int slab = blockIdx.x;
    const int f0 = blockIdx.y * frames_per_cta;
    const int f1 = min(Tn, f0 + frames_per_cta);          // own frames [f0, f1)
    const int f_last = min(Tn - 1, f1);                   // halo frame for the last dot
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    long long chunk[kSegUnroll];
    bool ok[kSegUnroll];
#pragma unroll
    for (int u = 0; u < kSegUnroll; ++u) {
        chunk[u] = (long long)slab * (kSegThreads * kSegUnroll) + u * kSegThreads + tid;
        ok[u] = chunk[u] < chunks_per_frame;
    }
    const uint4* base = reinterpret_cast<const uint4*>(feats);
    auto fetch = [&](int f, uint4 (&r)[kSegUnroll]) {
        const uint4* frame = base + (size_t)f * (size_t)chunks_per_frame;
#pragma unroll
        for (int u = 0; u < kSegUnroll; ++u) r[u] = ok[u] ? __ldg(frame + chunk[u]) : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 prev[kSegUnroll], cur[kSegUnroll], nxt[kSegUnroll];   // raw chunks: widened when used
#pragma unroll
    for (int u = 0; u < kSegUnroll; ++u) prev[u] = make_uint4(0u, 0u, 0u, 0u);
    fetch(f0, cur);
    // the next frame's loads are in flight while this frame is reduced; nothing inside the
    // loop waits for another warp
    for (int f = f0; f <= f_last; ++f) {
        if (f < f_last) fetch(f + 1, nxt);
        float nn = 0.f, dp = 0.f;
#pragma unroll
        for (int u = 0; u < kSegUnroll; ++u) {
            float c[VN], p[VN];
            widen16<T>(cur[u], c);
            widen16<T>(prev[u], p);
#pragma unroll
            for (int e = 0; e < VN; ++e) {
                nn = fmaf(c[e], c[e], nn);
                dp = fmaf(c[e], p[e], dp);
            }
        }
        nn = warp_sum(nn);
        dp = warp_sum(dp);
        if (lane == 0) { s_nn[f - f0][warp] = nn; s_dp[f - f0][warp] = dp; }
#pragma unroll
        for (int u = 0; u < kSegUnroll; ++u) { prev[u] = cur[u]; cur[u] = nxt[u]; }
    }
    __syncthreads();
    // the warps' sums in warp order: <v_f, v_f> for own frames, <v_{f-1}, v_f> for every frame after the first
    const int nf = f_last - f0 + 1;
    if (tid < nf) {
        const int f = f0 + tid;
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) { a += s_nn[tid][w]; b += s_dp[tid][w]; }
        if (f < f1) part_nrm[(size_t)slab * Tn + f] = a;
        if (f > f0) part_dot[(size_t)slab * Tn + (f - 1)] = b;
    }
}

// MEANPOOL: mean over the N tokens of each frame, a thread per 16-byte column chunk, sixteen rows' loads in flight (one
// at a time, a thread's chain of N round trips was what the kernel lasted), added in row order.
constexpr int kMeanThreads = 64, kMeanRows = 16;
template <typename T>
__global__ void __launch_bounds__(kMeanThreads)
seg_mean_kernel(const T* __restrict__ feats, int N, int d, float* __restrict__ mean) {
    grid_dep_wait();
    constexpr int VN = Vec16<T>::N;
    const int f = blockIdx.y;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c * VN >= d) return;
    const T* base = feats + ((size_t)f * N) * d + (size_t)c * VN;
    float acc[VN];
    Vec16<T>::zero(acc);
    for (int p0 = 0; p0 < N; p0 += kMeanRows) {
        uint4 raw[kMeanRows];
#pragma unroll
        for (int u = 0; u < kMeanRows; ++u)
            if (p0 + u < N) raw[u] = __ldg(reinterpret_cast<const uint4*>(base + (size_t)(p0 + u) * d));
#pragma unroll
        for (int u = 0; u < kMeanRows; ++u) {
            if (p0 + u < N) {
                float v[VN];
                widen16<T>(raw[u], v);
#pragma unroll
                for (int e = 0; e < VN; ++e) acc[e] += v[e];
            }
        }
    }
    const float inv = 1.0f / (float)N;
#pragma unroll
    for (int e = 0; e < VN; ++e) mean[(size_t)f * d + c * VN + e] = acc[e] * inv;
}

// dot / norm of consecutive mean vectors: one CTA per frame, written as a single "slab".
__global__ void __launch_bounds__(256)
seg_meandot_kernel(const float* __restrict__ mean, int Tn, int d, float* __restrict__ part_dot,
                   float* __restrict__ part_nrm) {
    grid_dep_wait();
    __shared__ float red[2][8];
    const int f = blockIdx.x;
    const float* a = mean + (size_t)f * d;
    const float* b = mean + (size_t)(f + 1 < Tn ? f + 1 : f) * d;
    float nn = 0.f, dp = 0.f;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        nn = fmaf(a[i], a[i], nn);
        dp = fmaf(a[i], b[i], dp);
    }
    nn = warp_sum(nn);
    dp = warp_sum(dp);
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = nn; red[1][threadIdx.x >> 5] = dp; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float x = 0.f, y = 0.f;
        for (int w = 0; w < 8; ++w) { x += red[0][w]; y += red[1][w]; }
        part_nrm[f] = x;
        if (f + 1 < Tn) part_dot[f] = y;
    }
}

// Order-preserving key of a similarity; NaN (a non-finite frame) ranks above everything.
__device__ __forceinline__ uint32_t sim_key(float f) { return f != f ? 0xFFFFFFFFu : float_key(f); }

// Adds the slab partials in slab order, forms the cosines, picks the k-1 smallest
// (rank by counting; ties to the lower index) and writes boundaries, CSR offsets
// and per-frame event ids.  T <= kMaxFrames.  One CTA of 1024 threads, with more than 256 frames a cluster of four or eight
// whose CTAs add up their share of the frames' partials for everybody, rank their share of the frames and leave the
// flags with the first CTA, which does the rest: one CTA needs a sweep of dependent loads per 128 frames and T * T / 4
// comparisons (512 frames of 36 partials: 15.9 us under ncu, 9.4 with four).  The sums' order is the same.
inline int finish_ctas(int Tn) { return Tn <= 256 ? 1 : Tn <= 512 ? 4 : 8; }
template <bool kCl>
__global__ void __launch_bounds__(1024)
seg_finish_kernel(const float* __restrict__ part_dot, const float* __restrict__ part_nrm, int nslab,
                  int Tn, int k, float* __restrict__ sims, int32_t* __restrict__ boundaries,
                  int32_t* __restrict__ event_offsets, int32_t* __restrict__ frame_event) {
    const int C = kCl ? (int)gridDim.x : 1, crank = kCl ? (int)blockIdx.x : 0;
    if constexpr (kCl) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    grid_dep_wait();
    extern __shared__ float sm_f[];
    const int Tp = (Tn + 3) & ~3;
    float* s_sim = sm_f;                                   // [Tp]   (Tn-1 used)
    float* s_nrm = sm_f + Tp;                              // [Tp]   norms, later the similarities' keys
    uint32_t* s_simkey = reinterpret_cast<uint32_t*>(s_nrm);
    int* s_flag = reinterpret_cast<int*>(sm_f + 2 * Tp);   // [Tp]  boundary after frame i
    __shared__ int s_scan[32];
    const int tid = threadIdx.x, nthr = blockDim.x;

    // The partial sums: 128 consecutive frames per sweep, eight groups of 128 threads; a group takes the
    // slabs 8 apart, so a warp's load is 128 contiguous bytes of one slab (one CTA's L1 handles a sector
    // per cycle: whole sectors matter), six loads in flight; the eight groups' sums are then added in
    // group order.
    __shared__ float s_pn[8][128], s_pd[8][128];
    if constexpr (kCl) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // everybody has started
    for (int f0 = crank * 128; f0 < Tn; f0 += C * 128) {
        const int fl = tid & 127, part = tid >> 7;            // nthr == 1024
        const int f = f0 + fl;
        float a = 0.f, b = 0.f;
        if (f < Tn) {
            const bool has_dot = f < Tn - 1;
            constexpr int kB = 6;                           // loads in flight; the additions keep their order
            for (int s0 = part; s0 < nslab; s0 += 8 * kB) {
                float x[kB], y[kB];
#pragma unroll
                for (int u = 0; u < kB; ++u) {
                    const int s = s0 + 8 * u;
                    x[u] = s < nslab ? part_nrm[(size_t)s * Tn + f] : 0.f;
                    y[u] = s < nslab && has_dot ? part_dot[(size_t)s * Tn + f] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < kB; ++u) {
                    if (s0 + 8 * u < nslab) { a += x[u]; b += y[u]; }
                }
            }
        }
        s_pn[part][fl] = a;
        s_pd[part][fl] = b;
        __syncthreads();
        if (tid < 128 && f < Tn) {
            float an = 0.f, ad = 0.f;
#pragma unroll
            for (int g = 0; g < 8; ++g) { an += s_pn[g][tid]; ad += s_pd[g][tid]; }
            const float norm = fmaxf(sqrtf(an), kEps);
            if constexpr (!kCl) {
                s_nrm[f] = norm;
                s_sim[f] = ad;                              // dot product for now
            } else {
                for (int c = 0; c < C; ++c) {
                    cg::this_cluster().map_shared_rank(s_nrm, c)[f] = norm;
                    cg::this_cluster().map_shared_rank(s_sim, c)[f] = ad;
                }
            }
        }
        __syncthreads();
    }
    if constexpr (kCl) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    __syncthreads();
    // Integer keys give a total order even with non-finite similarities (a NaN ranks as the largest value), so exactly
    // k-1 boundaries are flagged whatever the input holds.
    for (int i = tid; i < Tn - 1; i += nthr) {
        const float c = s_sim[i] / (s_nrm[i] * s_nrm[i + 1]);
        s_sim[i] = c;
        if (crank == 0) sims[i] = c;
    }
    __syncthreads();
    for (int i = tid; i < Tp; i += nthr) s_simkey[i] = i < Tn - 1 ? sim_key(s_sim[i]) : 0xFFFFFFFFu;
    __syncthreads();
    // Rank by counting: P lanes share a frame, each compares it with every P-th group of four keys; in the groups before
    // the frame's own an equal key ranks lower, in those after it higher.  (One thread per frame, comparing floats one by
    // one: 25 us of this kernel at 512 frames.)
    const int nb = k - 1;
    const int share = (Tn + C - 1) / C, own_lo = min(Tn, crank * share), own_hi = min(Tn, own_lo + share);   // the frames this CTA ranks
    const int p_log2 = share > 512 ? 0 : share > 256 ? 1 : share > 128 ? 2 : 3, P = 1 << p_log2;
    int* flags = s_flag;
    if constexpr (kCl) flags = cg::this_cluster().map_shared_rank(s_flag, 0);
    for (int i0 = own_lo; i0 < own_hi; i0 += nthr >> p_log2) {
        const int i = i0 + (tid >> p_log2), part = tid & (P - 1);
        int rank = 0;
        if (i < own_hi && i < Tn - 1 && nb > 0) {
            const uint32_t v = s_simkey[i];
            const uint4* keys4 = reinterpret_cast<const uint4*>(s_simkey);
            const int own = i >> 2, nq = (Tn + 2) >> 2;
            int q = part;
#pragma unroll 4
            for (; q < own; q += P) {
                const uint4 w = keys4[q];
                rank += (w.x <= v) + (w.y <= v) + (w.z <= v) + (w.w <= v);
            }
            if (q == own) {
                const uint4 w = keys4[q];
                const int r = i & 3;
                rank += (w.x < v || (w.x == v && 0 < r)) + (w.y < v || (w.y == v && 1 < r)) + (w.z < v || (w.z == v && 2 < r)) + (w.w < v);
                q += P;
            }
#pragma unroll 4
            for (; q < nq; q += P) {
                const uint4 w = keys4[q];
                rank += (w.x < v) + (w.y < v) + (w.z < v) + (w.w < v);
            }
        }
        for (int o = 1; o < P; o <<= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, o);
        if (part == 0 && i < own_hi) flags[i] = i < Tn - 1 && rank < nb;
    }
    if constexpr (kCl) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (crank > 0) return;
    } else {
        __syncthreads();
    }
    // exclusive scan of the flags: contiguous ranges per thread, a shuffle scan inside each warp,
    // then the warps' totals
    const int per = (Tn + nthr - 1) / nthr;
    const int lo = min(Tn, tid * per), hi = min(Tn, lo + per);
    int local = 0;
    for (int i = lo; i < hi; ++i) local += s_flag[i];
    const int lane = tid & 31, warp = tid >> 5;
    int incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_scan[warp] = incl;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += s_scan[w];
    int run = before + incl - local;                       // boundaries before frame lo
    for (int i = lo; i < hi; ++i) {
        frame_event[i] = run;                              // event id = boundaries strictly before i
        if (s_flag[i] && run < nb) {
            boundaries[run] = i;
            event_offsets[run + 1] = i + 1;
            ++run;
        }
    }
    if (tid == 0) {
        event_offsets[0] = 0;
        event_offsets[k] = Tn;
    }
}

template <typename T>
static int launch_segment(const void* feats, int Tn, int N, int d, int k, int sim_mode, float* sims,
                          int32_t* boundaries, int32_t* event_offsets, int32_t* frame_event, void* ws,
                          cudaStream_t st) {
    constexpr int VN = 16 / sizeof(T);
    Carver cv(ws);
    int nslab;
    float *part_dot, *part_nrm;
    if (sim_mode == METOK_SIM_FLATTEN) {
        const long long chunks = (long long)N * d / VN;
        nslab = (int)((chunks + kSegThreads * kSegUnroll - 1) / (kSegThreads * kSegUnroll));
        // Frames per CTA: the run with the fewest frames read one after the other, over all rounds of CTAs; a CTA reads one
        // frame more than it owns and takes about another frame's time to start (64 x 196 x 1152: two frames a CTA were two
        // rounds, four are one; 375 x 256 x 1872: sixteen left the third round half empty, thirteen fill it).
        int fpc = 1;
        long long best = -1;
        for (int f = 1; f <= kSegMaxRun; ++f) {
            const long long ctas = (long long)nslab * ceil_div(Tn, f), rounds = (ctas + kSegCtasPerSm * kNumSMs - 1) / (kSegCtasPerSm * kNumSMs);
            const long long cost = rounds * (f + 2);
            if (best < 0 || cost <= best) { best = cost; fpc = f; }
        }
        part_dot = cv.take<float>((size_t)nslab * Tn);
        part_nrm = cv.take<float>((size_t)nslab * Tn);
        dim3 grid(nslab, ceil_div(Tn, fpc));
        {
            METOK_TIMED("seg_partial_kernel", st);
            launch_chained(seg_partial_kernel<T>, grid, dim3(kSegThreads), 0, st, reinterpret_cast<const T*>(feats), Tn, chunks, fpc,
                           part_dot, part_nrm);
        }
        METOK_LAUNCH_CHECK();
    } else {
        nslab = 1;
        part_dot = cv.take<float>((size_t)Tn);
        part_nrm = cv.take<float>((size_t)Tn);
        float* mean = cv.take<float>((size_t)Tn * d);
        dim3 grid(ceil_div(d / VN, kMeanThreads), Tn);
        {
            METOK_TIMED("seg_mean_kernel", st);
            launch_chained(seg_mean_kernel<T>, grid, dim3(kMeanThreads), 0, st, reinterpret_cast<const T*>(feats), N, d, mean);
        }
        METOK_LAUNCH_CHECK();
        {
            METOK_TIMED("seg_meandot_kernel", st);
            launch_chained(seg_meandot_kernel, dim3(Tn), dim3(256), 0, st, mean, Tn, d, part_dot, part_nrm);
        }
        METOK_LAUNCH_CHECK();
    }
    const size_t smem = (size_t)((Tn + 3) & ~3) * 3 * sizeof(float);
    if (smem > 32 * 1024)                                  // with the kernel's own 8.3 KB; more than 256 frames, so a cluster
        METOK_ALLOW_SMEM(seg_finish_kernel<true>, smem);
    {
        METOK_TIMED("seg_finish_kernel", st);
        launch_chained_clusters(finish_ctas(Tn), finish_ctas(Tn) > 1 ? seg_finish_kernel<true> : seg_finish_kernel<false>, dim3(finish_ctas(Tn)), dim3(1024), smem, st, part_dot, part_nrm, nslab, Tn, k, sims, boundaries, event_offsets,
                                             frame_event);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

}  // namespace metok

using namespace metok;

extern "C" size_t metok_segment_events_workspace_bytes(int dtype, int T, int N, int d, int sim_mode) {
    if (T < 1 || N < 1 || d < 1) return 0;
    const int VN = dtype == METOK_F32 ? 4 : 8;
    Carver cv(nullptr);
    if (sim_mode == METOK_SIM_FLATTEN) {
        const long long chunks = ((long long)N * d + VN - 1) / VN;
        const size_t nslab = (size_t)((chunks + kSegThreads * kSegUnroll - 1) / (kSegThreads * kSegUnroll));
        cv.take<float>(nslab * T);
        cv.take<float>(nslab * T);
    } else {
        cv.take<float>((size_t)T);
        cv.take<float>((size_t)T);
        cv.take<float>((size_t)T * d);
    }
    return cv.total();
}

extern "C" int metok_segment_events(const void* feats, int dtype, int T, int N, int d, int k, int sim_mode,
                                    float* sims, int32_t* boundaries, int32_t* event_offsets,
                                    int32_t* frame_event, void* ws, size_t ws_bytes, void* stream) {
    if (!feats || !sims || !boundaries || !event_offsets || !frame_event) return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (sim_mode != METOK_SIM_FLATTEN && sim_mode != METOK_SIM_MEANPOOL) return METOK_ERR_INVALID_ARG;
    if (T < 1 || N < 1 || d < 1 || k < 1 || k > T) return METOK_ERR_INVALID_ARG;
    if (!aligned16(feats) || (reinterpret_cast<uintptr_t>(sims) & 3) || (reinterpret_cast<uintptr_t>(boundaries) & 3) ||
        (reinterpret_cast<uintptr_t>(event_offsets) & 3) || (reinterpret_cast<uintptr_t>(frame_event) & 3))
        return METOK_ERR_INVALID_ARG;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (((long long)d * eb) % 16 != 0 || T > kMaxFrames) return METOK_ERR_UNSUPPORTED;
    const size_t need = metok_segment_events_workspace_bytes(dtype, T, N, d, sim_mode);
    if (!ws || ws_bytes < need || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (dtype == METOK_F32)
        return launch_segment<float>(feats, T, N, d, k, sim_mode, sims, boundaries, event_offsets, frame_event, ws, st);
    return launch_segment<__nv_bfloat16>(feats, T, N, d, k, sim_mode, sims, boundaries, event_offsets, frame_event,
                                         ws, st);
}

// --------------------------------------------------------------------------- //
// metok_segment_score_events: segmentation and the per-token text relevance of Eq. 5
// in ONE pass over V: per token row its squared norm, its dot product with the text
// embedding and its dot product with the same position's row of the previous frame.
// Token score and 1/norm are final in the kernel; the norms and dots of a frame leave it as sums over four
// neighbouring positions (of single positions in fp32 where there are few), which seg_finish adds up in a fixed order.
//
// fp32 rows (seg_score_kernel): a warp owns one token position and a run of frames (from 48 positions on the
// four warps of a CTA neighbouring positions and the same frames), holds
// the row in registers (the next row's loads in flight meanwhile) and the previous row in
// shared memory, and takes the three sums with multiply-adds.
//
// bf16 rows (seg_score_mma_kernel).  The multiply-add form costs 40 instructions per 16
// bytes (widening, three fma per element) and needs the whole row in registers, which
// leaves an SM with 12 warps.  Here the rows land in shared memory by 16-byte
// asynchronous copies (a ring of kFsDepth stages per warp, no registers held while in
// flight) and the sums run on the tensor cores.  A warp owns one position and
// EIGHT consecutive frames; a stage holds 512 contiguous bytes of those eight rows and
// of the frame before them (one copy instruction per row, 16 bytes per lane: the memory
// system sees long pieces of a row).  A stage is consumed as eight 64-byte slices, two m16n8k16 mma each, and all three
// sums come out of the same mma: B is the eight frames (columns), A the same eight frames (rows 0-7), the text (row 8) and
// the frame before the run (row 9; rows 10-15 repeat the text and are not read).  C then holds the squared norms on its
// diagonal, the dots of neighbouring frames next to it, <text, frame> in row 8 and the first frame's dot with its
// predecessor at C[9][0].  Lane (g, q) = (lane / 4, lane % 4) reads chunk q of frame g's slice (dwords m0..m3) and chunk q
// of row 8 + g (t0..t3); the order of k inside a dot product is free as long as both operands use the same one, so the
// first mma takes (m0, t0, m2, t2) as A and (m0, m2) as B, the second the odd dwords: nothing is rearranged between lanes.
// Products of bf16 are exact in fp32 and the sums are fp32 (an accumulator for the even dwords, one for the odd ones).
// The kernel is meant to be bound by HBM; with separate mma for each of the three sums (54 instructions per 64 bytes
// of a row, eight warps an SM) it was bound by instruction latency: 512 x 144 rows of 1024 in 41.7 us, 31 now; 128 x 144 of
// 3584 30.7 and 27.
// --------------------------------------------------------------------------- //
namespace metok {

constexpr int kFsThreads = 128;

// kTogether: the warps of a CTA take neighbouring positions of the same frames, and their norms and dots are added in the CTA, in
// warp order, so that seg_finish has a quarter of the partial sums to read (169 of them for 61 frames: 9.3 us, 6.2 with 43); an
// idle warp of a run's last CTA repeats the last position and counts nothing.  Otherwise every warp has a position and a run of
// its own and leaves sums of its own.
template <typename T, int kCH, bool kTogether>
__global__ void __launch_bounds__(kFsThreads, kCH <= 4 ? 7 : kCH <= 10 ? 4 : 3)
seg_score_kernel(const T* __restrict__ feats, const T* __restrict__ text, int Tn, int N, int d, int frames_per_warp,
                 float* __restrict__ part_dot, float* __restrict__ part_nrm, float* __restrict__ token_score,
                 float* __restrict__ inv_norm) {
    grid_dep_wait();
    constexpr int VN = Vec16<T>::N;
    extern __shared__ float s_t[];                 // [d], in planes of 4 floats per chunk (conflict-free 16-byte reads)
                                                   // then [warps][nchunk] raw 16-byte chunks: the previous frame's row
    __shared__ float s_red[kFsThreads / 32];
    __shared__ float s_tn;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nchunk = d / VN;
    for (int i = tid; i < d; i += kFsThreads) {
        const int c = i / VN, q = i % VN;
        s_t[(q >> 2) * (nchunk * 4) + c * 4 + (q & 3)] = to_float(text[i]);
    }
    __syncthreads();
    float a = 0.f;
    for (int i = tid; i < d; i += kFsThreads) a = fmaf(s_t[i], s_t[i], a);
    a = warp_sum(a);
    if (lane == 0) s_red[warp] = a;
    __syncthreads();
    if (tid == 0) {
        float sum = 0.f;
        for (int w = 0; w < kFsThreads / 32; ++w) sum += s_red[w];
        s_tn = fmaxf(sqrtf(sum), kEps);
    }
    __syncthreads();
    const float tn = s_tn;
    constexpr int kWarps = kFsThreads / 32;
    __shared__ float s_nn[kTogether ? 2 : 1][kWarps][32], s_dp[kTogether ? 2 : 1][kWarps][32];   // of 32 frames each
    const int pgroups = kTogether ? (N + kWarps - 1) / kWarps : N;
    const int at = kTogether ? blockIdx.x : blockIdx.x * kWarps + warp;
    const int run = at / pgroups, pg = at - run * pgroups;
    const bool mine = !kTogether || pg * kWarps + warp < N;
    const int p = !kTogether ? pg : mine ? pg * kWarps + warp : N - 1;
    const int f0 = run * frames_per_warp;
    if (!kTogether && f0 >= Tn) return;                     // behind the last run
    const int f1 = min(Tn, f0 + frames_per_warp);           // own frames [f0, f1)
    const int f_last = min(Tn - 1, f1);                     // halo frame for the last dot
    const uint4* base = reinterpret_cast<const uint4*>(feats);
    uint4* prev = reinterpret_cast<uint4*>(s_t + d) + (size_t)warp * nchunk;   // d floats = a multiple of 16 bytes
    uint4 cur[kCH], nxt[kCH];
#pragma unroll
    for (int u = 0; u < kCH; ++u) {
        const int c = u * 32 + lane;
        if (c < nchunk) prev[c] = make_uint4(0u, 0u, 0u, 0u);
    }
    auto fetch = [&](int f, uint4 (&r)[kCH]) {
        const uint4* x = base + ((size_t)f * N + p) * (size_t)nchunk;
#pragma unroll
        for (int u = 0; u < kCH; ++u) {
            const int c = u * 32 + lane;
            r[u] = c < nchunk ? __ldg(x + c) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    int flushed = 0;                                        // blocks of 32 frames that are added up
    auto flush = [&]() {
        __syncthreads();
        const int c = flushed++, f = f0 + c * 32 + lane;
        const float (*v)[32] = warp == 0 ? s_nn[c & 1] : s_dp[c & 1];
        if (warp < 2 && f < (warp == 0 ? f1 : f_last)) {
            float a = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) a += v[w][lane];
            (warp == 0 ? part_nrm : part_dot)[(size_t)pg * Tn + f] = a;
        }
    };
    fetch(f0, cur);
    // the next row's loads are in flight while this row is reduced
    for (int f = f0; f <= f_last; ++f) {
        const size_t row = (size_t)f * N + p;
        if (f < f_last) fetch(f + 1, nxt);
        float nn = 0.f, dt = 0.f, dp = 0.f;
#pragma unroll
        for (int u = 0; u < kCH; ++u) {
            const int c = u * 32 + lane;
            if (c < nchunk) {
                float v[VN], pv[VN];
                widen16<T>(cur[u], v);
                widen16<T>(prev[c], pv);
                prev[c] = cur[u];                           // a lane only ever touches its own chunks
#pragma unroll
                for (int h = 0; h < VN / 4; ++h) {
                    const float4 tt = reinterpret_cast<const float4*>(s_t + h * (nchunk * 4))[c];
                    nn = fmaf(v[4 * h + 0], v[4 * h + 0], nn); dt = fmaf(v[4 * h + 0], tt.x, dt); dp = fmaf(v[4 * h + 0], pv[4 * h + 0], dp);
                    nn = fmaf(v[4 * h + 1], v[4 * h + 1], nn); dt = fmaf(v[4 * h + 1], tt.y, dt); dp = fmaf(v[4 * h + 1], pv[4 * h + 1], dp);
                    nn = fmaf(v[4 * h + 2], v[4 * h + 2], nn); dt = fmaf(v[4 * h + 2], tt.z, dt); dp = fmaf(v[4 * h + 2], pv[4 * h + 2], dp);
                    nn = fmaf(v[4 * h + 3], v[4 * h + 3], nn); dt = fmaf(v[4 * h + 3], tt.w, dt); dp = fmaf(v[4 * h + 3], pv[4 * h + 3], dp);
                }
            }
        }
        nn = warp_sum(nn);
        dt = warp_sum(dt);
        dp = warp_sum(dp);
        const int i = f - f0;
        if (lane == 0 && i > 0) {                           // dot of frames f-1 and f at position p
            if constexpr (kTogether) s_dp[((i - 1) >> 5) & 1][warp][(i - 1) & 31] = mine ? dp : 0.f;
            else part_dot[(size_t)p * Tn + (f - 1)] = dp;
        }
        // A block of 32 frames is complete with the dot that reaches into the next one, and is added up before anything of the
        // next one is written: block c + 2's first entries, in the buffers of block c, then come after the barrier of block
        // c + 1, and whoever adds up block c has read it before that barrier.
        if (kTogether && i > 0 && (i & 31) == 0) flush();
        if (lane == 0 && f < f1) {
            const float n = fmaxf(sqrtf(nn), kEps);
            if constexpr (kTogether) s_nn[(i >> 5) & 1][warp][i & 31] = mine ? nn : 0.f;
            else part_nrm[(size_t)p * Tn + f] = nn;
            if (mine) {
                token_score[row] = dt / (n * tn);
                inv_norm[row] = 1.0f / n;
            }
        }
#pragma unroll
        for (int u = 0; u < kCH; ++u) cur[u] = nxt[u];
    }
    while (kTogether && flushed * 32 < f1 - f0) flush();
}

// D += A * B for one m16n8k16 bf16 tile, fp32 accumulators; A is a 16-byte chunk as loaded.
__device__ __forceinline__ void mma_bf16_m16n8k16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

constexpr int kFsCtasPerSm = 2;                    // what the rings leave room for
constexpr int kFsDepth = 4;                        // stages of a warp's ring
constexpr int kFsFrames = 8;                       // frames per warp = row groups of the mma tile
constexpr int kFsSlices = 8;                       // 64-byte slices of a row per stage: 512 contiguous bytes
constexpr int kFsRowPitch = kFsSlices * 64 + 64;   // bytes between a stage's rows (see the bank note in the kernel)
constexpr int kFsStageBytes = (kFsFrames + 1) * kFsRowPitch;

// Shared memory: the text embedding, zero-padded to whole slices; then per warp kFsDepth
// stages of nine rows (512 bytes of frame f0 - 1, then of frames f0 .. f0 + 7).
template <bool kFull>                               // kFull: the row is a whole number of 512-byte pieces
__global__ void __launch_bounds__(kFsThreads)
seg_score_mma_kernel(const __nv_bfloat16* __restrict__ feats, const __nv_bfloat16* __restrict__ text, int Tn, int N,
                     int d, float* __restrict__ part_dot, float* __restrict__ part_nrm,
                     float* __restrict__ token_score, float* __restrict__ inv_norm) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char s_dyn[];
    constexpr int kFsWarps = kFsThreads / 32;
    __shared__ float s_red[kFsWarps];
    __shared__ float s_tn;
    __shared__ float s_nn[2][kFsWarps][kFsFrames], s_dp[2][kFsWarps][kFsFrames];   // alternate from unit to unit
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nchunk = d / 8;
    const int nslice = (nchunk + 3) >> 2;
    const int nsuper = (nslice + kFsSlices - 1) / kFsSlices;
    uint4* s_text = reinterpret_cast<uint4*>(s_dyn);
    // A unit is eight frames of four consecutive positions, one per warp: their norms and dots are added in the CTA
    // (in warp order), so that seg_finish has a quarter of the partial sums to read.  Units run position first.
    const int pgroups = (N + kFsWarps - 1) / kFsWarps;
    const int nunits = pgroups * ((Tn + kFsFrames - 1) / kFsFrames);
    const int g = lane >> 2, q = lane & 3;
    const size_t frame_pitch = (size_t)N * nchunk;          // 16-byte chunks from a frame's row to the next frame's
    // Copies: a stage holds 512 contiguous bytes (eight 64-byte slices) of each of the nine rows -- the
    // frame before the run, then the run's eight frames.  One copy instruction moves a row's 512 bytes
    // (16 per lane), so what reaches the memory system is long contiguous pieces of a row.  Rows of a
    // stage lie kFsRowPitch bytes apart: with 16 words more than a multiple of 32 the 16-byte reads of
    // the eight lanes of a quarter warp (two frames, four chunks each) fall into different banks.
    unsigned char* ring = s_dyn + (size_t)nslice * 4 * sizeof(uint4) + (size_t)warp * kFsDepth * kFsStageBytes;
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + (uint32_t)lane * 16u;
    const unsigned char* mine = ring + (g + 1) * kFsRowPitch + q * 16;
    // row 8 + g of A: the frame before the run (g = 1) or the text
    const unsigned char* other = g == 1 ? ring + q * 16 : reinterpret_cast<const unsigned char*>(s_text) + q * 16;
    // the copies run kFsDepth - 1 pieces ahead of the sums, into the next units too
    int i_unit = blockIdx.x, i_left = 0, i_lo = 0, i_hi = 0;
    int i_chunk = lane;                                     // this lane's chunk of the next piece's rows
    uint32_t i_stage = 0;
    const uint4* i_src = nullptr;                           // that chunk of row i_lo, the first of the nine rows that exists
    auto issue_unit = [&]() {
        const int run = i_unit / pgroups;
        // an idle warp repeats the last position and writes nothing
        const int p = min((i_unit - run * pgroups) * kFsWarps + warp, N - 1);
        const int f0 = run * kFsFrames;
        i_lo = f0 == 0 ? 1 : 0;                             // row 0: the frame before the run
        i_hi = min(kFsFrames + 1, Tn - f0 + 1);
        i_left = nsuper;
        i_chunk = lane;
        i_src = reinterpret_cast<const uint4*>(feats) + ((size_t)(f0 - 1 + i_lo) * N + p) * (size_t)nchunk + lane;
    };
    auto issue = [&]() {                                    // one group per call
        if (i_unit < nunits) {
            const bool in = kFull || i_chunk < nchunk;
            const uint4* src = in ? i_src : reinterpret_cast<const uint4*>(feats);
            const size_t step = in ? frame_pitch : 0;
            const uint32_t to = dst + i_stage;
            if (i_hi - i_lo == kFsFrames + 1) {
#pragma unroll
                for (int r = 0; r <= kFsFrames; ++r, src += step) sm100::cp_async16_zfill(to + r * kFsRowPitch, src, in ? 16u : 0u);
            } else {                                        // rows that do not exist are written as zeros (0 bytes read)
#pragma unroll 1
                for (int r = 0; r <= kFsFrames; ++r) {
                    const bool ok = r >= i_lo && r < i_hi;
                    sm100::cp_async16_zfill(to + r * kFsRowPitch, src, ok && in ? 16u : 0u);
                    if (ok && r + 1 < i_hi) src += step;
                }
            }
            i_stage = i_stage == (kFsDepth - 1) * kFsStageBytes ? 0u : i_stage + kFsStageBytes;
            i_chunk += kFsSlices * 4;
            i_src += kFsSlices * 4;
            if (--i_left == 0) {
                i_unit += gridDim.x;
                if (i_unit < nunits) issue_unit();
            }
        }
        sm100::cp_async_commit();
    };
    if (i_unit < nunits) issue_unit();
#pragma unroll 1
    for (int j = 0; j < kFsDepth - 1; ++j) issue();

    float a = 0.f;
    for (int c = tid; c < nslice * 4; c += kFsThreads) {
        const uint4 r = c < nchunk ? __ldg(reinterpret_cast<const uint4*>(text) + c) : make_uint4(0u, 0u, 0u, 0u);
        s_text[c] = r;
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
            a = fmaf(lo, lo, a);
            a = fmaf(hi, hi, a);
        }
    }
    a = warp_sum(a);
    if (lane == 0) s_red[warp] = a;
    __syncthreads();
    if (tid == 0) {
        float sum = 0.f;
        for (int w = 0; w < kFsWarps; ++w) sum += s_red[w];
        s_tn = fmaxf(sqrtf(sum), kEps);
    }
    __syncthreads();
    const float tn = s_tn;

    uint32_t stage = 0;
    int par = 0;
#pragma unroll 1
    for (int unit = blockIdx.x; unit < nunits; unit += gridDim.x, par ^= 1) {
        const int run = unit / pgroups, pg = unit - run * pgroups;
        const int p = pg * kFsWarps + warp;
        const int f0 = run * kFsFrames;
        const int f = f0 + g;                               // this lane's frame
        const bool has = p < N && f < Tn;
        float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};   // even and odd dwords
#pragma unroll 1
        for (int sup = 0; sup < nsuper; ++sup) {
            sm100::cp_async_wait<kFsDepth - 2>();           // this lane's copies of the piece have landed
            __syncwarp();                                   // ... and every lane's; the piece before it has been read by all
            issue();                                        // into the stage that held the piece before
            const unsigned char* at = mine + stage;
            const unsigned char* at2 = other + (g == 1 ? (int)stage : sup * (kFsSlices * 64));
            stage = stage == (kFsDepth - 1) * kFsStageBytes ? 0u : stage + kFsStageBytes;
#pragma unroll
            for (int i = 0; i < kFsSlices; ++i) {
                if (kFull || sup * kFsSlices + i < nslice) {
                    const uint4 x = *reinterpret_cast<const uint4*>(at + i * 64);
                    const uint4 y = *reinterpret_cast<const uint4*>(at2 + i * 64);
                    mma_bf16_m16n8k16(acc[0], make_uint4(x.x, y.x, x.z, y.z), x.x, x.z);
                    mma_bf16_m16n8k16(acc[1], make_uint4(x.y, y.y, x.w, y.w), x.y, x.w);
                }
            }
        }
        // lane (g, q) holds columns 2q and 2q + 1 of rows g and 8 + g
        float c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] = acc[0][i] + acc[1][i];
        // <text, frame g> is C[8][g], in lane (0, g / 2)
        const float t0 = __shfl_sync(0xFFFFFFFFu, c[2], g >> 1), t1 = __shfl_sync(0xFFFFFFFFu, c[3], g >> 1);
        if (q == (g >> 1)) {                                // C[g][g]
            const float nn = g & 1 ? c[1] : c[0];
            s_nn[par][warp][g] = has ? nn : 0.f;
            if (has) {
                const size_t r = (size_t)f * N + p;
                const float n = fmaxf(sqrtf(nn), kEps);
                token_score[r] = (g & 1 ? t1 : t0) / (n * tn);
                inv_norm[r] = 1.0f / n;
            }
        }
        // s_dp[j]: frame f0 + j with the frame before it, C[j - 1][j]; for the run's first frame C[9][0]
        if (g < 7 && q == ((g + 1) >> 1)) s_dp[par][warp][g + 1] = p < N ? (g & 1 ? c[0] : c[1]) : 0.f;
        if (lane == 4) s_dp[par][warp][0] = p < N ? c[2] : 0.f;
        __syncthreads();
        if (tid < kFsFrames && f0 + tid < Tn) {
            float nn = 0.f, dp = 0.f;
#pragma unroll
            for (int w = 0; w < kFsWarps; ++w) { nn += s_nn[par][w][tid]; dp += s_dp[par][w][tid]; }
            const int ff = f0 + tid;
            part_nrm[(size_t)pg * Tn + ff] = nn;
            if (ff > 0) part_dot[(size_t)pg * Tn + (ff - 1)] = dp;    // dots of frames ff-1 and ff, four positions
        }
    }
    sm100::cp_async_wait_all();
}

// Frame runs sized so that all warps are resident at once: a second, partly filled wave of
// CTAs would cost as much time as the first.
template <typename KernelT>
static int seg_score_runs(KernelT kernel, size_t smem, int Tn, int N, int* frames_per_warp) {
    if (smem > 40 * 1024)
        METOK_ALLOW_SMEM(kernel, smem);
    int per_sm = 0;
    METOK_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kFsThreads, smem));
    const long long slots = (long long)kNumSMs * (per_sm > 0 ? per_sm : 1) * (kFsThreads / 32);
    long long nruns = slots / N;
    nruns = nruns < 1 ? 1 : nruns > Tn ? Tn : nruns;
    *frames_per_warp = ceil_div(Tn, (int)nruns);
    return METOK_OK;
}

template <typename T, int kCH>
static int launch_seg_score(const void* feats, const void* text, int Tn, int N, int d, int k, float* sims,
                            int32_t* boundaries, int32_t* event_offsets, int32_t* frame_event,
                            float* token_score, float* inv_norm, void* ws, cudaStream_t st) {
    Carver cv(ws);
    float* part_dot = cv.take<float>((size_t)N * Tn);
    float* part_nrm = cv.take<float>((size_t)N * Tn);
    int fpw = 1;
    int nslab = N;                                         // partial sums per frame that seg_finish adds up
    if constexpr (sizeof(T) == 2) {
        const int nslice = (d / 8 + 3) / 4;
        const size_t smem_t = (size_t)nslice * 4 * sizeof(uint4) + (size_t)(kFsThreads / 32) * kFsDepth * kFsStageBytes;
        auto kernel = (d / 8) % (4 * kFsSlices) == 0 ? seg_score_mma_kernel<true> : seg_score_mma_kernel<false>;
        if (smem_t > 40 * 1024)
            METOK_ALLOW_SMEM(kernel, smem_t);
        nslab = ceil_div(N, kFsThreads / 32);
        METOK_TIMED("seg_score_kernel", st);
        launch_chained(kernel, dim3(std::min(nslab * ceil_div(Tn, kFsFrames), kNumSMs * kFsCtasPerSm)), dim3(kFsThreads), smem_t, st,
            reinterpret_cast<const __nv_bfloat16*>(feats), reinterpret_cast<const __nv_bfloat16*>(text), Tn, N, d,
            part_dot, part_nrm, token_score, inv_norm);
    } else {
        const size_t smem_t = (size_t)d * sizeof(float) + (size_t)(kFsThreads / 32) * d * sizeof(T);
        // Few positions are few partial sums: adding them in the CTA then costs more, at its end and in idle warps, than
        // seg_finish gains.  The call with every warp alone / together, frames x positions x width: 400 x 1 x 2048 11.0 / 12.8 us,
        // 300 x 17 x 1156 15.0 / 16.4, 300 x 29 x 1024 16.4 / 18.4, 300 x 32 x 1156 19.7 / 20.4, 61 x 41 x 1156 11.0 / 11.4,
        // 150 x 49 x 1156 18.7 / 17.9, 61 x 61 x 1024 11.7 / 11.0, 61 x 169 x 1156 20.5 / 18.7.
        constexpr int kWarps = kFsThreads / 32;
        const bool together = N >= 48;
        auto kernel = together ? seg_score_kernel<T, kCH, true> : seg_score_kernel<T, kCH, false>;
        if (together) nslab = ceil_div(N, kWarps);
        const int rc = seg_score_runs(kernel, smem_t, Tn, together ? nslab * kWarps : N, &fpw);
        if (rc != METOK_OK) return rc;
        const int runs = ceil_div(Tn, fpw);
        METOK_TIMED("seg_score_kernel", st);
        launch_chained(kernel, dim3(together ? nslab * runs : ceil_div(N * runs, kWarps)), dim3(kFsThreads), smem_t, st,
            reinterpret_cast<const T*>(feats), reinterpret_cast<const T*>(text), Tn, N, d, fpw, part_dot, part_nrm,
            token_score, inv_norm);
    }
    METOK_LAUNCH_CHECK();
    const size_t smem = (size_t)((Tn + 3) & ~3) * 3 * sizeof(float);
    if (smem > 32 * 1024)                                  // with the kernel's own 8.3 KB; more than 256 frames, so a cluster
        METOK_ALLOW_SMEM(seg_finish_kernel<true>, smem);
    {
        METOK_TIMED("seg_finish_kernel", st);
        launch_chained_clusters(finish_ctas(Tn), finish_ctas(Tn) > 1 ? seg_finish_kernel<true> : seg_finish_kernel<false>, dim3(finish_ctas(Tn)), dim3(1024), smem, st, part_dot, part_nrm, nslab, Tn, k, sims, boundaries, event_offsets,
                                             frame_event);
    }
    METOK_LAUNCH_CHECK();
    return METOK_OK;
}

}  // namespace metok

extern "C" size_t metok_segment_score_events_workspace_bytes(int dtype, int T, int N, int d) {
    (void)dtype; (void)d;
    if (T < 1 || N < 1) return 0;
    Carver cv(nullptr);
    cv.take<float>((size_t)N * T);
    cv.take<float>((size_t)N * T);
    return cv.total();
}

extern "C" int metok_segment_score_events(const void* feats, int dtype, int T, int N, int d, int k,
                                          const void* text_emb, float* sims, int32_t* boundaries,
                                          int32_t* event_offsets, int32_t* frame_event, float* token_score,
                                          float* token_inv_norm, void* ws, size_t ws_bytes, void* stream) {
    if (!feats || !text_emb || !sims || !boundaries || !event_offsets || !frame_event || !token_score || !token_inv_norm)
        return METOK_ERR_INVALID_ARG;
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (T < 1 || N < 1 || d < 1 || k < 1 || k > T) return METOK_ERR_INVALID_ARG;
    if (!aligned16(feats) || !aligned16(text_emb)) return METOK_ERR_INVALID_ARG;
    const int eb = dtype == METOK_F32 ? 4 : 2;
    if (((long long)d * eb) % 16 != 0 || T > kMaxFrames) return METOK_ERR_UNSUPPORTED;
    const long long nchunk = (long long)d * eb / 16;
    if (nchunk > 32 * 16) return METOK_ERR_UNSUPPORTED;          // rows of more than 8 KiB: use the two separate calls
    const size_t need = metok_segment_score_events_workspace_bytes(dtype, T, N, d);
    if (!ws || ws_bytes < need || !aligned16(ws)) return METOK_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
#define METOK_FS(TYPE, CH)                                                                                        \
    return launch_seg_score<TYPE, CH>(feats, text_emb, T, N, d, k, sims, boundaries, event_offsets, frame_event, \
                                      token_score, token_inv_norm, ws, st)
    if (dtype == METOK_F32) {
        if (nchunk <= 32 * 4) METOK_FS(float, 4);
        if (nchunk <= 32 * 8) METOK_FS(float, 8);
        if (nchunk <= 32 * 10) METOK_FS(float, 10);              // four CTAs per SM, not three (61 x 169 rows of 1028 / 1156 / 1280: 22.0 / 23.1 / 23.0 -> 20.5 / 21.5 / 21.4 us; 256 x 144 x 1280: 51.4 -> 44.9)
        METOK_FS(float, 16);
    }
    METOK_FS(__nv_bfloat16, 4);                                  // the bf16 kernel has no per-width variants
#undef METOK_FS
}

// --------------------------------------------------------------------------- //
// metok_segment_events_static: the same computation with the scratch in a fixed
// array that lives inside the library image instead of a caller workspace.
// --------------------------------------------------------------------------- //
namespace metok {
constexpr size_t kStaticScratchBytes = (size_t)1 << 20;      // 1 MiB per GPU that loads the library
static __device__ __align__(256) unsigned char g_seg_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
static void* g_seg_scratch_addr[kMaxDevices] = {nullptr};    // device address of the array, per device

// `g_seg_scratch` in host code is only a handle; the address kernels can use has to be
// asked for, once per device, with that device current.
static int static_scratch_address(void** out, cudaStream_t st) {
    int dev = -1;
    METOK_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return METOK_ERR_UNSUPPORTED;
    if (!g_seg_scratch_addr[dev]) {
        // the look-up is not a stream operation: made while `st` is being captured it could end the
        // caller's capture, so the first call on a device has to come before any capture
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        METOK_CUDA_TRY(cudaStreamIsCapturing(st, &cs));
        if (cs != cudaStreamCaptureStatusNone) return METOK_ERR_UNSUPPORTED;
        void* p = nullptr;
        METOK_CUDA_TRY(cudaGetSymbolAddress(&p, g_seg_scratch));
        g_seg_scratch_addr[dev] = p;
    }
    *out = g_seg_scratch_addr[dev];
    return METOK_OK;
}
}  // namespace metok

extern "C" size_t metok_segment_events_static_capacity(void) { return metok::kStaticScratchBytes; }

extern "C" int metok_segment_events_static(const void* feats, int dtype, int T, int N, int d, int k, int sim_mode,
                                           float* sims, int32_t* boundaries, int32_t* event_offsets,
                                           int32_t* frame_event, void* stream) {
    if (dtype != METOK_F32 && dtype != METOK_BF16) return METOK_ERR_INVALID_ARG;
    if (T < 1 || N < 1 || d < 1) return METOK_ERR_INVALID_ARG;
    const size_t need = metok_segment_events_workspace_bytes(dtype, T, N, d, sim_mode);
    if (need > metok::kStaticScratchBytes) return METOK_ERR_TOO_LARGE;
    void* scratch = nullptr;
    const int rc = metok::static_scratch_address(&scratch, reinterpret_cast<cudaStream_t>(stream));
    if (rc != METOK_OK) return rc;
    return metok_segment_events(feats, dtype, T, N, d, k, sim_mode, sims, boundaries, event_offsets, frame_event,
                                scratch, metok::kStaticScratchBytes, stream);
}
