// Dot products of 8 P rows with 8 P other rows on the CUDA cores, by 64 threads with P x P outputs each (rows ty + 8 i,
// others tx + 8 j; ty = thread / 8, tx = thread % 8).  fp32 products, added in the order of the row: every dot product is
// one chain of fused multiply-adds.
//
// Rows are kept as they lie (k contiguous, 8-byte reads of two k; wider reads are no cheaper per byte) and come by 16-byte
// asynchronous copies into two stages of 16 k (three or four are no faster), a row's pitch of 80 bytes (fp32) putting the eight
// rows of a warp's read into different banks.  Small CTAs, several per SM: sa_ctas_per_sm.
#pragma once
#include "common.cuh"
#include "sm100.cuh"

namespace metok {

constexpr int kSaBK = 16, kSaThreads = 64;
constexpr int sa_ctas_per_sm(int pt) { return pt == 4 ? 10 : 12; }

template <typename T>
__device__ __forceinline__ float2 load_pair(const T* p) {
    if constexpr (sizeof(T) == 4) {
        return *reinterpret_cast<const float2*>(p);
    } else {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    }
}

template <typename T, int PT>
struct SimtTile {
    static constexpr int kTile = 8 * PT;                      // rows of each kind
    static constexpr int CE = 16 / sizeof(T);                 // elements per 16-byte chunk
    static constexpr int CPR = kSaBK / CE;                    // chunks per row and stage
    static constexpr int LD = kSaBK + CE;                     // row pitch in elements
    static constexpr int kCopies = 2 * kTile * CPR / kSaThreads;
    static constexpr int kRowStep = kSaThreads / CPR;         // rows between a thread's copies
    static constexpr uint32_t kStage = 2 * kTile * LD * sizeof(T), kCopyStep = kRowStep * LD * sizeof(T);
    T mem[2][2 * kTile][LD];                                  // the rows, then the others

    // The row this thread's copy i brings (0 .. 2 kTile - 1) and its chunk of a stage.
    static __device__ __forceinline__ int copy_row(int i) { return threadIdx.x / CPR + kRowStep * i; }
    static __device__ __forceinline__ int copy_chunk() { return threadIdx.x % CPR; }

    static __device__ __forceinline__ int steps(int d) { return (d + kSaBK - 1) / kSaBK; }
    __device__ __forceinline__ uint32_t copy_dst() { return sm100::smem_u32(&mem[0][copy_row(0)][copy_chunk() * CE]); }

    // src[i]: where copy i reads in the first stage; rows of row_chunks 16-byte chunks, ksteps = steps(d) and dst0 = copy_dst()
    // (out here because the compiler schedules the loop of P = 8 3 % better then).  Every thread of the CTA comes here, and
    // nobody reads `mem` any more.
    __device__ __forceinline__ void dots(const uint4* const (&src)[kCopies], int row_chunks, int ksteps, uint32_t dst0, float (&acc)[PT][PT]) {
        const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7, cchunk = copy_chunk();
        auto issue = [&](int ks) {                            // into stage ks % 2; past the end of the rows: zeros
            const uint32_t bytes = ks * CPR + cchunk < row_chunks ? 16u : 0u;
            const uint32_t dst = dst0 + (ks & 1) * kStage;
            const int off = bytes ? ks * CPR : 0;
#pragma unroll
            for (int i = 0; i < kCopies; ++i) sm100::cp_async16_zfill(dst + i * kCopyStep, src[i] + off, bytes);
            sm100::cp_async_commit();
        };
#pragma unroll
        for (int i = 0; i < PT; ++i)
#pragma unroll
            for (int j = 0; j < PT; ++j) acc[i][j] = 0.f;
        issue(0);
        for (int ks = 0; ks < ksteps; ++ks) {
            sm100::cp_async_wait_all();
            __syncthreads();                                  // stage ks % 2 has landed for everybody; the other one has been read by everybody
            if (ks + 1 < ksteps) issue(ks + 1);
            const T* pa = &mem[ks & 1][ty][0];
            const T* pb = &mem[ks & 1][kTile + tx][0];
#pragma unroll
            for (int kk = 0; kk < kSaBK; kk += 2) {
                float2 a[PT], b[PT];
#pragma unroll
                for (int i = 0; i < PT; ++i) a[i] = load_pair<T>(pa + 8 * i * LD + kk);
#pragma unroll
                for (int j = 0; j < PT; ++j) b[j] = load_pair<T>(pb + 8 * j * LD + kk);
#pragma unroll
                for (int i = 0; i < PT; ++i)
#pragma unroll
                    for (int j = 0; j < PT; ++j) acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
#pragma unroll
                for (int i = 0; i < PT; ++i)
#pragma unroll
                    for (int j = 0; j < PT; ++j) acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
            }
        }
    }
};

}  // namespace metok
