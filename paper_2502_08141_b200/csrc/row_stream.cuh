// Rows of fp32 weights, streamed through a warp's own buffers in shared memory a chunk of 1024 (or 512) elements at a time.
//
// Everything that looks at a weight once (its error, its residual) is bound by memory as long as it gets by on a dozen
// instructions per element, and for that a lane has to hold half an absmax block: the block's maximum is then one shuffle away (with
// a block spread over sixteen lanes, 128 bits each, it takes a shuffle per element).  So the chunk passes through shared memory:
// asynchronous coalesced copies in, kRowDepth buffers deep, and lane l takes elements 32 l .. 32 l + 31, its eight 16-byte pieces in an
// order that keeps the lanes of a wavefront on different banks.
//
// A CTA of kRowWarps warps takes rows blockIdx.x, + gridDim.x, ...; the chunks of all its rows, numbered through, go to its warps in
// turn, and a warp's copies run ahead over the ends of rows.  With every row on eight warps the CTAs of a persistent grid end
// together, whatever their rows' precisions.  (A warp to a row at a time and a CTA to every eight of them, 5120 x 5120 at 85/15 %: 26.2 us for the
// error, this 19.5.)
#pragma once
#include "lowra_common.cuh"

namespace lowra {

constexpr int kRowWarps = 8;
constexpr int kRowDepth = 3;       // buffers per warp: two chunks under way while one is worked on
// PER: elements per lane, 32 or 16; a chunk is 32 * PER elements.  32 spread a chunk's fixed cost further (error of 4096 x 4096 at 60/35/5 %:
// 14.5 against 16.7 us); 16 where they leave a quarter of the lanes less without work (K = 512: 4.9 against 5.7 us).
constexpr int row_ctas(int per) { return per == 32 ? 2 : 3; }   // CTAs per SM
inline int row_per_lane(int K) { return (K + 511) / 512 == 1 || (K + 511) / 512 == 3 ? 16 : 32; }

// A warp's place in the CTA's numbered chunks: row number i (of the CTA's rows) and chunk j of it.
struct RowPlace {
    int i, j;
};
struct RowWalk {
    int per_row, step_i, step_j;   // chunks per row; a warp's next chunk is kRowWarps further on
    __device__ RowWalk(int K, int chunk) : per_row((K + chunk - 1) / chunk), step_i(kRowWarps / per_row), step_j(kRowWarps % per_row) {}
    __device__ RowPlace start(int warp) const { return RowPlace{warp / per_row, warp % per_row}; }
    __device__ void next(RowPlace& p) const {
        p.i += step_i;
        p.j += step_j;
        if (p.j >= per_row) { p.j -= per_row; ++p.i; }
    }
};

__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// L2 policy of what is read or written once
__device__ __forceinline__ uint64_t once_policy() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void copy16_once(void* dst, const void* src, uint64_t policy) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "l"(policy) : "memory");
}

// the chunk at src (valid elements, a multiple of 128) on its way into buf
template <int PER>
__device__ __forceinline__ void chunk_copy(unsigned char* buf, const float* src, int valid, int lane, uint64_t policy) {
#pragma unroll
    for (int u = 0; u < PER / 4; ++u) {
        const int e = 4 * (32 * u + lane);
        if (e < valid) copy16_once(buf + 4 * e, src + e, policy);
    }
}
// byte offset of 16-byte piece t of this lane's elements: all of them for every lane, in an order of its own
template <int PER>
__device__ __forceinline__ int piece_at(int t, int lane) { return 4 * PER * lane + 16 * (t ^ (PER == 32 ? lane & 7 : (lane >> 1) & 3)); }

}  // namespace lowra
