// One row's 64-element absmax block from codes to bf16, in registers: what the kernels that feed the tensor cores share.
// A Scaled<B> holds the row's 2^B levels multiplied by the block's absmax and rounded to bf16 (exactly as lowra_decode does),
// in the form in which expand16 picks them: sixteen elements, two per word (the earlier one in the low half).
//   1 bit : both patterns differ by d; one multiply-add forms two elements (3 instructions a pair);
//   2 bits: the four patterns are two words, and one byte permute picks a pair out of them; what that needs - the codes c of
//           the pair as the nibbles 2 c, 2 c + 1 - comes from two multiplications for every two pairs;
//   4 bits: the low and the high bytes of the sixteen patterns are four words each; a byte permute looks four codes up, further ones put the
//           bytes together, the fourth bit of a code choosing between the halves of the table (a table in shared memory costs 9 and two loads).
// What bounds it: the half-rate pipe that permutes, shifts and logic share, the multiplications being on another.  Cycles of a scheduler for a
// block of 64 elements of 32 rows: 194 at 1 bit, 201 at 2 (258 with low and high bytes looked up by themselves, as at 4 bits), 438 at 4 (468 with four
// codes at a time and masked selectors).
#pragma once

#include "lowra_common.cuh"

namespace lowra {

// PRMT with a selector whose nibbles are known to be below 8 (__byte_perm masks them)
__device__ __forceinline__ uint32_t pick_bytes(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

template <int B> struct Scaled;
template <> struct Scaled<1> {
    // Both halves: the pattern L of level 0; H - L modulo 2^32, which may be negative: L + b (H - L), for a bit b, is one of the two patterns, so nothing is
    // carried from the low half to the high one, whichever is the larger.
    uint32_t base, d;
    __device__ __forceinline__ void set(const float* y, float a) {
        const uint32_t LH = pack_bf16x2(__fmul_rn(y[0], a), __fmul_rn(y[1], a)), L = LH & 0xFFFFu;
        base = L * 0x10001u; d = (LH >> 16) - L;
    }
    // elements 16 q .. 16 q + 15 of the block whose codes are w[0 .. 1]
    __device__ __forceinline__ void expand16(const uint32_t* w, int q, uint32_t (&o)[8]) const {
        const uint32_t h = (q & 1) ? (w[q >> 1] >> 16) : (w[q >> 1] & 0xFFFFu);
        const uint32_t z = h | (h << 15);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = ((z >> (2 * i)) & 0x10001u) * d + base;
    }
};
template <> struct Scaled<2> {
    uint32_t p01, p23;       // the four patterns
    __device__ __forceinline__ void set(const float* y, float a) {
        p01 = pack_bf16x2(__fmul_rn(y[0], a), __fmul_rn(y[1], a));
        p23 = pack_bf16x2(__fmul_rn(y[2], a), __fmul_rn(y[3], a));
    }
    __device__ __forceinline__ void expand16(const uint32_t* w, int q, uint32_t (&o)[8]) const {
#pragma unroll
        for (int k = 0; k < 4; ++k) {   // pairs k and 4 + k: their codes in a byte each, times 2, and that plus 1 beside it
            const uint32_t c = (((w[q] >> (4 * k)) & 0x000F000Fu) * 0x41u) & 0x03030303u, sel = c * 0x22u + 0x10101010u;
            o[k] = pick_bytes(p01, p23, sel);
            o[4 + k] = pick_bytes(p01, p23, sel >> 16);
        }
    }
};
template <> struct Scaled<4> {
    uint32_t lo[4], hi[4];   // low and high bytes of the sixteen patterns
    __device__ __forceinline__ void set(const float* y, float a) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t p = pack_bf16x2(__fmul_rn(y[4 * i], a), __fmul_rn(y[4 * i + 1], a));
            const uint32_t r = pack_bf16x2(__fmul_rn(y[4 * i + 2], a), __fmul_rn(y[4 * i + 3], a));
            lo[i] = __byte_perm(p, r, 0x6420u);
            hi[i] = __byte_perm(p, r, 0x7531u);
        }
    }
    __device__ __forceinline__ void expand16(const uint32_t* w, int q, uint32_t (&o)[8]) const {
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // eight codes at a time
            const uint32_t x = w[2 * q + h], sel = x & 0x77777777u, top = (x >> 3) & 0x11111111u;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t sl = i ? sel >> 16 : sel;
                const uint32_t upper = pick_bytes(0x0000FF00u, 0u, i ? top >> 16 : top);   // 0xFF where the code is 8 or more
                const uint32_t l = (pick_bytes(lo[0], lo[1], sl) & ~upper) | (pick_bytes(lo[2], lo[3], sl) & upper);
                const uint32_t u = (pick_bytes(hi[0], hi[1], sl) & ~upper) | (pick_bytes(hi[2], hi[3], sl) & upper);
                o[4 * h + 2 * i] = __byte_perm(l, u, 0x5140u);
                o[4 * h + 2 * i + 1] = __byte_perm(l, u, 0x7362u);
            }
        }
    }
};

}  // namespace lowra
