// One row's 64-element absmax block from codes to bf16, in registers: what the kernels that feed the tensor cores share.
// A Scaled<B> holds the row's 2^B levels multiplied by the block's absmax and rounded to bf16 (exactly as lowra_decode does),
// in the form in which expand16 picks them: sixteen elements, two per word (the earlier one in the low half).
//   1 bit : both patterns differ by d; one multiply-add forms two elements (3 instructions a pair);
//   2 bits: the low and the high bytes of the four patterns are a word each; a byte permute looks four codes up, further
//           ones put the bytes of neighbouring elements together (3.6 instructions a pair; picking 16-bit patterns pair by pair, 6);
//   4 bits: likewise with four words each, the fourth bit of a code choosing between the halves of the table (5.5 instructions a
//           pair, no memory; a table in shared memory costs 9 and two loads).
#pragma once

#include "lowra_common.cuh"

namespace lowra {

template <int B> struct Scaled;
template <> struct Scaled<1> {
    uint32_t base, d, f;     // both halves: the smaller pattern; the difference of the patterns; 0x10001 if level 0 is the larger one
    __device__ __forceinline__ void set(const float* y, float a) {
        const uint32_t LH = pack_bf16x2(__fmul_rn(y[0], a), __fmul_rn(y[1], a));
        const uint32_t L = LH & 0xFFFFu, H = LH >> 16, lo = min(L, H);
        base = lo * 0x10001u; d = max(L, H) - lo; f = (L > H) ? 0x10001u : 0u;
    }
    // elements 16 q .. 16 q + 15 of the block whose codes are w[0 .. 1]
    __device__ __forceinline__ void expand16(const uint32_t* w, int q, uint32_t (&o)[8]) const {
        const uint32_t h = (q & 1) ? (w[q >> 1] >> 16) : (w[q >> 1] & 0xFFFFu);
        const uint32_t z = h | (h << 15);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = (((z >> (2 * i)) & 0x10001u) ^ f) * d + base;
    }
};
template <> struct Scaled<2> {
    uint32_t lo, hi;         // low and high bytes of the four patterns
    __device__ __forceinline__ void set(const float* y, float a) {
        const uint32_t p = pack_bf16x2(__fmul_rn(y[0], a), __fmul_rn(y[1], a)), r = pack_bf16x2(__fmul_rn(y[2], a), __fmul_rn(y[3], a));
        lo = __byte_perm(p, r, 0x6420u);
        hi = __byte_perm(p, r, 0x7531u);
    }
    __device__ __forceinline__ void expand16(const uint32_t* w, int q, uint32_t (&o)[8]) const {
        const uint32_t even = w[q] & 0x33333333u, odd = (w[q] >> 2) & 0x33333333u;   // the codes of every second element, one per nibble
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t e = h ? even >> 16 : even, d = h ? odd >> 16 : odd;
            const uint32_t el = __byte_perm(lo, 0u, e), eh = __byte_perm(hi, 0u, e), dl = __byte_perm(lo, 0u, d), dh = __byte_perm(hi, 0u, d);
            const uint32_t e01 = __byte_perm(el, eh, 0x5140u), e23 = __byte_perm(el, eh, 0x7362u);
            const uint32_t d01 = __byte_perm(dl, dh, 0x5140u), d23 = __byte_perm(dl, dh, 0x7362u);
            o[4 * h] = __byte_perm(e01, d01, 0x5410u);
            o[4 * h + 1] = __byte_perm(e01, d01, 0x7632u);
            o[4 * h + 2] = __byte_perm(e23, d23, 0x5410u);
            o[4 * h + 3] = __byte_perm(e23, d23, 0x7632u);
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
        for (int h = 0; h < 4; ++h) {   // four codes at a time
            const uint32_t x = w[2 * q + (h >> 1)] >> (16 * (h & 1));
            const uint32_t sel = x & 0x7777u;
            const uint32_t upper = __byte_perm(0x0000FF00u, 0u, (x >> 3) & 0x1111u);   // 0xFF where the code is 8 or more
            const uint32_t l = (__byte_perm(lo[0], lo[1], sel) & ~upper) | (__byte_perm(lo[2], lo[3], sel) & upper);
            const uint32_t u = (__byte_perm(hi[0], hi[1], sel) & ~upper) | (__byte_perm(hi[2], hi[3], sel) & upper);
            o[2 * h] = __byte_perm(l, u, 0x5140u);
            o[2 * h + 1] = __byte_perm(l, u, 0x7362u);
        }
    }
};

}  // namespace lowra
