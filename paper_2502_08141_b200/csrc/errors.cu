// lowra_quant_error: summed square error per output channel and, optionally, the residual W - W_hat.
// lowra_channel_errors: the same error under 1, 2 and 4 bits at once (one read of W), without a layout.
//
// The precision assigner minimises the summed square error between the weights and their quantised
// counterparts (paper Section 5 and its footnote; Section 5.1 starts from every channel's error under 1, 2 and
// 4 bits), and an iterative low-rank initialiser factorises the residual W - W_hat after quantising (appendix on
// the low-rank initialisers).  Both come out of one pass over W, fused: block absmax, normalise, bucket, look the
// level up, scale and round to bf16 exactly as lowra_encode followed by lowra_decode would - without writing codes
// or W_hat - then
//     residual = fl32(x - w_hat)            one fp32 subtraction per element (optional output)
//     SSE_row  = sum of residual^2          four neighbouring squares are added in fp32, those partial sums in fp64,
//                                           fixed reduction tree (reproducible, the same for a row wherever it stands)
// so SSE agrees with the exact sum to 2^-21 relative at worst (residual rounded to fp32: 2^-23; a square and two
// additions in fp32: 3 * 2^-24 more), typically far closer.
//
// Traffic: 4 bytes per element read (+ 4 written with the residual), streamed as row_stream.cuh says: a lane works on half an absmax block at a
// time.  At 1 and 2 bits the two or four values w_hat are formed once per half block, and every one is subtracted under its own condition; at 4 bits
// a branch-free binary search finds the level.  The residual is written over the weights in shared memory and leaves in one bulk copy
// per chunk.
// What bounds it: memory at 1 and 2 bits (5120 x 5120 at 85/15 % with the residual 36.8 us, 87 % of the copy rate; without it 19.5), instruction
// issue at 4 bits and for all three precisions at once (45 instructions an element in 74 % of the slots; 4096 x 4096: 20.4 -> 18.5 us with conditional
// additions and subtractions instead of selections, and what comes in pairs in packed instructions; 30.9 -> 27.6, a value normalised once for all).
#include "row_stream.cuh"

namespace lowra {

namespace {

constexpr int kErrThreads = 32 * kRowWarps;
constexpr int kErrRows = 16;   // rows of a CTA between two barriers (their sums per warp are kept in shared memory)

struct ErrParams {
    RowLayout L;
    const float* W;           // [N, K] original order
    const float* maps;        // [N, 16]
    const float* thresholds;  // [N, 16]
    double* sse;              // [N]
    float* residual;          // [N, K] or null
};

// What is left of x after the value its bucket stands for, 1 bit (two values) and 2 bits (four): every candidate's difference, the last one that the encoder's search
// passes through stands (at 2 bits the middle threshold first, then the one on its side, so that codes and errors agree in whatever order the thresholds are).
// Comparisons and selections go to the half-rate pipe, conditional subtractions to the other one.
__device__ __forceinline__ float residual_of(float x, float n, const float (&w)[2], const float (&t)[1]) {
    float r;
    asm("{\n\t.reg .pred p;\n\tsetp.le.f32 p, %4, %5;\n\tsub.rn.f32 %0, %1, %2;\n\t@p sub.rn.f32 %0, %1, %3;\n\t}"
        : "=&f"(r) : "f"(x), "f"(w[0]), "f"(w[1]), "f"(t[0]), "f"(n));
    return r;
}
__device__ __forceinline__ float residual_of(float x, float n, const float (&w)[4], const float (&t)[3]) {
    float r;
    asm("{\n\t.reg .pred p, q, s;\n\tsetp.le.f32 p, %7, %9;\n\tsetp.le.and.f32 q, %6, %9, !p;\n\tsetp.le.and.f32 s, %8, %9, p;\n\tsub.rn.f32 %0, %1, %2;\n\t"
        "@q sub.rn.f32 %0, %1, %3;\n\t@p sub.rn.f32 %0, %1, %4;\n\t@s sub.rn.f32 %0, %1, %5;\n\t}"
        : "=&f"(r) : "f"(x), "f"(w[0]), "f"(w[1]), "f"(w[2]), "f"(w[3]), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(n));
    return r;
}

// A row's codebook at B bits for one half block: the values its buckets stand for there (1 and 2 bits), and the thresholds; or (4 bits) where
// levels and thresholds lie, which a binary search on addresses reads.
template <int B>
struct HalfBlock {
    float w[1 << B], t[(1 << B) - 1];
    __device__ __forceinline__ HalfBlock(const float* y, float m) {
#pragma unroll
        for (int k = 0; k < (1 << B); ++k) w[k] = __uint_as_float(pack_bf16x2(0.0f, __fmul_rn(y[k], m)) & 0xFFFF0000u);
#pragma unroll
        for (int k = 0; k + 1 < (1 << B); ++k) t[k] = y[kTableStride + k];
    }
    __device__ __forceinline__ float residual(float x, float n) const { return residual_of(x, n, w, t); }
};
template <>
struct HalfBlock<4> {
    uint32_t at;
    float t7, m;
    __device__ __forceinline__ HalfBlock(const float* y, float m_) : at((uint32_t)__cvta_generic_to_shared(y + kTableStride)), t7(y[kTableStride + 7]), m(m_) {}
    __device__ __forceinline__ float residual(float x, float n) const {
        const uint32_t a = threshold_place(at, t7, n);
        return __fsub_rn(x, __uint_as_float(pack_bf16x2(0.0f, __fmul_rn(lds_f32(a - 4u * kTableStride), m))));
    }
};

template <bool PACKED>
__device__ __forceinline__ float2 normalised(float a, float b, float inv) {
    return PACKED ? mul2(make_float2(a, b), make_float2(inv, inv)) : make_float2(__fmul_rn(a, inv), __fmul_rn(b, inv));
}

// Error of four neighbouring elements: four squares in fp32, then into the fp64 sum.  PACKED: without residuals to keep, where instructions bound the kernel (three
// precisions on 4096 x 4096); residuals next to one another for both purposes cost moves (at 4 bits 24.4 -> 28.1).
template <bool PACKED>
__device__ __forceinline__ double four_squares(const float (&r)[4]) {
    if (!PACKED) return (double)__fadd_rn(__fmaf_rn(r[0], r[0], __fmul_rn(r[1], r[1])), __fmaf_rn(r[2], r[2], __fmul_rn(r[3], r[3])));
    const float2 even = make_float2(r[0], r[2]), odd = make_float2(r[1], r[3]);
    const float2 s = fma2(even, even, mul2(odd, odd));
    return (double)__fadd_rn(s.x, s.y);
}

// Error of a lane's part of a block at B bits (inv: what normalises it; m: the block's absmax; y: the row's levels in shared memory, its
// thresholds behind them); with RES the residuals take the weights' places.  The number of thresholds <= n picks the level
// (thresholds sorted, as the encoder assumes).
template <int B, bool RES, int PER>
__device__ __forceinline__ double half_block_error(float (&x)[PER], float inv, float m, const float* y) {
    const HalfBlock<B> book(y, m);
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < PER / 4; ++q) {
        float r[4];
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            const float2 n = normalised<!RES>(x[4 * q + e], x[4 * q + e + 1], inv);
            r[e] = book.residual(x[4 * q + e], n.x);
            r[e + 1] = book.residual(x[4 * q + e + 1], n.y);
        }
        acc += four_squares<!RES>(r);
        if (RES) { x[4 * q] = r[0]; x[4 * q + 1] = r[1]; x[4 * q + 2] = r[2]; x[4 * q + 3] = r[3]; }
    }
    return acc;
}
// At all three precisions: the tables one behind the other.
template <int PER>
__device__ __forceinline__ void half_block_errors(const float (&x)[PER], float inv, float m, const float* y, double (&acc)[3]) {
    const HalfBlock<1> one_bit(y, m);
    const HalfBlock<2> two_bits(y + 32, m);
    const HalfBlock<4> four_bits(y + 64, m);
    double sum[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < PER / 4; ++q) {
        float r[3][4];
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            const float2 n2 = normalised<true>(x[4 * q + e], x[4 * q + e + 1], inv);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float v = x[4 * q + e + i], n = i ? n2.y : n2.x;
                r[0][e + i] = one_bit.residual(v, n);
                r[1][e + i] = two_bits.residual(v, n);
                r[2][e + i] = four_bits.residual(v, n);
            }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) sum[k] += four_squares<true>(r[k]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] += sum[k];
}

// sum over the warp, in a fixed order
__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// NP = 1: the error at the rows' own precisions, rows in stored order; NP = 3: at all three.  PER: elements per lane; AHEAD: chunks on
// their way in.
template <int NP, bool RES, int PER, int AHEAD, typename Params>
__device__ __forceinline__ void error_rows(const Params& P, int N, int K) {
    constexpr int kTables = NP * 2 * kTableStride * (int)sizeof(float);
    constexpr int kChunk = 32 * PER;
    constexpr int kBuffer = kChunk * (int)sizeof(float) + kTables;
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* part = reinterpret_cast<double*>(smem + kRowWarps * kRowDepth * kBuffer);   // [kErrRows][kRowWarps][NP]
    int* row_ids = reinterpret_cast<int*>(part + kErrRows * kRowWarps * NP);            // [kErrRows]
    unsigned char* mine = smem + warp * kRowDepth * kBuffer;
    for (int i = threadIdx.x; i < kErrRows * kRowWarps * NP; i += kErrThreads) part[i] = 0.0;
    __syncthreads();
    pdl_enter();
    const uint64_t once = once_policy();
    const int rows = (N - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    // stored rows from the last to the first; original row of the CTA's row i
    auto row_of = [&](int i) {
        const int p = (int)blockIdx.x + i * (int)gridDim.x;
        if constexpr (NP == 3) return p;
        else return i < rows ? (int)__ldg(P.L.perm + (N - 1 - p)) : 0;
    };
    const RowWalk walk(K, kChunk);
    RowPlace at = walk.start(warp), ahead = at;
    int r_of[AHEAD + 1];                      // rows of the chunks under way and of the one after them
    {
        RowPlace a = at;
#pragma unroll
        for (int d = 0; d <= AHEAD; ++d) { r_of[d] = row_of(a.i); walk.next(a); }
    }
    auto copy_ahead = [&](int buffer, int r) {
        const RowPlace a = ahead;
        walk.next(ahead);
        if (a.i < rows) {
            unsigned char* buf = mine + buffer * kBuffer;
            chunk_copy<PER>(buf, P.W + (size_t)r * K + (size_t)a.j * kChunk, min(K - a.j * kChunk, kChunk), lane, once);
            if (lane < 8 * NP) {   // per precision 64 bytes of levels, 64 of thresholds
                const size_t plane = NP == 3 ? (size_t)(lane >> 3) * N * kTableStride : 0;
                const float* src = ((lane & 4) ? P.thresholds : P.maps) + plane + (size_t)r * kTableStride + 4 * (lane & 3);
                copy16_async(buf + kChunk * sizeof(float) + 16 * lane, src);
            }
        }
        copies_commit();
    };
#pragma unroll
    for (int d = 0; d < AHEAD; ++d) copy_ahead(d, r_of[d]);
    int buffer = 0;
    double acc[NP] = {};
    for (int i0 = 0; i0 < rows; i0 += kErrRows) {
        const int i1 = min(i0 + kErrRows, rows);
        while (at.i < i1) {
            copies_wait<AHEAD - 1>();
            __syncwarp();
            unsigned char* buf = mine + buffer * kBuffer;
            const int r = r_of[0], valid = min(K - at.j * kChunk, kChunk);
            const float* tables = reinterpret_cast<const float*>(buf + kChunk * sizeof(float));
            float x[PER];
            float m = 0.0f;
            const bool in = PER * lane < valid;
#pragma unroll
            for (int t = 0; t < PER / 4; ++t) {
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                if (in) f = *reinterpret_cast<const float4*>(buf + piece_at<PER>(t, lane));
                x[4 * t] = f.x; x[4 * t + 1] = f.y; x[4 * t + 2] = f.z; x[4 * t + 3] = f.w;
                m = fmaxf(fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y))), fmaxf(fabsf(f.z), fabsf(f.w)));
            }
            for (int d = 1; d < kBlock / PER; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
            const float inv = (m == 0.0f) ? 0.0f : __frcp_rn(m);
            if (in) {
                if constexpr (NP == 3) {
                    half_block_errors<PER>(x, inv, m, tables, acc);
                } else {
                    const int p = N - 1 - ((int)blockIdx.x + at.i * (int)gridDim.x);
                    if (p < P.L.class_start[1]) acc[0] += half_block_error<1, RES, PER>(x, inv, m, tables);
                    else if (p < P.L.class_start[2]) acc[0] += half_block_error<2, RES, PER>(x, inv, m, tables);
                    else acc[0] += half_block_error<4, RES, PER>(x, inv, m, tables);
                }
            }
            if constexpr (RES) {
                if (in) {
#pragma unroll
                    for (int t = 0; t < PER / 4; ++t) *reinterpret_cast<float4*>(buf + piece_at<PER>(t, lane)) = make_float4(x[4 * t], x[4 * t + 1], x[4 * t + 2], x[4 * t + 3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(P.residual + (size_t)r * K + (size_t)at.j * kChunk),
                                 "r"((uint32_t)__cvta_generic_to_shared(buf)), "r"((uint32_t)valid * 4u), "l"(once) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kRowDepth - AHEAD) : "memory");   // the buffer that is filled next has been read
                }
            }
            __syncwarp();
            if (lane == 0 && at.j == 0) row_ids[at.i - i0] = r;
            const RowPlace was = at;
            walk.next(at);
            if (at.i != was.i) {
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const double v = warp_total(acc[k]);
                    if (lane == 0) part[((was.i - i0) * kRowWarps + warp) * NP + k] = v;
                    acc[k] = 0.0;
                }
            }
#pragma unroll
            for (int d = 0; d < AHEAD; ++d) r_of[d] = r_of[d + 1];
            copy_ahead(buffer + AHEAD < kRowDepth ? buffer + AHEAD : buffer + AHEAD - kRowDepth, r_of[AHEAD - 1]);
            r_of[AHEAD] = row_of(ahead.i);
            buffer = buffer + 1 == kRowDepth ? 0 : buffer + 1;
        }
        __syncthreads();
        for (int s = threadIdx.x; s < (i1 - i0) * NP; s += kErrThreads) {
            double v = 0.0;
            // from the warp that had the row's first chunk: a row's sum does not depend on its place
            const int first = (i0 + s / NP) * walk.per_row;
#pragma unroll
            for (int w = 0; w < kRowWarps; ++w) {
                double& slot = part[((s / NP) * kRowWarps + (first + w) % kRowWarps) * NP + s % NP];
                v += slot;
                slot = 0.0;
            }
            P.sse[(size_t)row_ids[s / NP] * NP + s % NP] = v;
        }
        __syncthreads();
    }
    copies_wait<0>();
    if (RES && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

template <bool RES, int PER, int AHEAD>
__global__ void __launch_bounds__(kErrThreads, row_ctas(PER)) error_kernel(const __grid_constant__ ErrParams P) {
    error_rows<1, RES, PER, AHEAD>(P, P.L.N, P.L.K);
}

// ---- all three precisions in one pass (the assigner's input: every channel's error under 1, 2 and 4 bits) ----
struct Err3Params {
    const float* W;           // [N, K]
    const float* maps;        // [3][N][16]: tables of the 1-, 2- and 4-bit codebooks of every row
    const float* thresholds;  // [3][N][16]
    double* sse;              // [N][3]
    int N, K;
};

template <int PER>
__global__ void __launch_bounds__(kErrThreads, row_ctas(PER)) error3_kernel(const __grid_constant__ Err3Params P) {
    error_rows<3, false, PER, kRowDepth - 1>(P, P.N, P.K);
}

template <int NP, int PER, typename Params>
lowra_status launch_errors(void (*kernel)(Params), const Params& P, int N, SmemLimit* limit, void* stream) {
    const size_t smem = kRowWarps * kRowDepth * (32 * PER * sizeof(float) + NP * 2 * kTableStride * sizeof(float)) + kErrRows * (kRowWarps * NP * sizeof(double) + sizeof(int));
    if (ensure_smem_limit(reinterpret_cast<const void*>(kernel), smem, limit) != LOWRA_OK) return LOWRA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(N < row_ctas(PER) * kNumSMs ? N : row_ctas(PER) * kNumSMs), 1, 1);
    cfg.blockDim = dim3(kErrThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P) == cudaSuccess ? LOWRA_OK : LOWRA_ERR_CUDA;
}

}  // namespace
}  // namespace lowra

extern "C" lowra_status lowra_quant_error(const lowra_layout* layout, const float* W_dev, const float* maps_dev,
                                          const float* thresholds_dev, double* sse_dev, float* residual_dev,
                                          void* stream) {
    using namespace lowra;
    lowra_status st = check_layout(layout);
    if (st != LOWRA_OK) return st;
    if (!W_dev || !maps_dev || !thresholds_dev || !sse_dev) return LOWRA_ERR_NULL;
    if (!aligned16(W_dev) || !aligned16(maps_dev) || !aligned16(thresholds_dev) || !aligned16(sse_dev) ||
        (residual_dev && !aligned16(residual_dev)))
        return LOWRA_ERR_ALIGN;
    st = check_device();
    if (st != LOWRA_OK) return st;
    ErrParams P;
    P.L = make_row_layout(layout);
    P.W = W_dev;
    P.maps = maps_dev;
    P.thresholds = thresholds_dev;
    P.sse = sse_dev;
    P.residual = residual_dev;
    static SmemLimit limits[5] = {};
    if (row_per_lane(layout->K) == 16)
        return residual_dev ? launch_errors<1, 16>(error_kernel<true, 16, 2>, P, layout->N, &limits[0], stream)
                            : launch_errors<1, 16>(error_kernel<false, 16, 2>, P, layout->N, &limits[1], stream);
    if (!residual_dev) return launch_errors<1, 32>(error_kernel<false, 32, 2>, P, layout->N, &limits[2], stream);
    // Where weights and residuals do not fit into L2 twice over and most rows are cheap ones, memory is the better for fewer reads between
    // the writes: one chunk ahead against two, 11008 x 4096 at 60/35/5 %: 60.8 against 63.1 us; but 4096 x 4096 22.5 against 20.7 us, and
    // 11008 x 4096 at 4 bits 66.9 against 61.4.
    const bool writes_wait = 8ull * layout->N * layout->K > 2ull * 126 * 1024 * 1024 && layout->counts[2] < layout->N / 2;
    return writes_wait ? launch_errors<1, 32>(error_kernel<true, 32, 1>, P, layout->N, &limits[3], stream)
                       : launch_errors<1, 32>(error_kernel<true, 32, 2>, P, layout->N, &limits[4], stream);
}

extern "C" lowra_status lowra_channel_errors(int32_t N, int32_t K, const float* W_dev, const float* maps3_dev,
                                             const float* thresholds3_dev, double* sse3_dev, void* stream) {
    using namespace lowra;
    if (!W_dev || !maps3_dev || !thresholds3_dev || !sse3_dev) return LOWRA_ERR_NULL;
    if (N < 1 || K < 128 || K % 128 != 0) return LOWRA_ERR_SHAPE;
    if (!aligned16(W_dev) || !aligned16(maps3_dev) || !aligned16(thresholds3_dev) || (reinterpret_cast<uintptr_t>(sse3_dev) & 7u) != 0)
        return LOWRA_ERR_ALIGN;
    lowra_status st = check_device();
    if (st != LOWRA_OK) return st;
    Err3Params P;
    P.W = W_dev;
    P.maps = maps3_dev;
    P.thresholds = thresholds3_dev;
    P.sse = sse3_dev;
    P.N = N;
    P.K = K;
    static SmemLimit limits[2] = {};
    return row_per_lane(K) == 16 ? launch_errors<3, 16>(error3_kernel<16>, P, N, &limits[0], stream)
                                 : launch_errors<3, 32>(error3_kernel<32>, P, N, &limits[1], stream);
}
