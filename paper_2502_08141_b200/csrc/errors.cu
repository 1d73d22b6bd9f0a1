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
// time.  At 1 and 2 bits the two or four values w_hat are formed once per half block and picked by comparison; at 4 bits
// a branch-free binary search finds the level.  The residual is written over the weights in shared memory and leaves in one bulk copy
// per chunk.
// What bounds it: memory at 1 and 2 bits (5120 x 5120 at 85/15 % with the residual 44.6 -> 37.3 us, 85 % of the copy rate; without it 26.2 ->
// 20.7), the half-rate pipe for comparisons, selections and address arithmetic at 4 bits and for all three precisions at once (4096 x 4096: 29.1 ->
// 21.1 and 40.7 -> 31 us).
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

// Error of a lane's part of a block at B bits (inv: what normalises it; m: the block's absmax; y: the row's levels in shared memory, its
// thresholds behind them); with RES the residuals take the weights' places.  The number of thresholds <= n picks the level
// (thresholds sorted, as the encoder assumes).
template <int B, bool RES, int PER>
__device__ __forceinline__ double half_block_error(float (&x)[PER], float inv, float m, const float* y) {
    const float* t = y + kTableStride;
    double acc = 0.0;
    float wh[B == 4 ? 1 : 1 << B], th[B == 4 ? 1 : (1 << B) - 1];
    if (B <= 2) {
#pragma unroll
        for (int k = 0; k < (1 << B); ++k) wh[k] = __uint_as_float(pack_bf16x2(0.0f, __fmul_rn(y[k], m)) & 0xFFFF0000u);
#pragma unroll
        for (int k = 0; k + 1 < (1 << B); ++k) th[k] = t[k];
    }
    const float t7 = t[7];
    const uint32_t t_at = (uint32_t)__cvta_generic_to_shared(t);
#pragma unroll
    for (int q = 0; q < PER / 4; ++q) {
        float res[4];
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            const float n0 = __fmul_rn(x[4 * q + e], inv), n1 = __fmul_rn(x[4 * q + e + 1], inv);
            float w0, w1;
            if (B <= 2) {
                auto pick = [&](float n) {
                    if (B == 1) return th[0] <= n ? wh[1] : wh[0];
                    const bool hi = th[B == 2 ? 1 : 0] <= n;
                    const bool lo = (hi ? th[B == 2 ? 2 : 0] : th[0]) <= n;
                    const float a = hi ? wh[B == 2 ? 2 : 0] : wh[0], b = hi ? wh[B == 2 ? 3 : 0] : wh[1];
                    return lo ? b : a;
                };
                w0 = pick(n0);
                w1 = pick(n1);
            } else {
                // binary search on shared-memory addresses: the thresholds lie behind the levels
                auto level = [&](float n) {
                    uint32_t a = t7 <= n ? t_at + 32u : t_at;
                    a += lds_f32(a + 12u) <= n ? 16u : 0u;
                    a += lds_f32(a + 4u) <= n ? 8u : 0u;
                    a += lds_f32(a) <= n ? 4u : 0u;
                    return lds_f32(a - 4u * kTableStride);
                };
                const uint32_t h = pack_bf16x2(__fmul_rn(level(n0), m), __fmul_rn(level(n1), m));
                w0 = __uint_as_float(h << 16);
                w1 = __uint_as_float(h & 0xFFFF0000u);
            }
            res[e] = __fsub_rn(x[4 * q + e], w0);
            res[e + 1] = __fsub_rn(x[4 * q + e + 1], w1);
        }
        // four squares in fp32, then into the fp64 sum
        acc += (double)__fadd_rn(__fmaf_rn(res[0], res[0], __fmul_rn(res[1], res[1])), __fmaf_rn(res[2], res[2], __fmul_rn(res[3], res[3])));
        if (RES) { x[4 * q] = res[0]; x[4 * q + 1] = res[1]; x[4 * q + 2] = res[2]; x[4 * q + 3] = res[3]; }
    }
    return acc;
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
                    acc[0] += half_block_error<1, false, PER>(x, inv, m, tables);
                    acc[1] += half_block_error<2, false, PER>(x, inv, m, tables + 32);
                    acc[2] += half_block_error<4, false, PER>(x, inv, m, tables + 64);
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
