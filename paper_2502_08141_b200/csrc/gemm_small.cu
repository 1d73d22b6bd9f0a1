// Forward pass for few tokens (generation, short prompts, small token groups of several adapters):
//     Y = X . deq(Wq)^T + s * (X . A) . B
// With a handful of tokens the work is reading the weight's codes once (1 - 2 bits per weight), a few microseconds of memory
// time: what counts is how many SMs share it and how long the longest chain of dependent steps is.  The persistent
// tensor-core kernel (gemm_fused.cu) has tiles of 256 channels and 256 tokens, of which a 4096 x 4096 weight is 16: cut in four, their
// slices handed over, it takes 26 us for 1 token as for 65.  Here two launches share the work finely instead (1 token 8.9, 16 tokens 10.7):
//   project_kernel   T = bf16(s X A): a CTA per 16 tokens and slice of the contraction, the slices of a cluster added up
//                    through distributed shared memory.
//   small_kernel     a CTA takes 64 stored rows of one precision and a slice of the contraction, its warps 16 rows and half
//                    of that slice each.  The weights never leave the registers: in a block of 256 input features lane
//                    (g, t) of a warp holds the 64-element absmax block t of the rows g and g + 8 - one wide load of codes,
//                    one absmax - and dequantises it straight into the A fragments of mma.m16n8k16.  The order in which the
//                    contraction indices are fed is free as long as both operands agree, so lane t's fragments are
//                    simply its own next four elements, for the weights and for the tokens alike.  The tokens of the slice
//                    lie in shared memory.  Slices are added up as above; the low-rank term enters as further steps of
//                    the same accumulation.
// It starts while project_kernel runs and waits for it only before the low-rank term (programmatic dependent launch).  For a small weight with a low rank
// every CTA of small_kernel forms T itself, and there is no other launch.
// No flags, no waits that need a limit, any number of such calls may share the GPU.
#include <type_traits>

#include "dequant.cuh"
#include "gemm_params.cuh"
#include "ptx.cuh"

namespace lowra {

namespace {

constexpr int kSmallThreads = 256;
constexpr int kSmallRows = 64;          // stored rows per CTA
constexpr int kMergedPitch = kSmallRows + 4;   // fp32 words: neighbouring tokens of a tile of sums 4 banks apart
constexpr int kSmallSpan = 256;         // contraction indices per step of a warp: one absmax block for each of four lanes

struct Unit { int member, m0; };        // up to 8 NT8 tokens of one member
template <int NB>
__device__ __forceinline__ Unit unit_at(const SmallParams<NB>& P, int u, int tokens) {
    Unit r = {0, 0};
    for (int i = 0; NB > 1 && i + 1 < P.count; ++i) {
        const int n = (P.m[i].M + tokens - 1) / tokens;
        if (u < n) break;
        u -= n;
        r.member = i + 1;
    }
    r.m0 = u * tokens;
    return r;
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async_16_zfill(uint32_t saddr, const void* gptr, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr), "l"(gptr), "r"(valid ? 16u : 0u) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t saddr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(saddr));
    return v;
}
__device__ __forceinline__ void st_cluster_f32(uint32_t caddr, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(caddr), "f"(v) : "memory"); }
__device__ __forceinline__ void st_cluster_f4(uint32_t caddr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(caddr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// ------------------------------------------------------------------------------------------------ T = bf16(s X A)
constexpr int kProjectBatch = 4;        // steps of 16 contraction indices a warp fetches at a time

// bytes of A a CTA fetches at a time (more than its warps' sums, 512 (r + 8), which later take the same place)
__host__ __device__ constexpr size_t project_fetch_bytes(int r) { return (size_t)(kSmallThreads / 32) * kProjectBatch * 16 * (r * 2 + 16); }

// slices of the projection's contraction: up to eight, 128 indices or more each
__host__ __device__ constexpr int project_slices(int K) {
    int slices = 1;
    while (slices < 8 && K >= 256 * slices) slices *= 2;
    return slices;
}

// Grid: (slices of the contraction = cluster, tiles of 16 tokens of all members).  What bounds it: latency, all of which the product waits for.  No division on the
// way (by powers of two: shifts), sums padded and in wide accesses: 16 tokens on 4096 x 4096 with the product 11.9 -> 11.0 us a call, rank 128 and 30 tokens on
// 2048 x 2048 13.1 -> 10.9; in units_kernel, which found its slices' bounds by 64-bit divisions, six groups of 101 tokens on 4096 x 4096 43.8 -> 39.8.
template <int NB>
__global__ void __launch_bounds__(kSmallThreads) project_kernel(const __grid_constant__ SmallParams<NB> P) {
    extern __shared__ __align__(16) unsigned char project_smem[];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // the next kernel reads its operands right away, so it may start only now that everything before this kernel is complete
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cluster_arrive();   // "this CTA runs": waited for before its shared memory is written from elsewhere
    if (P.clear_status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *P.status = 0u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int slices = (int)gridDim.x, slice = (int)blockIdx.x;
    const Unit un = unit_at(P, (int)blockIdx.y, 16);
    const SmallMember& W = P.m[un.member];
    const int n_steps = P.K / 16;
    const int slices_log = 31 - __clz(slices);
    const int s0 = (int)(((long long)slice * n_steps) >> slices_log), s1 = (int)(((long long)(slice + 1) * n_steps) >> slices_log);
    const int pitch = P.r * 2 + 16;                                   // bytes per contraction index of A in shared memory
    unsigned char* mine = project_smem + (size_t)warp * (kProjectBatch * 16 * pitch);
    const int n_j8 = P.r / 8;
    float acc[16][4];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
    const int row0 = un.m0 + g, row1 = row0 + 8;
    const uint32_t* x0 = reinterpret_cast<const uint32_t*>(W.X + (size_t)row0 * P.K) + t;
    const uint32_t* x1 = reinterpret_cast<const uint32_t*>(W.X + (size_t)row1 * P.K) + t;
    const bool v0 = row0 < W.M, v1 = row1 < W.M;
    constexpr int kWarps = kSmallThreads / 32;
    for (int first = s0 + warp; first < s1; first += kWarps * kProjectBatch) {
        uint32_t xa[kProjectBatch][4];
        __syncwarp();   // the previous batch has been read
#pragma unroll
        for (int u = 0; u < kProjectBatch; ++u) {
            const int st = first + u * kWarps;
            xa[u][0] = xa[u][1] = xa[u][2] = xa[u][3] = 0u;
            if (st < s1) {
                const int k = lane & 15;
                for (int j = lane >> 4; j < n_j8; j += 2)
                    cp_async_16_zfill(ptx::smem_u32(mine + (u * 16 + k) * pitch + j * 16), W.A + (size_t)(st * 16 + k) * P.r + j * 8, true);
                if (v0) { xa[u][0] = __ldg(x0 + st * 8); xa[u][2] = __ldg(x0 + st * 8 + 4); }
                if (v1) { xa[u][1] = __ldg(x1 + st * 8); xa[u][3] = __ldg(x1 + st * 8 + 4); }
            }
        }
        ptx::cp_async_commit();
        ptx::cp_async_wait<0>();
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kProjectBatch; ++u) {
            if (first + u * kWarps >= s1) break;
            const uint32_t a_row = ptx::smem_u32(mine + (u * 16 + (lane & 15)) * pitch + (lane >> 4) * 16);
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                if (j >= n_j8) break;
                uint32_t b0, b1, b2, b3;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3) : "r"(a_row + (uint32_t)j * 16u) : "memory");
                mma_bf16(acc[j], xa[u][0], xa[u][1], xa[u][2], xa[u][3], b0, b1);
                mma_bf16(acc[j + 1], xa[u][0], xa[u][1], xa[u][2], xa[u][3], b2, b3);
            }
        }
    }
    // the warps' sums, then the CTA's, then the cluster's, each in a fixed order
    __syncthreads();
    float* red = reinterpret_cast<float*>(project_smem);              // [warps][16 tokens][r + 8]: half a warp's stores meet different banks
    const int red_pitch = P.r + 8;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (j >= n_j8) break;
        float* d = red + (warp * 16 + g) * red_pitch + j * 8 + 2 * t;
        *reinterpret_cast<float2*>(d) = make_float2(acc[j][0], acc[j][1]);
        *reinterpret_cast<float2*>(d + 8 * red_pitch) = make_float2(acc[j][2], acc[j][3]);
    }
    __syncthreads();
    // every CTA of the cluster owns a share of the sums, 16 / slices tokens: its own sums of a share go into the owner's shared memory
    const int rows_log = 4 - slices_log, share = P.r << rows_log;
    float* sums = reinterpret_cast<float*>(project_smem + project_fetch_bytes(P.r));   // [slices][share]: behind what this CTA may still be reading
    const uint32_t recv = ptx::smem_u32(sums);
    cluster_wait();
    const int row = (int)threadIdx.x >> 4, col0 = 4 * ((int)threadIdx.x & 15);        // sixteen threads to a token, four ranks each
    for (int col = col0; col < P.r; col += 64) {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float4 v = *reinterpret_cast<const float4*>(red + (w * 16 + row) * red_pitch + col);
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        const uint32_t at = recv + (uint32_t)(slice * share + (row & ((1 << rows_log) - 1)) * P.r + col) * 4u;
        st_cluster_f4(ptx::map_to_cta(at, (uint32_t)(row >> rows_log)), sum);
    }
    ptx::cluster_sync();
    const int mine_row = un.m0 + (slice << rows_log) + row;
    if (row < (1 << rows_log) && mine_row < W.M) {
        for (int col = col0; col < P.r; col += 64) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int c = 0; c < slices; ++c) {
                const float4 b = *reinterpret_cast<const float4*>(sums + c * share + row * P.r + col);
                a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            }
            *reinterpret_cast<uint2*>(W.T + (size_t)mine_row * P.rp + col) = make_uint2(pack_bf16x2(P.s * a.x, P.s * a.y), pack_bf16x2(P.s * a.z, P.s * a.w));
        }
    }
    // columns between the rank and its padded width are zero
    if (slice == 0 && un.m0 + row < W.M)
        for (int col = P.r + col0; col < P.rp; col += 64) *reinterpret_cast<uint2*>(W.T + (size_t)(un.m0 + row) * P.rp + col) = make_uint2(0u, 0u);
}

// ------------------------------------------------------------------------------------------------ the product
// What a lane fetches of one row for one step: the codes of a 64-element block (8, 16 or 32 bytes) and its absmax.
template <int B>
struct Codes {
    uint32_t w[2 * B];
    float a;
};
template <int B>
__device__ __forceinline__ void fetch_codes(Codes<B>& c, const uint8_t* row, const float* absmax, int blk, bool valid) {
    if (!valid) {
#pragma unroll
        for (int i = 0; i < 2 * B; ++i) c.w[i] = 0u;
        c.a = 0.0f;
        return;
    }
    const uint8_t* p = row + (size_t)blk * (8 * B);
    if (B == 1) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
        c.w[0] = v.x; c.w[1] = v.y;
    } else {
#pragma unroll
        for (int i = 0; i < B / 2; ++i) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(p) + i);
            c.w[4 * i] = v.x; c.w[4 * i + 1] = v.y; c.w[4 * i + 2] = v.z; c.w[4 * i + 3] = v.w;
        }
    }
    c.a = __ldg(absmax + blk);
}

template <int B>
__device__ __forceinline__ void load_levels(float (&y)[1 << B], const float* row) {
    if (B == 1) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(row));
        y[0] = v.x; y[1] = v.y;
    } else {
#pragma unroll
        for (int i = 0; i < (1 << B) / 4; ++i) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(row) + i);
            y[4 * i] = v.x; y[4 * i + 1] = v.y; y[4 * i + 2] = v.z; y[4 * i + 3] = v.w;
        }
    }
}

// Where 16-byte piece j (0 .. 7) of block t of token row m lies in a staged [tokens][256] tile: the pieces of a block are
// exchanged among themselves so that the eight lanes of a shared-memory wavefront read eight different columns.
__device__ __forceinline__ uint32_t token_piece(int m, int t, int j) {
    return (uint32_t)(m * (kSmallSpan * 2) + (t * 8 + (j ^ (t | ((m & 1) << 2)))) * 16);
}

// Sixteen elements of the lane's block of either row, times the tokens (xs: where the block's first piece lies for token g).  A sum's steps wait for
// one another, so the tokens take turns.
template <int B, int NT8>
__device__ __forceinline__ void multiply_16(float (&acc)[NT8][4], const Scaled<B>& s0, const Scaled<B>& s1, const Codes<B>& c0, const Codes<B>& c1, int q, uint32_t xs) {
    uint32_t o0[8], o1[8];
    s0.expand16(c0.w, q, o0);
    s1.expand16(c1.w, q, o1);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint4 x[NT8];
#pragma unroll
        for (int nt = 0; nt < NT8; ++nt) x[nt] = ld_shared_v4((xs ^ (32u * q + 16u * h)) + (uint32_t)(nt * 8 * kSmallSpan * 2));
#pragma unroll
        for (int nt = 0; nt < NT8; ++nt) mma_bf16(acc[nt], o0[4 * h], o1[4 * h], o0[4 * h + 1], o1[4 * h + 1], x[nt].x, x[nt].y);
#pragma unroll
        for (int nt = 0; nt < NT8; ++nt) mma_bf16(acc[nt], o0[4 * h + 2], o1[4 * h + 2], o0[4 * h + 3], o1[4 * h + 3], x[nt].z, x[nt].w);
    }
}

// A warp's sixteen rows times the tokens, over the contraction's slots slot0 .. slot1 - 1 of `slots` (neighbouring ranges of it); before and
// after each one's steps begin(slot) and end(slot, acc).
template <int B, int NT8, typename Begin, typename End>
__device__ __forceinline__ void multiply_rows(int K, const SmallMember& W, int m0, int p0, int p_end, int slot0, int slot1, int slots,
                                              uint32_t x_smem, int half, Begin begin, End end) {
    constexpr int c = B >> 1;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n_span = (K + kSmallSpan - 1) / kSmallSpan, nb = K / kBlock;
    const int slots_log = 31 - __clz(slots);          // (a power of two; n_span is below 2^27: K is an int32)
    auto bound = [&](int slot) { return (int)(((long long)slot * n_span) >> slots_log); };
    const int b0 = bound(slot0), b1 = bound(slot1);
    // rows g and g + 8 of the warp's sixteen
    const bool live0 = p0 + g < p_end, live1 = p0 + g + 8 < p_end;
    const int q0 = live0 ? p0 + g : p_end - 1, q1 = live1 ? p0 + g + 8 : p_end - 1;
    const int r0 = __ldg(W.L.perm + q0), r1 = __ldg(W.L.perm + q1);
    const uint8_t* row0 = W.packed + packed_row_offset(W.L, c, q0, r0);
    const uint8_t* row1 = W.packed + packed_row_offset(W.L, c, q1, r1);
    const float* am0 = W.absmax + (size_t)absmax_row_of(W.L, q0, r0) * nb;
    const float* am1 = W.absmax + (size_t)absmax_row_of(W.L, q1, r1) * nb;
    const float* y0 = W.maps + (size_t)r0 * kTableStride;
    const float* y1 = W.maps + (size_t)r1 * kTableStride;
    // tokens of one step: fetched by the four warps that share it, two steps in flight
    constexpr uint32_t kStep = 8u * NT8 * kSmallSpan * 2u;
    const int warp4 = (threadIdx.x >> 5) & 3;
    const uint32_t stage_at = x_smem + token_piece(warp4, lane >> 3, lane & 7);
    const uint32_t read_at = x_smem + token_piece(g, t, 0);          // piece j of its block: read_at ^ 16 j
    auto stage = [&](int b) {
        if (b < b1) {
            // a warp to every fourth token, a lane to a 16-byte piece of its 512 bytes
            const int k = b * kSmallSpan + lane * 8, left = k < K ? W.M - m0 - warp4 : 0;
            const uint16_t* src = W.X + (size_t)(m0 + warp4) * K + k;
            const uint32_t dst = stage_at + (uint32_t)((b - b0) & 1) * kStep;
#pragma unroll
            for (int i = 0; i < 2 * NT8; ++i)
                cp_async_16_zfill(dst + (uint32_t)(4 * i * kSmallSpan * 2), 4 * i < left ? src + (size_t)(4 * i) * K : W.X, 4 * i < left);
        }
        ptx::cp_async_commit();
    };
    Codes<B> n0, n1;
    auto fetch = [&](int b) {
        const int blk = 4 * b + t;
        fetch_codes<B>(n0, row0, am0, blk, live0 && b < b1 && blk < nb);
        fetch_codes<B>(n1, row1, am1, blk, live1 && b < b1 && blk < nb);
    };
    fetch(b0);
    stage(b0);
    float ya[1 << B], yb[1 << B];
    if (B <= 2) {
        load_levels<B>(ya, y0);
        load_levels<B>(yb, y1);
    }
    int b = b0;
    for (int slot = slot0; slot < slot1; ++slot) {
        begin(slot);
        float acc[NT8][4];
#pragma unroll
        for (int i = 0; i < NT8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
        for (const int slot_end = bound(slot + 1); b < slot_end; ++b) {
            const Codes<B> c0 = n0, c1 = n1;
            fetch(b + 1);
            stage(b + 1);
            Scaled<B> s0, s1;
            if (B == 4) {   // (sixteen levels of two rows are too many registers to keep: read again, from L1)
                load_levels<B>(ya, y0);
                s0.set(ya, c0.a);
                load_levels<B>(ya, y1);
                s1.set(ya, c1.a);
            } else {
                s0.set(ya, c0.a);
                s1.set(yb, c1.a);
            }
            ptx::cp_async_wait<1>();
            ptx::named_barrier_sync(1 + half, 128);
            const uint32_t xs = read_at + (uint32_t)((b - b0) & 1) * kStep;
#pragma unroll
            for (int q = 0; q < 4; ++q) multiply_16<B, NT8>(acc, s0, s1, c0, c1, q, xs);
            if (b + 2 < b1) ptx::named_barrier_sync(1 + half, 128);   // the tokens have been read: the buffer may be filled again
        }
        end(slot, acc);
    }
}

// T of up to 16 tokens by one CTA of the product, for itself: a weight so small that the projection's launch costs more.  A lies in shared memory as in memory,
// behind it are the warps' sums [slices][warps][16 tokens][r + 8] and T [16][r + 8]; the tokens are those staged for the product (one step per slot).  The same sums in
// the same order as project_kernel's, the slices' steps side by side (one after the other 0.15 - 0.3 us longer).  Ends with a barrier.
constexpr int kOwnK = 512, kOwnRank = 32, kOwnSlices = 4;
static_assert(project_slices(kOwnK) == kOwnSlices && project_slices(kOwnK - 1) < kOwnSlices, "slices");
struct OwnT {
    unsigned char* a;
    float* sums;
    uint16_t* T;
    static __host__ __device__ constexpr size_t bytes(int K, int r) { return (size_t)K * r * 2 + (size_t)project_slices(K) * 8 * 16 * (r + 8) * 4 + 16 * (r + 8) * 2; }
    __device__ OwnT(unsigned char* smem, int K, int r) : a(smem), sums(reinterpret_cast<float*>(smem + K * r * 2)), T(reinterpret_cast<uint16_t*>(sums + (K < 256 ? 1 : K < 512 ? 2 : 4) * 8 * 16 * (r + 8))) {}
    __device__ __forceinline__ void fetch(const uint16_t* A, int K, int r) const {
        for (int i = threadIdx.x; i < K * r / 8; i += kSmallThreads) cp_async_16_zfill(ptx::smem_u32(a) + 16u * i, A + 8 * i, true);
        ptx::cp_async_commit();
    }
    // x_of(step of 256): where its tokens are staged
    template <int NT8, typename X>
    __device__ __forceinline__ void form(int K, int r, float s, X x_of) const {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        const int log = K < 256 ? 0 : K < 512 ? 1 : 2, n_steps = K / 16;
        ptx::cp_async_wait<0>();
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kOwnSlices; ++c) {
            if (c >= 1 << log) break;
            float acc[kOwnRank / 8][4];
#pragma unroll
            for (int j = 0; j < kOwnRank / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
#pragma unroll 1
            for (int st = ((c * n_steps) >> log) + warp; st < ((c + 1) * n_steps) >> log; st += 8) {
                const int k = st * 16 % kSmallSpan;
                uint32_t x[4] = {0u, 0u, 0u, 0u};
                const uint32_t at = x_of(st / 16) + token_piece(lane & (NT8 == 1 ? 7 : 15), k / 64, k % 64 / 8 + (NT8 == 1 ? lane >> 3 & 1 : lane >> 4));
                if (NT8 == 1) asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(x[0]), "=r"(x[2]) : "r"(at) : "memory");
                else asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(at) : "memory");
                const uint32_t a_row = ptx::smem_u32(a) + (uint32_t)((st * 16 + (lane & 15)) * r * 2 + (lane >> 4) * 16);
#pragma unroll
                for (int j = 0; j < kOwnRank / 8; j += 2) {
                    if (8 * j >= r) break;
                    uint32_t b0, b1, b2, b3;
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3) : "r"(a_row + 16u * j) : "memory");
                    mma_bf16(acc[j], x[0], x[1], x[2], x[3], b0, b1);
                    mma_bf16(acc[j + 1], x[0], x[1], x[2], x[3], b2, b3);
                }
            }
            float* d = sums + ((c * 8 + warp) * 16 + g) * (r + 8) + 2 * t;
#pragma unroll
            for (int j = 0; j < kOwnRank / 8; ++j) {
                if (8 * j >= r) break;
                *reinterpret_cast<float2*>(d + 8 * j) = make_float2(acc[j][0], acc[j][1]);
                *reinterpret_cast<float2*>(d + 8 * (r + 8) + 8 * j) = make_float2(acc[j][2], acc[j][3]);
            }
        }
        __syncthreads();
        const int row = (int)threadIdx.x >> 3, col = 4 * ((int)threadIdx.x & 7);
        if (row < 16 && col < r) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < kOwnSlices; ++c) {
                if (c >= 1 << log) break;
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                    const float4 b = *reinterpret_cast<const float4*>(sums + ((c * 8 + w) * 16 + row) * (r + 8) + col);
                    sum.x += b.x; sum.y += b.y; sum.z += b.z; sum.w += b.w;
                }
                v.x += sum.x; v.y += sum.y; v.z += sum.z; v.w += sum.w;
            }
            *reinterpret_cast<uint2*>(T + row * (r + 8) + col) = make_uint2(pack_bf16x2(s * v.x, s * v.y), pack_bf16x2(s * v.z, s * v.w));
        }
        __syncthreads();
    }
};

// Grid: (row groups, for each the slices of the contraction; token tiles of all members).  Every slice has two slots, whose sums are added up
// first, then the slices' sums one after the other; where that happens does not change the result:
//   spread: a slice per CTA, a slot per half of its warps; the slices of a group are a cluster, and every CTA of it adds up a share of the rows,
//           which the others' warps write into its shared memory;
//   MERGED: one CTA does all slices of a group, each half of its warps every other half of them.  For grids of several waves: a CTA costs
//           about 4 us beside its steps (its launch in a cluster, the way from a row's number to its codes, a barrier of the cluster).
// OWN: one slice, and every CTA forms T itself (OwnT); no launch goes before this one.
template <int NT8, int NB, bool MERGED, int CTAS, bool OWN>
__global__ void __launch_bounds__(kSmallThreads, CTAS) small_kernel(const __grid_constant__ SmallParams<NB> P, const int slices) {
    extern __shared__ __align__(128) unsigned char small_smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (OWN) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (P.clear_status && blockIdx.x == 0 && threadIdx.x == 0) *P.status = 0u;
    }
    if (!MERGED) cluster_arrive();   // "this CTA runs": waited for before its shared memory is written from elsewhere
    constexpr int kTokens = 8 * NT8;
    constexpr uint32_t kTokenBytes = 2u * kTokens * kSmallSpan * 2u;     // two steps of one half of the warps
    float* sums = reinterpret_cast<float*>(small_smem + 2 * kTokenBytes);   // spread: [slots][tokens][share of the rows]; MERGED: see end()
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const OwnT own(reinterpret_cast<unsigned char*>(sums + 2 * kTokens * kSmallRows), P.K, P.r);
    if (OWN) own.fetch(P.m[0].A, P.K, P.r);
    const int rank = MERGED ? 0 : (int)ptx::cluster_ctarank();
    int grp = MERGED ? (int)blockIdx.x : ((int)gridDim.x - 1 - (int)blockIdx.x) >> (31 - __clz(slices));     // (spread: the long rows of 4 bits first)
    const Unit un = unit_at(P, (int)blockIdx.y, kTokens);
    const SmallMember& W = P.m[un.member];
    // the group's rows: 64 neighbouring stored rows of one precision class
    int c = 0;
    for (; c < 2; ++c) {
        const int n = (W.L.class_start[c + 1] - W.L.class_start[c] + kSmallRows - 1) / kSmallRows;
        if (grp < n) break;
        grp -= n;
    }
    const int p_first = W.L.class_start[c] + grp * kSmallRows, p_end = W.L.class_start[c + 1];
    const bool any = p_first < p_end;                                    // (members with other class counts have fewer groups)
    if (MERGED && !any) return;
    const int tile = warp & 3, half = warp >> 2;
    const int p0 = p_first + tile * 16;
    const int slots = slices * 2, slot0 = MERGED ? half * slices : rank * 2 + half, slot1 = MERGED ? slot0 + slices : slot0 + 1;
    const int share_log = 6 - (31 - __clz(slices)), share = 1 << share_log;
    // the up-projection's fragments for this warp's rows: steps of 16 ranks, dealt to the slots; a slot's first one is fetched
    // before its steps and put together when it is needed
    const uint16_t *u0 = W.B, *u1 = W.B;
    if (any && slot0 * 16 < P.r) {
        u0 += __ldg(W.L.perm + min(p0 + g, p_end - 1));
        u1 += __ldg(W.L.perm + min(p0 + g + 8, p_end - 1));
    }
    const size_t N = (size_t)P.N;
    uint32_t raw[8];
    auto fetch_up = [&](int step) {
        const size_t j = (size_t)(step * 16 + 2 * t) * N;
        raw[0] = __ldg(u0 + j); raw[1] = __ldg(u0 + j + N); raw[2] = __ldg(u0 + j + 8 * N); raw[3] = __ldg(u0 + j + 9 * N);
        raw[4] = __ldg(u1 + j); raw[5] = __ldg(u1 + j + N); raw[6] = __ldg(u1 + j + 8 * N); raw[7] = __ldg(u1 + j + 9 * N);
    };
    auto begin = [&](int slot) {
        if (slot * 16 < P.r) fetch_up(slot);
    };
    auto end = [&](int slot, float (&acc)[NT8][4]) {
        if constexpr (OWN) {             // (a warp has one slot, of one step at most: the second of two steps is the second half's)
            const uint32_t staged = ptx::smem_u32(small_smem);
            const bool two = P.K > kSmallSpan;
            own.form<NT8>(P.K, P.r, P.s, [&](int step) { return staged + (two && step == 0 ? 0u : kTokenBytes); });
            const int m = (int)threadIdx.x >> 4, col = 4 * ((int)threadIdx.x & 15);          // (the padded rank is 64)
            if (blockIdx.x == 0 && m < W.M)  // for the gradients
                *reinterpret_cast<uint2*>(W.T + (size_t)m * P.rp + col) = col < P.r ? *reinterpret_cast<const uint2*>(own.T + m * (P.r + 8) + col) : make_uint2(0u, 0u);
        } else {
            asm volatile("griddepcontrol.wait;" ::: "memory");           // T is in place
        }
        for (int i = slot; i * 16 < P.r; i += slots) {
            if (i != slot) fetch_up(i);
            const uint32_t a0 = raw[0] | (raw[1] << 16), a1 = raw[4] | (raw[5] << 16), a2 = raw[2] | (raw[3] << 16), a3 = raw[6] | (raw[7] << 16);
#pragma unroll
            for (int nt = 0; nt < NT8; ++nt) {
                const int m = un.m0 + nt * 8 + g;
                uint32_t b0 = 0u, b1 = 0u;
                if (OWN) {
                    const uint32_t* tr = reinterpret_cast<const uint32_t*>(own.T + (nt * 8 + g) * (P.r + 8) + i * 16) + t;
                    b0 = tr[0];
                    b1 = tr[4];
                } else if (m < W.M) {
                    const uint32_t* tr = reinterpret_cast<const uint32_t*>(W.T + (size_t)m * P.rp + i * 16) + t;
                    b0 = __ldcg(tr);
                    b1 = __ldcg(tr + 4);
                }
                mma_bf16(acc[nt], a0, a1, a2, a3, b0, b1);
            }
        }
        if (MERGED) {
            // Tiles of sums: 0 that of the first half's slices so far, 1 its slot that waits for the slice's other one, 2 + i the
            // second half's slice i.  Every thread reads and writes its own places.
            const int i = (slot - slot0) >> 1;
            const bool odd = (slot & 1) != 0;
            float* at = sums + (half == 0 ? (i == 0 ? 0 : 1) : 2 + i) * (kTokens * kMergedPitch) + 2 * t * kMergedPitch + tile * 16 + g;
            float* first = sums + 2 * t * kMergedPitch + tile * 16 + g;
#pragma unroll
            for (int nt = 0; nt < NT8; ++nt) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int o = (nt * 8 + (e & 1)) * kMergedPitch + (e >> 1) * 8;
                    const float sum = odd ? at[o] + acc[nt][e] : acc[nt][e];
                    if (half == 0 && odd && i > 0) first[o] += sum;
                    else at[o] = sum;
                }
            }
        } else {
            const uint32_t to = ptx::smem_u32(sums) + (uint32_t)((slot * kTokens + 2 * t) << share_log) * 4u;
            cluster_wait();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = tile * 16 + 8 * h + g;
                const uint32_t at = ptx::map_to_cta(to + (uint32_t)(row & (share - 1)) * 4u, (uint32_t)(row >> share_log));
#pragma unroll
                for (int nt = 0; nt < NT8; ++nt) {
                    st_cluster_f32(at + (uint32_t)((nt * 8) << share_log) * 4u, acc[nt][2 * h]);
                    st_cluster_f32(at + (uint32_t)((nt * 8 + 1) << share_log) * 4u, acc[nt][2 * h + 1]);
                }
            }
        }
    };
    if (any) {
        const uint32_t xs = ptx::smem_u32(small_smem) + (uint32_t)half * kTokenBytes;
        if (c == 0) multiply_rows<1, NT8>(P.K, W, un.m0, p0, p_end, slot0, slot1, slots, xs, half, begin, end);
        else if (c == 1) multiply_rows<2, NT8>(P.K, W, un.m0, p0, p_end, slot0, slot1, slots, xs, half, begin, end);
        else multiply_rows<4, NT8>(P.K, W, un.m0, p0, p_end, slot0, slot1, slots, xs, half, begin, end);
    } else {
        cluster_wait();
    }
    if (MERGED) {
        __syncthreads();
        for (int i = threadIdx.x; i < kTokens * kSmallRows; i += kSmallThreads) {
            const int m = i / kSmallRows, row = i % kSmallRows;
            if (un.m0 + m >= W.M || p_first + row >= p_end) continue;
            const float* from = sums + m * kMergedPitch + row;
            float sum = from[0];
            for (int s = 0; s < slices / 2; ++s) sum += from[(2 + s) * (kTokens * kMergedPitch)];
            W.Y[(size_t)(un.m0 + m) * P.N + __ldg(W.L.perm + p_first + row)] = (uint16_t)pack_bf16x2(sum, 0.0f);
        }
        return;
    }
    ptx::cluster_sync();
    for (int i = threadIdx.x; any && i < (kTokens << share_log); i += kSmallThreads) {
        const int m = i >> share_log, row = (rank << share_log) + (i & (share - 1));
        if (un.m0 + m >= W.M || p_first + row >= p_end) continue;
        float sum = 0.0f;
        for (int s = 0; s < slices; ++s) sum += sums[((2 * s * kTokens) << share_log) + i] + sums[(((2 * s + 1) * kTokens) << share_log) + i];
        W.Y[(size_t)(un.m0 + m) * P.N + __ldg(W.L.perm + p_first + row)] = (uint16_t)pack_bf16x2(sum, 0.0f);
    }
}

// ------------------------------------------------------------------------------------------------ several units of one weight
// Token groups of several adapters on one weight, and groups of more than 32 tokens: a CTA takes 64 rows as above and one unit of up to 32 tokens,
// and does all slices of the contraction.  No cluster, and every unit is as many eights of tokens wide as it has.  The halves of the warps take a
// slot of every slice each; the second half hands its sums to the first one's threads, which hold the same places, add them up in the
// order of the other two forms - a group's result does not depend on its company, nor on the kernel - and store them.
// The CTAs go out in the order of their length, so that the last ones, which leave SMs idle, are short: by precision and width of the unit together
// (unit_cost; by precision alone 26 % of the SMs' time was idle: six groups of 101 tokens on 4096 x 4096 at 30/50/20 % 51 -> 43.8 us, at 85/15 % 45.9 -> 39.6).
constexpr int kUnitTokens = 32;
constexpr int kUnitRuns = 3 * 2 * kSmallMembers;
struct UnitOrder {                               // runs of CTAs: a unit's row groups of one precision
    int32_t count, end[kUnitRuns];               // end: the first CTA after the run
    uint8_t member[kUnitRuns], first[kUnitRuns], cls[kUnitRuns];     // the unit's member, and its first token in units
};

__device__ __forceinline__ void barrier_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

template <int B, int NT8, int NB>
__device__ __forceinline__ void unit_rows(const SmallParams<NB>& P, const SmallMember& W, int m0, int p0, int p_end, int slices, unsigned char* smem) {
    constexpr uint32_t kStep = 8u * NT8 * kSmallSpan * 2u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, half = warp >> 2;
    const int K = P.K, n_span = (K + kSmallSpan - 1) / kSmallSpan, nb = K / kBlock, slots = 2 * slices;
    const int slots_log = 31 - __clz(slots);          // (a power of two; n_span is below 2^27: K is an int32)
    auto bound = [&](int slot) { return (int)(((long long)slot * n_span) >> slots_log); };
    const bool live0 = p0 + g < p_end, live1 = p0 + g + 8 < p_end;
    const int q0 = live0 ? p0 + g : p_end - 1, q1 = live1 ? p0 + g + 8 : p_end - 1;
    const int r0 = __ldg(W.L.perm + q0), r1 = __ldg(W.L.perm + q1);
    const uint8_t* row0 = W.packed + packed_row_offset(W.L, B >> 1, q0, r0) + t * (8 * B);
    const uint8_t* row1 = W.packed + packed_row_offset(W.L, B >> 1, q1, r1) + t * (8 * B);
    const float* am0 = W.absmax + (size_t)absmax_row_of(W.L, q0, r0) * nb + t;
    const float* am1 = W.absmax + (size_t)absmax_row_of(W.L, q1, r1) * nb + t;
    const float* y0 = W.maps + (size_t)r0 * kTableStride;
    const float* y1 = W.maps + (size_t)r1 * kTableStride;
    // tokens of a step: two buffers for either half of the warps; a warp to every fourth token, a lane to a 16-byte piece of its 512 bytes
    const uint32_t x_smem = ptx::smem_u32(smem) + (uint32_t)half * 2u * kStep;
    float* handed = reinterpret_cast<float*>(smem + 4u * kStep) + (threadIdx.x & 127);      // two buffers of [4 NT8][128 threads]
    float* total = handed + 2 * (4 * NT8 * 128);                                            // the slices so far, likewise
    const int warp4 = warp & 3, tokens = W.M - m0 - warp4;
    const uint32_t stage_at = x_smem + token_piece(warp4, lane >> 3, lane & 7), read_at = x_smem + token_piece(g, t, 0);
    const uint16_t* x_src = W.X + (size_t)(m0 + warp4) * K + lane * 8;
    auto stage = [&](int b, uint32_t turn) {
        const int k = b * kSmallSpan;
        const bool in = k + lane * 8 < K;
        const uint16_t* src = x_src + k;
#pragma unroll
        for (int i = 0; i < 2 * NT8; ++i) {
            const bool valid = in && 4 * i < tokens;
            cp_async_16_zfill(stage_at + turn * kStep + (uint32_t)(4 * i * kSmallSpan * 2), valid ? src + (size_t)(4 * i) * K : W.X, valid);
        }
    };
    Codes<B> n0, n1;
    auto fetch = [&](int b) {
        const bool in = 4 * b + t < nb;
        fetch_codes<B>(n0, row0, am0, 4 * b, live0 && in);
        fetch_codes<B>(n1, row1, am1, 4 * b, live1 && in);
    };
    uint32_t raw[8];
    auto fetch_up = [&](int step) {
        const size_t N = (size_t)P.N, j = (size_t)(step * 16 + 2 * t) * N;
        const uint16_t *u0 = W.B + r0 + j, *u1 = W.B + r1 + j;
        raw[0] = __ldg(u0); raw[1] = __ldg(u0 + N); raw[2] = __ldg(u0 + 8 * N); raw[3] = __ldg(u0 + 9 * N);
        raw[4] = __ldg(u1); raw[5] = __ldg(u1 + N); raw[6] = __ldg(u1 + 8 * N); raw[7] = __ldg(u1 + 9 * N);
    };
    float ya[1 << B], yb[1 << B];
    if (B <= 2) {
        load_levels<B>(ya, y0);
        load_levels<B>(yb, y1);
    }
    uint32_t turn = 0u;
    if (bound(half) < bound(half + 1)) {
        fetch(bound(half));
        stage(bound(half), 0u);
    }
    ptx::cp_async_commit();
#pragma unroll 1
    for (int slice = 0; slice < slices; ++slice) {
        const int slot = 2 * slice + half, b1 = bound(slot + 1), after = slice + 1 < slices ? bound(slot + 2) : -1;
        float acc[NT8][4];
#pragma unroll
        for (int i = 0; i < NT8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
        if (slot * 16 < P.r) fetch_up(slot);
#pragma unroll 1
        for (int b = bound(slot); b < b1; ++b) {
            ptx::cp_async_wait<0>();
            ptx::named_barrier_sync(1 + half, 128);      // the step's tokens are there, those of the step before have been read
            const int next = b + 1 < b1 ? b + 1 : after;
            const Codes<B> c0 = n0, c1 = n1;
            if (next >= 0) {
                stage(next, turn ^ 1u);
                fetch(next);
            }
            ptx::cp_async_commit();
            Scaled<B> s0, s1;
            if (B == 4) {   // (sixteen levels of two rows are too many registers to keep: read again, from L1)
                load_levels<B>(ya, y0);
                s0.set(ya, c0.a);
                load_levels<B>(ya, y1);
                s1.set(ya, c1.a);
            } else {
                s0.set(ya, c0.a);
                s1.set(yb, c1.a);
            }
            const uint32_t xs = read_at + turn * kStep;
#pragma unroll
            for (int q = 0; q < 4; ++q) multiply_16<B, NT8>(acc, s0, s1, c0, c1, q, xs);
            turn ^= 1u;
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");               // T is in place
        for (int i = slot; i * 16 < P.r; i += slots) {
            if (i != slot) fetch_up(i);
            const uint32_t a0 = raw[0] | (raw[1] << 16), a1 = raw[4] | (raw[5] << 16), a2 = raw[2] | (raw[3] << 16), a3 = raw[6] | (raw[7] << 16);
#pragma unroll
            for (int nt = 0; nt < NT8; ++nt) {
                const int m = m0 + nt * 8 + g;
                uint32_t t0 = 0u, t1 = 0u;
                if (m < W.M) {
                    const uint32_t* tr = reinterpret_cast<const uint32_t*>(W.T + (size_t)m * P.rp + i * 16) + t;
                    t0 = __ldcg(tr);
                    t1 = __ldcg(tr + 4);
                }
                mma_bf16(acc[nt], a0, a1, a2, a3, t0, t1);
            }
        }
        // the slice's two sums: buffer slice mod 2 full (barriers 3, 4), and read (5, 6)
        float* at = handed + (slice & 1) * (4 * NT8 * 128);
        if (half == 1) {
            if (slice >= 2) ptx::named_barrier_sync(5 + (slice & 1), 256);
#pragma unroll
            for (int i = 0; i < 4 * NT8; ++i) at[i * 128] = acc[i >> 2][i & 3];
            barrier_arrive(3 + (slice & 1), 256);
        } else {
            ptx::named_barrier_sync(3 + (slice & 1), 256);
#pragma unroll
            for (int i = 0; i < 4 * NT8; ++i) acc[i >> 2][i & 3] = (slice > 0 ? total[i * 128] : 0.0f) + (acc[i >> 2][i & 3] + at[i * 128]);
            if (slice + 2 < slices) barrier_arrive(5 + (slice & 1), 256);
            if (slice + 1 < slices) {
#pragma unroll
                for (int i = 0; i < 4 * NT8; ++i) total[i * 128] = acc[i >> 2][i & 3];
                continue;
            }
#pragma unroll
            for (int nt = 0; nt < NT8; ++nt) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int m = m0 + nt * 8 + 2 * t + e;
                    if (m >= W.M) continue;
                    if (live0) W.Y[(size_t)m * P.N + r0] = (uint16_t)pack_bf16x2(acc[nt][e], 0.0f);
                    if (live1) W.Y[(size_t)m * P.N + r1] = (uint16_t)pack_bf16x2(acc[nt][2 + e], 0.0f);
                }
            }
        }
    }
}

template <int NB>
__global__ void __launch_bounds__(kSmallThreads, 2) units_kernel(const __grid_constant__ SmallParams<NB> P, const __grid_constant__ UnitOrder order, const int slices) {
    extern __shared__ __align__(128) unsigned char small_smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int run = 0, above = order.count - 1;
    while (run < above) {
        const int mid = (run + above) >> 1;
        if ((int)blockIdx.x < order.end[mid]) above = mid;
        else run = mid + 1;
    }
    const SmallMember& W = P.m[order.member[run]];
    const int m0 = order.first[run] * kUnitTokens, c = order.cls[run], grp = (int)blockIdx.x - (run > 0 ? order.end[run - 1] : 0);
    const int p0 = W.L.class_start[c] + grp * kSmallRows + (int)((threadIdx.x >> 5) & 3) * 16, p_end = W.L.class_start[c + 1];
    const int tokens = W.M - m0;
    auto work = [&](auto bits) {
        constexpr int B = decltype(bits)::value;
        if (tokens <= 8) unit_rows<B, 1, NB>(P, W, m0, p0, p_end, slices, small_smem);
        else if (tokens <= 16) unit_rows<B, 2, NB>(P, W, m0, p0, p_end, slices, small_smem);
        else if (tokens <= 24) unit_rows<B, 3, NB>(P, W, m0, p0, p_end, slices, small_smem);
        else unit_rows<B, 4, NB>(P, W, m0, p0, p_end, slices, small_smem);
    };
    if (c == 0) work(std::integral_constant<int, 1>());
    else if (c == 1) work(std::integral_constant<int, 2>());
    else work(std::integral_constant<int, 4>());
}

// Whether a CTA for every group of 64 rows and unit beats one for every slice of it, for a weight of n[0], n[1], n[2] channels at 1, 2 and 4 bits and so many
// units, the largest member of `most` tokens.  Both in microseconds, two CTAs to an SM: of the former 3 and 1.2 for every slice, of the latter 5.5; and
// 2 (1, 2 bits) to 2.6 (4 bits) for a step.  The long ones leave SMs idle at the end, more so where all are alike; a few of them with rows of 4 bits, more
// than 16 tokens and ranks up to 64 are 1.5 slower.  Over 288 calls that take units (256 to 13824 channels, 512 to 13824 features, 2 to 8 groups, single calls of
// 33 to 64 tokens, ranks 16 to 128, six mixes) they take 0.90 of the slices' time in the mean; the choice is 0.5 % behind the better form, 10 % at most,
// and 10 calls are more than 3 % behind the slices (25 without the 1.5: 264 x 512, 44 tokens at 2 and 4 bits 7.9 us, 9.1 by units).
// (Against the slices, us: 4096 x 4096 at 30/50/20 %, 101 tokens in 6 groups 66.0 -> 48.6 (43 in order of length), 64 in 8 72 -> 46, 60 in 3 34.4 -> 29.9, 16 in
// 8 48.5 -> 38.7; at 4 bits 101 in 6 66.4 -> 55.4.  Not taken: 4 in 2 there 19.3 -> 19.8, 64 in one 26.9 -> 31.5; 4096 x 11008 of 4 bits 60 in 3 71 -> 83.)
bool units_faster(const int* n, int K, int r, int units, int most, int slices) {
    if (units < 2) return false;
    const int N = n[0] + n[1] + n[2], ctas = ((n[0] + 63) / 64 + (n[1] + 63) / 64 + (n[2] + 63) / 64) * units;
    const bool alike = n[0] == N || n[1] == N || n[2] == N;
    const float wide = n[2] > 0 && most > 16 && r <= 64 && ctas <= kNumSMs ? 1.5f : 0.0f;
    const float step = 2.0f + 0.6f * (float)n[2] / (float)N, steps = 0.5f * (float)((K + kSmallSpan - 1) / kSmallSpan);
    const float waves = (float)ctas / (2 * kNumSMs), spread = waves * slices, whole = waves + (alike ? 0.35f : 0.15f);
    return (whole > 1.0f ? whole : 1.0f) * (3.0f + wide + 1.2f * slices + step * steps) < (spread > 1.0f ? spread : 1.0f) * (5.5f + step * steps / slices);
}

template <int NB>
bool units_pay(const SmallParams<NB>& P, int slices) {
    int units = 0, most = 0;
    for (int i = 0; i < P.count; ++i) {
        units += (P.m[i].M + kUnitTokens - 1) / kUnitTokens;
        most = P.m[i].M > most ? P.m[i].M : most;
    }
    const int* start = P.m[0].L.class_start;
    const int n[3] = {start[1] - start[0], start[2] - start[1], start[3] - start[2]};
    return units_faster(n, P.K, P.r, units, most, slices);
}

// How long a CTA takes at so many bits (class) and eights of tokens, relative to the others (us on 4096 features, several at a time).
float unit_cost(int cls, int eights) {
    constexpr float kCost[3][4] = {{13.7f, 17.0f, 18.8f, 22.4f}, {19.7f, 23.7f, 25.9f, 28.9f}, {27.0f, 30.0f, 33.0f, 36.5f}};
    return kCost[cls][eights - 1];
}

template <int NB>
lowra_status launch_units(const SmallParams<NB>& P, int slices, cudaStream_t stream) {
    struct Run { float cost; int groups; uint8_t member, first, cls; } runs[kUnitRuns];
    int n = 0, widest = 1;
    for (int i = 0; i < P.count; ++i) {
        const SmallMember& m = P.m[i];
        for (int u = 0; u * kUnitTokens < m.M; ++u) {
            const int left = m.M - u * kUnitTokens, eights = left < kUnitTokens ? (left + 7) / 8 : kUnitTokens / 8;
            widest = eights > widest ? eights : widest;
            for (int c = 0; c < 3; ++c) {
                const Run run = {unit_cost(c, eights), (m.L.class_start[c + 1] - m.L.class_start[c] + kSmallRows - 1) / kSmallRows, (uint8_t)i, (uint8_t)u, (uint8_t)c};
                if (run.groups == 0) continue;
                int at = n++;
                for (; at > 0 && runs[at - 1].cost < run.cost; --at) runs[at] = runs[at - 1];
                runs[at] = run;
            }
        }
    }
    UnitOrder order;
    order.count = n;
    int ctas = 0;
    for (int i = 0; i < n; ++i) {
        ctas += runs[i].groups;
        order.end[i] = ctas;
        order.member[i] = runs[i].member;
        order.first[i] = runs[i].first;
        order.cls[i] = runs[i].cls;
    }
    const size_t smem = 4u * (8 * widest) * kSmallSpan * 2u + 3u * 4 * widest * 128 * 4u;
    static SmemLimit limit = {};
    if (ensure_smem_limit(reinterpret_cast<const void*>(units_kernel<NB>), smem, &limit) != LOWRA_OK) return LOWRA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(kSmallThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, units_kernel<NB>, P, order, slices) == cudaSuccess ? LOWRA_OK : LOWRA_ERR_CUDA;
}

template <int NT8, int NB, bool MERGED, int CTAS, bool OWN = false>
lowra_status launch_product(const SmallParams<NB>& P, int groups, int units, int slices, cudaStream_t stream) {
    const size_t smem = 4u * (8 * NT8) * kSmallSpan * 2u + (MERGED ? (2 + slices / 2) * (8 * NT8) * kMergedPitch * 4u : 2u * (8 * NT8) * kSmallRows * 4u) +
                        (OWN ? OwnT::bytes(P.K, P.r) : 0);
    static SmemLimit limit = {};
    if (ensure_smem_limit(reinterpret_cast<const void*>(small_kernel<NT8, NB, MERGED, CTAS, OWN>), smem, &limit) != LOWRA_OK) return LOWRA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)slices;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(MERGED ? groups : groups * slices), (unsigned)units, 1);
    cfg.blockDim = dim3(kSmallThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = MERGED || slices == 1 ? 1 : 2;           // (a CTA is a cluster of its own without being told, and 0.4 us less host time)
    return cudaLaunchKernelEx(&cfg, small_kernel<NT8, NB, MERGED, CTAS, OWN>, P, slices) == cudaSuccess ? LOWRA_OK : LOWRA_ERR_CUDA;
}

int product_slices(int N, int K) {
    const int n_span = (K + kSmallSpan - 1) / kSmallSpan, by_shape = (N + kSmallRows - 1) / kSmallRows;
    int slices = 1;
    while (slices < 8 && 4 * slices <= n_span && 2 * slices * by_shape <= 3 * kNumSMs) slices *= 2;
    return slices;
}

// Whether a grid of so many CTAs beside so many of the projection runs in one wave, two to an SM (clusters of eight and four leave SMs of a GPC over).
bool two_fit(int slices, int ctas, int projection) { return ctas + projection <= (slices == 8 ? 272 : slices == 4 ? 280 : 2 * kNumSMs); }

// Whether the spread form runs three CTAs to an SM, at 80 registers (some of which spill, most at 4 bits), or two at 128: `four` of N channels at 4 bits.  Measured
// over 32 shapes, six mixes, ranks 16 to 128, 1 to 24 tokens; two against three, us, in a captured graph:
//   two do not fit in one wave   three (6144 x 4096 at 60/35/5, 16 tokens, rank 64 16.4 13.1; all mixes and ranks 0.70 to 1.09 of the time), but for long steps with most rows at 4 bits
//   two fit                      two (1024 x 2048 at 60/35/5, 16 tokens, rank 16 5.4 6.2; 4096 x 1024, rank 32 6.3 7.2), but for four slices on nearly all SMs and short steps at
//                                ranks 48 and 64, from 9 tokens on without 4-bit rows (4096 x 4096 at 85/15, 16 tokens, rank 64 10.7 10.1), and 32 with up to 8 tokens and none
bool three_pay(int four, int N, int r, int n_span, int slices, int ctas, int projection, int nt8) {
    if (nt8 > 3) return false;                           // (no shared memory for a third)
    const bool short_steps = n_span <= 2 * (2 * slices);
    if (!two_fit(slices, ctas, projection)) return short_steps || four <= N / 2;
    if (slices != 4 || ctas < 128 || !short_steps || r > 64 || nt8 > 2) return false;
    return nt8 == 1 ? (four == 0 ? r > 16 : four <= N / 8 && r > 32) : four == 0 && r > 32;
}

// groups of 64 stored rows of one precision (of the member that has the most)
template <int NB>
int row_groups(const SmallParams<NB>& P) {
    int groups = 0;
    for (int i = 0; i < P.count; ++i) {
        int n = 0;
        for (int c = 0; c < 3; ++c) n += (P.m[i].L.class_start[c + 1] - P.m[i].L.class_start[c] + kSmallRows - 1) / kSmallRows;
        groups = n > groups ? n : groups;
    }
    return groups;
}

// Whether every CTA of a small weight (`groups` CTAs, `four` channels of 4 bits) forms T itself instead of a launch before it.  That saves a launch, 2.5 us of host time, which all
// calls show that allocate their output and scratch, and costs every CTA the reading of A and a chain of its own, which shows where the host is ahead.  One launch against two, us, nothing
// kept / output and workspace kept / in a captured graph:
//   512 x 512 at 50/50, rank 16, 8 tokens   5.4 8.0 / 4.9 5.9 / 4.5 4.0      256 x 256 at 50/50, rank 16, 16 tokens   5.3 7.7 / 4.6 5.7 / 4.2 4.5
//   at 60/35/5, rank 32, 16 tokens          6.8 8.0 / 6.8 5.9 / 6.4 5.6      4096 x 384 of 4 bits, rank 16, 16 tokens 6.9 7.9 / 7.6 6.1 / 5.9 5.6
// Not with ranks above 16 on more than 40 groups of rows, which each read so much of A (4096 x 384 at 60/35/5, rank 32, 16 tokens 8.7 7.9 / 8.6 7.1 / 7.4 6.2), nor above 256
// features with slow rows on more than 40 for more than 8 tokens (3072 x 512 of 4 bits, rank 16, 9 tokens 6.9 8.0 / 7.9 5.9 / 5.9 5.2) or 80 for fewer (8192 x 384 at 60/35/5, rank
// 16, 1 token 5.5 8.0 / 6.5 5.9 / 6.0 4.5).
bool forms_own_t(int K, int r, int tokens, int groups, int four) {
    if (K > kOwnK || r > kOwnRank || tokens > 16) return false;
    return groups <= (r > 16 ? 40 : K <= 256 || four == 0 ? kNumSMs : tokens > 8 ? 40 : 80);
}

template <int NB>
lowra_status launch_members(const SmallParams<NB>& P, cudaStream_t stream) {
    int m16 = 0, most = 0;
    const int groups = row_groups(P);
    for (int i = 0; i < P.count; ++i) {
        const SmallMember& m = P.m[i];
        m16 += (m.M + 15) / 16;
        most = m.M > most ? m.M : most;
    }
    const int n_span = (P.K + kSmallSpan - 1) / kSmallSpan, slices = product_slices(P.N, P.K);
    if constexpr (NB == 1) {
        const int* start = P.m[0].L.class_start;
        if (slices == 1 && forms_own_t(P.K, P.r, most, groups, start[3] - start[2]))
            return most <= 8 ? launch_product<1, NB, false, 2, true>(P, groups, 1, 1, stream) : launch_product<2, NB, false, 2, true>(P, groups, 1, 1, stream);
    }
    // ---- T: the contraction over up to eight CTAs, 128 indices or more each
    {
        const int slices = project_slices(P.K);
        const size_t smem = project_fetch_bytes(P.r) + (size_t)16 * P.r * 4;
        static SmemLimit limit = {};
        if (ensure_smem_limit(reinterpret_cast<const void*>(project_kernel<NB>), smem, &limit) != LOWRA_OK) return LOWRA_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)slices;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3((unsigned)slices, (unsigned)m16, 1);
        cfg.blockDim = dim3(kSmallThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        if (cudaLaunchKernelEx(&cfg, project_kernel<NB>, P) != cudaSuccess) return LOWRA_ERR_CUDA;
    }
    // ---- the product: slices of the contraction until the grid is about three CTAs per two places, as long as every warp keeps
    // a step of 256.  The choice depends on the weight's shape alone, so that a member's result does not depend on its company.
    const int nt8 = most <= 8 ? 1 : most <= 16 ? 2 : most <= 24 ? 3 : 4;
    if (P.one_weight && units_pay(P, slices)) return launch_units<NB>(P, slices, stream);
    int units = 0;
    for (int i = 0; i < P.count; ++i) units += (P.m[i].M + 8 * nt8 - 1) / (8 * nt8);
    // Merged where a CTA's own cost outweighs its steps: slots of one or two steps, few tokens, more CTAs than run at a time.  (Groups of
    // adapters on 4096 x 4096 at 30/50/20 %: 8 tokens in 4 groups 26.0 against 34.6 us spread, 16 in 8 48.5 against 60.0; but with up to 32
    // tokens a group 64 in 2 38.5 against 34.8; on 4096 x 11008 - slots of five steps - 6 in 3 54.5 against 46.1; one group 18.8 against 10.6.)
    if constexpr (NB > 1) {
        if (slices > 1 && nt8 <= 2 && n_span <= 2 * (2 * slices) && groups * slices * units > 2 * kNumSMs)
            return nt8 == 1 ? launch_product<1, NB, true, 2>(P, groups, units, slices, stream) : launch_product<2, NB, true, 2>(P, groups, units, slices, stream);
    }
    const int* start = P.m[0].L.class_start;
    const bool three = three_pay(start[3] - start[2], P.N, P.r, n_span, slices, groups * slices * units, 8 * m16, nt8);
    if (nt8 == 1) return three ? launch_product<1, NB, false, 3>(P, groups, units, slices, stream) : launch_product<1, NB, false, 2>(P, groups, units, slices, stream);
    if (nt8 == 2) return three ? launch_product<2, NB, false, 3>(P, groups, units, slices, stream) : launch_product<2, NB, false, 2>(P, groups, units, slices, stream);
    if (nt8 == 3) return three ? launch_product<3, NB, false, 3>(P, groups, units, slices, stream) : launch_product<3, NB, false, 2>(P, groups, units, slices, stream);
    return launch_product<4, NB, false, 2>(P, groups, units, slices, stream);
}

}  // namespace

// An estimate of a call's time in microseconds for so many units of up to 32 tokens, the largest member of `most`, on one weight of n[0], n[1], n[2] channels at
// 1, 2 and 4 bits: 2.8 for the projection and the start, then CTAs, two to an SM.  A step of 256 takes 2.5, 0.45 more at 4 bits; around a CTA's steps and its
// share of the low-rank term 5.4, and if it is alone on its SM all that takes 0.64 of it.  A CTA that does all slices takes 3.7 and 1.2 for every slice around its
// steps, of which two halves overlap (0.74), and waits 1.7 for 4-bit rows among others; of three on an SM the third does not wait for both.  Fitted to 520
// calls (256 to 13824 channels, 512 to 13824 features, ranks 16 to 128, six mixes): within 18 %.  Where two CTAs to an SM are more than one wave (and three may
// share it), 0.85 of that.
float small_estimate(const int32_t* n, int K, int r, int units, int most) {
    const int N = n[0] + n[1] + n[2], slices = product_slices(N, K);
    const int groups = (n[0] + kSmallRows - 1) / kSmallRows + (n[1] + kSmallRows - 1) / kSmallRows + (n[2] + kSmallRows - 1) / kSmallRows;
    const float rank = (float)r / 64.0f, step = 2.5f + 0.45f * (float)n[2] / (float)N, steps = 0.5f * (float)((K + kSmallSpan - 1) / kSmallSpan);
    const bool mixed = n[2] > 0 && n[2] < N;
    auto per_sm = [](int ctas) { return (ctas + kNumSMs - 1) / kNumSMs; };
    if (units_faster(n, K, r, units, most, slices)) {
        const int k = per_sm(groups * units);
        return 2.8f + (mixed ? 1.7f : 0.0f) + (3.7f + 1.2f * slices + 2.1f * rank + 0.74f * step * steps) * (k == 1 ? 0.64f : k == 2 ? 1.15f : 0.5f * k);
    }
    const int k = per_sm(groups * slices * units), n_span = (K + kSmallSpan - 1) / kSmallSpan;
    const bool packed = most <= 24 && !two_fit(slices, groups * slices * units, 8 * ((most + 15) / 16)) && (n_span <= 2 * (2 * slices) || n[2] <= N / 2);
    const float three = packed ? 0.85f : 1.0f;
    return 2.8f + (mixed ? 0.3f : 0.0f) + three * (5.4f + (2.2f * rank + step * steps) / slices) * (k / 2 + (k % 2 != 0 ? 0.64f : 0.0f));
}

bool small_takes_units(const SmallParams<kSmallMembers>& P) { return P.one_weight && units_pay(P, product_slices(P.N, P.K)); }

// (A call with one member carries 0.3 KB of kernel parameters instead of 1.5 KB, which its launches show.)
lowra_status launch_small(const SmallParams<kSmallMembers>& P, cudaStream_t stream) {
    if (P.count > 1) return launch_members<kSmallMembers>(P, stream);
    SmallParams<1> Q;
    Q.m[0] = P.m[0];
    Q.count = 1; Q.N = P.N; Q.K = P.K; Q.r = P.r; Q.rp = P.rp; Q.s = P.s; Q.status = P.status; Q.clear_status = P.clear_status; Q.one_weight = P.one_weight;
    return launch_members<1>(Q, stream);
}

}  // namespace lowra
