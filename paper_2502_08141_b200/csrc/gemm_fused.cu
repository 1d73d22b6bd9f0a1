// Fused dequant + LoRA tensor-core kernel (forward, backward-input, and a dense diagnostic mode).
//
// Persistent CTA pairs (clusters of two, one CTA per SM) walk over output tiles of 256 "operand rows" x 512 tokens:
//   forward : operand rows = output channels n;  Y tile [512 m x 256 n]  = X[m, :] . W_hat[n, :]
//   backward: operand rows = input features k;   dX tile [512 m x 256 k] = dY[m, :] . W_hat[:, k]
// The tokens (activations / output gradients) are the A operand of tcgen05.mma with cta_group::2, 256 of them at a time, and
// the operand rows (the weights) the B operand: either CTA of the pair keeps 128 tokens of each half and 128 operand rows in
// its shared memory, and receives its 128 tokens x 256 rows of the product in its tensor memory - a lane is a token, so the
// epilogue stores runs of neighbouring rows straight from registers.
// The tokens arrive by TMA.  Sixteen dequant warps per CTA produce the weights in shared memory from the packed codes
// (never from HBM as bf16), one 128-byte row per 64-element absmax block: K-major in the forward pass (a thread keeps one
// output channel for the whole tile), MN-major in the backward pass (every stage brings 64 new channels, dealt to the warps by
// the prologue).
// What paces the kernel.  The tensor core takes about 790 cycles for 256 tokens x 256 rows x 64 contraction indices per pair.
// A warp's visit to a stage - codes from registers, slot wait, 64 elements per lane expanded and stored, proxy fence, arrival -
// takes 2400 to 4300 cycles, nearly all of it latency of the shared-memory pipe that the tensor core keeps busy.  So (a) a
// dequantised weight serves 512 tokens, two MMAs, and (b) sixteen warps overlap their visits.  With eight warps and 256 tokens
// this kernel ran at 490 - 610 TFLOP/s on an 11008 x 4096 weight, with the weights left as zeros at 1520; the form before it (one-CTA
// MMAs of 128 x 256, a dequantised tile copied to the peer CTA over the cluster) at 1060 - 1100.
// The two accumulators of a tile (one per half of its tokens) fill the tensor memory.  So that the epilogue still overlaps the main
// loop, the first and the last kSkew stages of a tile are worked on half by half: the first half's accumulator is drained
// while the second half's last stages run, the second half's while the next tile's first half starts.
// The LoRA term is folded into the same accumulator as extra contraction blocks at the end of every tile: the
// up-projection factor comes by TMA straight from the caller's matrix, the down-projected activations T = s X A (resp.
// U = s dY B^T) by TMA from the workspace.  T itself is produced by this same kernel: for every token tile there is one
// extra "T tile" whose operand rows are the ranks, padded to 128.  T tiles come first in the tile order, their epilogue raises
// a flag per CTA, and the TMA producer of a regular tile waits (bounded) for that flag before it fetches T.  All CTAs are
// co-resident and a T tile waits for nothing but the other clusters that share it, so the wait cannot deadlock.
// Schedule: whole tiles dealt round-robin to the pairs, or (launcher's choice) ranges: equal consecutive pieces of the
// remaining weight tiles' contraction blocks per pair, partial tiles handed over through a scratch slot and added in the
// epilogue of the pair that starts the tile; or, in calls of few tiles, tiles shared by several pairs, each of which finishes some of
// the tile's columns (see the schedule in the kernel).
//
// Warp roles: 0 = TMA producer, 1 = MMA issuer (in the CTA of rank 0) and TMEM owner, 2-9 = epilogue, 10-25 = dequant.
// All mbarrier waits are bounded; a wait that runs out sets the status word and every role leaves.
#include <mutex>

#include "dequant.cuh"
#include "gemm_params.cuh"
#include "ptx.cuh"

namespace lowra {

namespace {

constexpr uint64_t kGraceNs = 50ull * 1000ull;   // after a failure: time for copies and MMAs still in flight to land
constexpr int kMinRange = 12;                    // schedule (plan_schedule): the shortest range of contraction blocks
constexpr int kMinShare = 8;                     // and a cluster's share of a T tile of two such ranges or more
constexpr int kTFlags = 8;                       // "T ready" flags of a CTA and token tile whose T is shared out
// Collecting partial tiles: they come in pieces of 32 rows x 128 tokens (16 KB, a ring entry), two rows' worth of pieces - one for
// either warp of a lane quarter - from every contributor per step.
constexpr int kPartSlots = kSlotsX + kSlotsW, kMaxContributors = kPartSlots / 2, kPartSteps = kPartSlots / 2;
// Where they start among the header's flags, behind those of the partial tiles: 32-byte aligned, for they are read together.
constexpr int kSharedTFlags = (kMaxClusters * kCluster + 7) / 8 * 8;
static_assert(kMaxContributors <= kTFlags, "a flag for every cluster that shares a T tile");
constexpr int kRankCols = 128;                   // columns of a T tile: the ranks, padded
static_assert(2 * kRankCols <= kPairR, "two T tiles in the place of one partial tile");
constexpr uint32_t kIdesc = ptx::umma_idesc_bf16(kHalfT, kPairR), kIdescT = ptx::umma_idesc_bf16(kHalfT, kRankCols);
constexpr uint32_t kIdescBmn = 1u << 16;         // operand B MN-major

struct Barriers {
    uint64_t full_x[kSlotsX];       // (rank 0) the TMA bytes of a ring entry have landed in both CTAs
    uint64_t empty_x[kSlotsX];      // the MMAs reading a ring entry have completed (raised in both CTAs)
    uint64_t full_w[kSlotsW];       // (rank 0) the dequant warps of both CTAs have filled a weight slot
    uint64_t empty_w[kSlotsW];      // the MMAs reading a weight slot have completed (raised in both CTAs)
    uint64_t tmem_full[2];          // an accumulator is complete (raised in both CTAs)
    uint64_t tmem_empty[2];         // (rank 0) the epilogue warps of both CTAs have drained an accumulator
    uint64_t drain;
    uint64_t part_full[kPartSteps]; // pieces of partial tiles have been copied into the (idle) operand ring
    uint32_t tmem_base;
    uint32_t abort;
    uint32_t epi_leave[2];          // the epilogue warps' common answer to "has somebody given up?"
    uint32_t seg_open;              // pieces whose first ring entry the TMA producer has found free
};
static_assert(sizeof(Barriers) <= kSmemBarriers, "barrier block");

// fields of the forward row word written by the prologue: bits 0-6 row offset inside the tile, 7-8 class
// (0, 1, 2 = 1, 2, 4 bits; 3 = row past N, to be zero-filled), 9-31 stored position
__device__ __forceinline__ int info_row(uint32_t w) { return (int)(w & 127u); }
__device__ __forceinline__ int info_class(uint32_t w) { return (int)((w >> 7) & 3u); }
__device__ __forceinline__ int info_pos(uint32_t w) { return (int)(w >> 9); }

// ---- dequantisation of one 64-element block to 64 bf16 (one 128-byte operand row) -----------------
// What a lane holds of its row: the packed codes of a block (8, 16 or 32 bytes), the block's absmax, the row's levels.
struct Block {
    uint32_t w[8];
    float a;
    float y[16];
};

__device__ __forceinline__ void load_codes(Block& blk, const uint8_t* p, const float* absmax, int cls) {
    if (cls == 0) {
        const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));
        blk.w[0] = t.x; blk.w[1] = t.y;
    } else if (cls < 3) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(p));
        blk.w[0] = t.x; blk.w[1] = t.y; blk.w[2] = t.z; blk.w[3] = t.w;
        if (cls == 2) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(p) + 1);
            blk.w[4] = u.x; blk.w[5] = u.y; blk.w[6] = u.z; blk.w[7] = u.w;
        }
    }
    if (cls < 3) blk.a = __ldg(absmax);
}
__device__ __forceinline__ void load_levels(Block& blk, const float* row, int cls) {
    if (cls == 0) {
        const float2 f = __ldg(reinterpret_cast<const float2*>(row));
        blk.y[0] = f.x; blk.y[1] = f.y;
    } else if (cls < 3) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i > 0 && cls != 2) break;
            const float4 f = __ldg(reinterpret_cast<const float4*>(row) + i);
            blk.y[4 * i] = f.x; blk.y[4 * i + 1] = f.y; blk.y[4 * i + 2] = f.z; blk.y[4 * i + 3] = f.w;
        }
    }
}

// The block as one 128-byte row of the swizzled operand tile: chunk t (elements 8t .. 8t+7) goes to 16-byte slot t ^ swz
// (128B swizzle).  Sixteen elements at a time, so that few registers are live.  Rows of two precisions may meet in a warp:
// every lane expands in its own way, but they store together - the stores into shared memory, which the tensor core keeps
// busy, are the dear part (a warp with two precisions that stored in two rounds set the pace of 256-token tiles: 0.74 us a stage
// against 0.52).
__device__ __forceinline__ void store_block(const Block& blk, int cls, uint32_t row_addr, uint32_t swz) {
    Scaled<1> s1;
    Scaled<2> s2;
    Scaled<4> s4;
    if (cls == 0) s1.set(blk.y, blk.a);
    else if (cls == 1) s2.set(blk.y, blk.a);
    else if (cls == 2) s4.set(blk.y, blk.a);
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
        uint32_t o[8];
        if (cls == 0) s1.expand16(blk.w, (int)q, o);
        else if (cls == 1) s2.expand16(blk.w, (int)q, o);
        else if (cls == 2) s4.expand16(blk.w, (int)q, o);
        else {
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = 0u;   // a row past the last one
        }
        __syncwarp();
        ptx::st_shared_v4(row_addr + (((2u * q) ^ swz) << 4), make_uint4(o[0], o[1], o[2], o[3]));
        ptx::st_shared_v4(row_addr + (((2u * q + 1u) ^ swz) << 4), make_uint4(o[4], o[5], o[6], o[7]));
    }
}

}  // namespace

// One piece of work of the persistent schedule: a T tile, a whole weight tile, or a slice of the contraction of a weight tile.
struct Seg {
    bool is_t;     // a LoRA down-projection tile rather than a weight tile
    bool lora;     // the LoRA blocks follow the dequantised ones (they belong to the slice that starts the tile)
    bool part;     // the slice does not start its tile: its fp32 sums go to this cluster's partial-tile slot
    bool pre;      // the slice starts its tile but does not end it: it collects the partial tiles of the clusters that
                   // hold the rest
    int prob;      // which weight of the batch
    int rt, mt;    // row tile, token tile
    int m0;        // the token tile's first token
    int nh;        // halves of the token tile that hold tokens
    int kb0, kb1;  // contraction blocks [kb0, kb1) of the tile
    int shares;    // > 1: this cluster and its neighbours hold a slice of the tile each, and each of them finishes a share of it
    int tile;      // weight tile index (ranges)
};

// NB: members the kernel's parameters have room for (1: the plain calls; kMaxBatch: the batch calls).  SHARED: with tiles that several clusters
// share (t_split or w_split above one), which long calls have none of: their loops pay for the code (512-token tiles by 1.5 to 2 % in the forward pass).
template <int MODE, int NB, bool SHARED>
__global__ void __launch_bounds__(kGemmThreads, 1)
fused_kernel(const __grid_constant__ KParams<NB> P, const __grid_constant__ KMaps<NB> TM) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    constexpr int CL = kCluster;
    constexpr uint32_t SW = kSlotsW, SX = kSlotsX;
    unsigned char* x_ring = smem_raw;                       // token entries, then weight slots (1024-byte aligned for the swizzle)
    unsigned char* w_ring = smem_raw + SX * kSmemSlot;
    Barriers* bars = reinterpret_cast<Barriers*>(smem_raw + kSmemRing);
    volatile uint32_t* abort_flag = &bars->abort;
    const uint64_t wait_ns = P.wait_ns;                // limit of every wait below (lowra_set_wait_limit; 1 s by default)
    if ((ptx::smem_u32(smem_raw) & 1023u) != 0u) {    // never seen; without it the operand descriptors would be wrong
        if (threadIdx.x == 0) atomicExch(P.status, (uint32_t)LOWRA_ERR_CUDA);
        return;
    }

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (the same in all lanes, for the compiler too)
    const uint32_t crank = blockIdx.x % (unsigned)CL; // rank in the cluster.  0: issues the MMAs of the pair and holds the barriers they wait for
    const int cid = (int)blockIdx.x / CL, NC = (int)gridDim.x / CL;   // this cluster, clusters in the grid
    const int super_t = P.super_total;                      // token tiles, all members one after the other
    const int n_t_tiles = MODE != kModeDense ? super_t : 0;   // all members' T tiles come first
    const int tile_t = P.halves * kHalfT;                   // tokens per tile
    // token tile gst of the call -> member and tile inside the member
    auto member_of = [&](int gst, Seg& t) {
        t.prob = 0;
        if (NB > 1) {
#pragma unroll
            for (int i = 1; i < NB; ++i)
                if (i < P.count && gst >= P.mem[i].st0) t.prob = i;
        }
        t.mt = gst - P.mem[t.prob].st0;
        t.m0 = t.mt * tile_t;
        t.nh = P.halves == 2 && P.mem[t.prob].M - t.m0 > kHalfT ? 2 : 1;
    };
    const int LB = P.lora_blocks;
    const int B = P.main_blocks + LB;                       // contraction blocks of a weight tile
    // Schedule.  The pieces of work are numbered g = 0, 1, ...: first the T tiles, then the weight tiles; cluster c
    // takes g = c, c + NC, c + 2 NC, ... ("rows" of NC pieces; the clusters then sweep the contraction in step and
    // share the token operand in time).  Whole tiles only: all rows, the last one partly empty.  With ranges (sk): only the
    // T tiles and the weight tiles before sk_first; the contraction blocks of the remaining weight tiles, laid end to end
    // (a tile's LoRA blocks first: they are worked on last, by the slice that starts the tile), are cut into consecutive
    // ranges of equal length, less what the T tile of a cluster costs, so a range starts and ends anywhere inside a tile.
    // A slice that does not start its tile leaves its fp32 sums in the cluster's partial-tile slot; the cluster
    // whose range starts the tile adds them in its epilogue, in a fixed order.  That piece is always the cluster's last, a slice
    // for somebody else always the first of its range, so collecting rarely waits.
    const bool sk = MODE != kModeDense && P.sk != 0;
    // Short calls: the T tiles are what everybody would wait for, so every one of them is shared as well (t_split > 1), by
    // the first clusters, and the weight tiles belong to the others - in ranges, or each shared by w_split of them.
    const int t_cl = SHARED && P.t_split > 1 ? n_t_tiles * P.t_split : 0;
    const int n_whole = sk ? n_t_tiles + P.sk_first : n_t_tiles + P.tiles_r * super_t;   // pieces dealt round-robin
    const int w_whole = t_cl > 0 ? (cid < t_cl ? 1 : 0) : n_whole > cid ? (n_whole - cid + NC - 1) / NC : 0;   // this cluster's
    auto sk_lo = [&](int c) -> int {   // where cluster c's range starts (the launcher keeps the products below 2^31)
        if (c < P.sk_c0) return 0;
        int x = (int)((uint32_t)P.sk_num * (uint32_t)(c - P.sk_c0) / (uint32_t)(NC - P.sk_c0)) - min(c, n_t_tiles) * P.sk_extra;
        const int in_tile = x % B;
        return in_tile < LB ? x - in_tile : x;      // never between two LoRA blocks
    };
    const int lo = sk ? sk_lo(cid) : 0, hi = sk ? sk_lo(cid + 1) : 0;
    const int tile0 = sk ? lo / B : 0;
    const int n_wsegs = (sk && hi > lo) ? (hi - tile0 * B + B - 1) / B : 0;
    const int n_segs = w_whole + n_wsegs;
    auto seg_at = [&](int i) {
        Seg t;
        t.part = t.pre = false;
        t.tile = 0;
        t.shares = 1;
        if (i < w_whole) {
            const int g = cid + i * NC;
            t.kb0 = 0; t.kb1 = P.main_blocks;
            if (t_cl > 0) {
                const int slice = cid % P.t_split;
                member_of(cid / P.t_split, t);
                t.is_t = true; t.lora = false; t.rt = 0;
                t.kb0 = P.main_blocks * slice / P.t_split; t.kb1 = P.main_blocks * (slice + 1) / P.t_split;
                t.shares = P.t_split;
            } else if (g < n_t_tiles) {
                member_of(g, t);
                t.is_t = true; t.lora = false; t.rt = 0;
            } else {
                const int idx = g - n_t_tiles;
                const int gst = idx / P.tiles_r;
                member_of(gst, t);
                t.is_t = false; t.lora = true; t.rt = idx - gst * P.tiles_r;
            }
        } else {
            const int k = i - w_whole;
            t.tile = tile0 + k;                             // counted from the first tile of the ranges
            const int first = t.tile * B;
            const int p0 = (k == 0) ? lo - first : 0, p1 = min(hi - first, B);   // positions: LoRA blocks, then main blocks
            t.kb0 = max(p0 - LB, 0);
            t.kb1 = max(p1 - LB, 0);
            const int idx = P.sk_first + t.tile;
            const int gst = idx / P.tiles_r;
            member_of(gst, t);
            t.is_t = false; t.rt = idx - gst * P.tiles_r;
            t.lora = p0 == 0;
            if (SHARED && P.w_split > 1) {
                t.shares = P.w_split;
            } else {
                t.part = p0 > 0;
                t.pre = p0 == 0 && p1 < B;
            }
        }
        return t;
    };
    // the clusters cid + 1 .. c_end - 1 hold the rest of the tile that this cluster's last piece starts
    auto contributors_end = [&](const Seg& t) {
        const int tile_end = (t.tile + 1) * B;
        int c_end = cid + 1;
        while (c_end < NC && sk_lo(c_end) < tile_end) ++c_end;
        return c_end;
    };
    // Pieces of a shared tile, 32 columns of a weight tile, 16 of a T tile: cluster k of S finishes those numbered k, k + S, ...; so the first
    // t_finishers clusters of a shared T tile have some, and raise a flag each.
    auto t_finishers = [&](const Seg& t) { return SHARED && P.t_split > 1 ? min(P.t_split, t.nh * (P.rp / 16)) : 1; };
    auto t_flags_of = [&](const Seg& t) { return P.mem[t.prob].flags + (t.mt * CL + (int)crank) * (SHARED && P.t_split > 1 ? kTFlags : 1); };
    // How many stages, from stage st of a piece's n, are worked on half by half before the next ones: see kSkew.
    auto run_of = [&](const Seg& t, int st, int n) { return (t.nh == 2 && (st == 0 || n - st <= kSkew)) ? min(kSkew, n - st) : 1; };

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < SX; ++s) {
            ptx::mbar_init(&bars->full_x[s], 1);
            ptx::mbar_init(&bars->empty_x[s], 1);
        }
        for (uint32_t s = 0; s < SW; ++s) {
            ptx::mbar_init(&bars->full_w[s], CL * 4);      // the four warps of either CTA that share a stage
            ptx::mbar_init(&bars->empty_w[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(&bars->tmem_full[a], 1);
            ptx::mbar_init(&bars->tmem_empty[a], CL * kEpilogueWarps);
        }
        ptx::mbar_init(&bars->drain, 1);
        for (int a = 0; a < kPartSteps; ++a) ptx::mbar_init(&bars->part_full[a], 1);
        bars->abort = 0u;
        bars->seg_open = 0u;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&TM.m[0].tmB);
        if (P.lora_blocks > 0) { ptx::prefetch_tensormap(&TM.m[0].tmT); ptx::prefetch_tensormap(&TM.m[0].tmFt); }
        if (P.lora_blocks > 0 || MODE == kModeDense) ptx::prefetch_tensormap(&TM.m[0].tmFl);
    }
    if (warp == 1) ptx::tmem_alloc_pair(&bars->tmem_base, kTmemCols);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();   // the peer's barriers exist before anybody touches them
    ptx::tc_fence_after();
    // Everything above overlapped the kernel before this one (programmatic dependent launch); what follows reads what
    // that kernel wrote (row deal, cleared flags and status word).
    if (MODE != kModeDense) pdl_enter();
    const uint32_t tmem_base = bars->tmem_base;
    // This call's number on the workspace: the value that means "up" in the flags (T ready, partial tile ready).
    uint32_t want = 1u;
    if (MODE != kModeDense) {
        want = *reinterpret_cast<const volatile uint32_t*>(P.epoch) + 1u;
        if (want == 0u) want = 1u;   // only on a workspace that was never initialised (its flags are cleared per call)
    }

    bool failed = false;

    if (warp == 0) {
        // ================================================================== TMA producer (of either CTA)
        // The whole warp walks through the loops, one lane issues (see the MMA warp).
        const bool leader = ptx::elect_one();
        uint32_t e = 0, ph = 0;                     // ring entry, and the parity of its use
        uint32_t it = 0;                            // running stage number: its weight slot is it % SW
        const uint32_t full0 = ptx::map_to_cta(ptx::smem_u32(&bars->full_x[0]), 0u);
        bool free_x = false;                        // the next entry has been seen free
        for (int i = 0; i < n_segs && !failed; ++i) {
            const Seg t = seg_at(i);
            const int r0 = t.rt * kPairR + (int)crank * kTileR;             // this CTA's operand rows
            const int m0 = t.m0 + (int)crank * 128;                         // and tokens (of the first half)
            const MemberMaps& tm = TM.m[t.prob];
            const int n_main = t.kb1 - t.kb0, n = n_main + (t.lora && MODE != kModeDense ? LB : 0);
            const bool w_main = t.is_t || MODE == kModeDense;               // main stages' weight operand comes by TMA as well
            bool first = true, t_ready = false;
            for (int st = 0; st < n && !failed;) {
                const int run = run_of(t, st, n);
                for (int h = 0; h < t.nh && !failed; ++h) {
                    const int m = m0 + h * kHalfT;
                    for (int u = st; u < st + run; ++u) {
                        const bool lora = u >= n_main;
                        const bool w = h == 0 && (lora || w_main);
                        if (lora && !t_ready) {
                            // T of these tokens is written by the CTAs of the same rank in other clusters: wait for their
                            // flags, then make those generic-proxy writes visible to the TMA (async proxy) reads below
                            const int n_flags = t_finishers(t);
                            const bool up = n_flags > 1 ? ptx::flags_wait(t_flags_of(t), n_flags, want, abort_flag, wait_ns)
                                                        : ptx::flag_wait(t_flags_of(t), want, abort_flag, wait_ns);
                            if (!__all_sync(0xffffffffu, up)) { failed = true; break; }
                            ptx::fence_proxy_async_all();
                            t_ready = true;
                        }
                        if (!free_x && !ptx::mbar_wait_lanes(&bars->empty_x[e], ph ^ 1u, abort_flag, wait_ns)) { failed = true; break; }
                        const uint32_t here = e;
                        if (++e == SX) { e = 0; ph ^= 1u; }
                        free_x = __all_sync(0xffffffffu, ptx::mbar_test_wait(&bars->empty_x[e], ph ^ 1u));   // (asked for ahead of its use)
                        const uint32_t bar = full0 + here * 8u;
                        unsigned char* x_s = x_ring + here * kSmemSlot;
                        const int c0 = (lora ? u - n_main : t.kb0 + u) * kTileC;
                        // the bytes of both CTAs are announced by rank 0, whose barrier counts them
                        if (!w) {
                            if (leader) {
                                if (crank == 0u) ptx::mbar_arrive_expect_tx(&bars->full_x[here], kSmemSlot * (uint32_t)CL);
                                ptx::tma_load_2d_pair(x_s, lora ? &tm.tmT : &tm.tmB, c0, m, bar);
                            }
                        } else {
                            // a parity wait tells a use of the slot from the one before only; the ring entry just found free
                            // says that the MMAs are no more than a ring's length behind
                            const uint32_t ws = (it + (uint32_t)(u - st)) % SW, use = (it + (uint32_t)(u - st)) / SW;
                            if (!ptx::mbar_wait_lanes(&bars->empty_w[ws], (use & 1u) ^ 1u, abort_flag, wait_ns)) { failed = true; break; }
                            unsigned char* w_s = w_ring + ws * kSmemSlot;
                            if (leader) {
                                if (crank == 0u) ptx::mbar_arrive_expect_tx(&bars->full_x[here], (kSmemSlot + (t.is_t ? 8192u : kSmemSlot)) * (uint32_t)CL);
                                if (MODE == kModeDense) {
                                    ptx::tma_load_2d_pair(w_s, &tm.tmFl, c0, r0, bar);
                                } else if (t.is_t) {
                                    // this CTA's 64 ranks (zeros past the rank): forward 64 features x 64 ranks from A [K, r],
                                    // backward 64 ranks x 64 channels from B [r, N]
                                    if (MODE == kModeForward) ptx::tma_load_2d_pair(w_s, &tm.tmFt, (int)crank * 64, c0, bar);
                                    else ptx::tma_load_2d_pair(w_s, &tm.tmFt, c0, (int)crank * 64, bar);
                                } else if (MODE == kModeForward) {   // channels x ranks from B [r, N]: two 64-channel boxes
                                    ptx::tma_load_2d_pair(w_s, &tm.tmFl, r0, c0, bar);
                                    ptx::tma_load_2d_pair(w_s + 8192, &tm.tmFl, r0 + 64, c0, bar);
                                } else {                             // features x ranks from A [K, r], K-major: one 64 x 128 box
                                    ptx::tma_load_2d_pair(w_s, &tm.tmFl, c0, r0, bar);
                                }
                                ptx::tma_load_2d_pair(x_s, lora ? &tm.tmT : &tm.tmB, c0, m, bar);
                            }
                        }
                        if (first) {
                            if (leader) *reinterpret_cast<volatile uint32_t*>(&bars->seg_open) = (uint32_t)i + 1u;
                            first = false;
                        }
                        __syncwarp();
                    }
                }
                st += run;
                it += (uint32_t)run;
            }
        }
        if (failed) bars->abort = 1u;
    } else if (warp == 1) {
        // ================================================================== MMA issuer (of the pair: rank 0)
        if (crank == 0u) {
            // This warp is the pacemaker of the pair, its instructions one dependent chain.  All its lanes walk through the
            // loops together, so that ring positions, descriptors and conditions are the warp's (uniform registers, which the
            // MMA instruction wants its operands in), and one lane issues.  With a single lane walking, an entry's four MMAs
            // cost 1060 - 1240 cycles of moves and branches against the tensor core's 790.  A barrier probe takes a hundred
            // cycles and more to answer, ready or not: the barriers of the next entry and the next stage are probed
            // (non-blocking) before the MMAs of an entry are issued, so the answers are back by the time they are needed.
            const bool leader = ptx::elect_one();
            uint32_t e = 0, ph = 0;          // ring entry, and the parity of its use
            uint32_t ws0 = 0;                // weight slot of the run's first stage
            uint32_t phw = 0;                // bit s: parity of the next use of weight slot s by the dequant warps
            uint32_t hc = 0;                 // accumulators handed out: they take turns
            bool ready_x = false, ready_w = false;
            const uint64_t adesc0 = ptx::umma_desc_k_sw128(ptx::smem_u32(x_ring));
            const uint64_t wk0 = ptx::umma_desc_k_sw128(ptx::smem_u32(w_ring)), wmn0 = ptx::umma_desc_mn_sw128(ptx::smem_u32(w_ring), 8192u);
            for (int i = 0; i < n_segs && !failed; ++i) {
                const Seg t = seg_at(i);
                const int n_main = t.kb1 - t.kb0, n = n_main + (t.lora && MODE != kModeDense ? LB : 0);
                const int n_deq = (t.is_t || MODE == kModeDense) ? 0 : n_main;        // stages whose weights are dequantised here
                const uint32_t idesc = t.is_t ? kIdescT : kIdesc;
                for (int st = 0; st < n && !failed;) {
                    const int run = run_of(t, st, n);
                    for (int h = 0; h < t.nh && !failed; ++h) {
                        const uint32_t acc = (hc + (uint32_t)h) & 1u;
                        const uint32_t d_tmem = tmem_base + acc * (uint32_t)kPairR;
                        if (st == 0) {   // the epilogue warps have drained the accumulator's last tile
                            if (!ptx::mbar_wait_lanes(&bars->tmem_empty[acc], (((hc + (uint32_t)h) >> 1) & 1u) ^ 1u, abort_flag, wait_ns)) { failed = true; break; }
                        }
                        uint32_t ws = ws0;
                        for (int u = st; u < st + run; ++u) {
                            const bool weights = u < n_deq;
                            if (weights && h == 0) {
                                if (!ready_w && !ptx::mbar_wait_lanes(&bars->full_w[ws], (phw >> ws) & 1u, abort_flag, wait_ns)) { failed = true; break; }
                                phw ^= 1u << ws;
                            }
                            if (!ready_x && !ptx::mbar_wait_lanes(&bars->full_x[e], ph, abort_flag, wait_ns)) { failed = true; break; }
                            ptx::tc_fence_after();
                            const uint32_t here = e, ws_next = ws + 1u == SW ? 0u : ws + 1u;
                            if (++e == SX) { e = 0; ph ^= 1u; }
                            ready_x = __all_sync(0xffffffffu, ptx::mbar_test_wait(&bars->full_x[e], ph));
                            if (MODE != kModeDense && h == 0) ready_w = __all_sync(0xffffffffu, ptx::mbar_test_wait(&bars->full_w[ws_next], (phw >> ws_next) & 1u));
                            // MN-major weight tiles (a contraction index is a 128-byte row of 64 operand rows): forward - the
                            // factor tiles, fetched from A [K, r] (T tiles) and B [r, N] (LoRA blocks); backward - the
                            // dequantised weights.  16 contraction indices are 32 bytes further in a K-major tile, 2 KB in
                            // an MN-major one.
                            const bool mn = MODE != kModeDense && (MODE == kModeForward ? !weights : weights);
                            const uint64_t adesc = adesc0 + here * (kSmemSlot >> 4);
                            const uint64_t bdesc = (mn ? wmn0 : wk0) + ws * (kSmemSlot >> 4);
                            const uint32_t bstep = mn ? 128u : 2u, id = idesc | (mn ? kIdescBmn : 0u);
                            if (leader) {
#pragma unroll
                                for (uint32_t kk = 0; kk < kTileC / 16; ++kk)
                                    ptx::umma_bf16_pair(d_tmem, adesc + 2u * kk, bdesc + bstep * kk, id, (u != 0 || kk != 0) ? 1u : 0u);
                                ptx::umma_commit_pair(&bars->empty_x[here]);
                                if (h + 1 == t.nh) ptx::umma_commit_pair(&bars->empty_w[ws]);
                            }
                            __syncwarp();
                            ws = ws_next;
                        }
                        if (st + run == n && !failed && leader) ptx::umma_commit_pair(&bars->tmem_full[acc]);
                        __syncwarp();
                    }
                    st += run;
                    ws0 += (uint32_t)run;
                    if (ws0 >= SW) ws0 -= SW;
                }
                hc += (uint32_t)t.nh;
            }
            if (failed) {
                bars->abort = 1u;
                if (leader) {
                    ptx::umma_commit_pair(&bars->drain);
                    ptx::mbar_wait(&bars->drain, 0u, nullptr, 2000000ull);
                }
                __syncwarp();
            }
        }
    } else if (warp < kFirstProducerWarp) {
        // ================================================================== epilogue
        const int q = warp & 3;                 // TMEM lane quarter this warp may read
        const int ch = (warp - kFirstEpilogueWarp) >> 2;   // and which half of the columns it takes
        constexpr uint32_t kThreads = kEpilogueWarps * 32;
        const int et = (warp - kFirstEpilogueWarp) * 32 + lane;
        const int my_tok = q * 32 + lane;       // this lane's token among the CTA's 128 of a half
        const uint32_t tmem_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t empty0 = ptx::map_to_cta(ptx::smem_u32(&bars->tmem_empty[0]), 0u);
        // The epilogue warps share named barriers, so they must leave together: one thread reads the abort
        // flag (any role may raise it at any time), the others take its answer after the barrier.  Two slots in
        // turn, so that the next question cannot overwrite an answer that a slow warp has not read yet.
        uint32_t agree_turn = 0;
        auto agree_abort = [&]() -> bool {
            if (et == 0) bars->epi_leave[agree_turn & 1u] = *abort_flag;
            ptx::named_barrier_sync(1, kThreads);
            const bool leave = *reinterpret_cast<volatile uint32_t*>(&bars->epi_leave[agree_turn & 1u]) != 0u;
            ++agree_turn;
            return leave;
        };
        auto release = [&](uint32_t acc) {      // the accumulator has been read (one arrival per warp and CTA)
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (crank == 0u) ptx::mbar_arrive(&bars->tmem_empty[acc]);
                else ptx::mbar_arrive_cluster(empty0 + acc * 8u);
            }
        };
        uint32_t hc = 0;
        for (int i = 0; i < n_segs && !failed; ++i) {
            const Seg t = seg_at(i);
            const int r0 = t.rt * kPairR, M = P.mem[t.prob].M;
            const int cols = t.is_t ? P.rp : min(kPairR, P.R - r0);   // rows of the tile that exist
            // the columns c0, c0 + 32, ... that this warp takes: half of the tile's; a T tile has few
            const int c_first = t.is_t ? ch * 32 : ch * 128, c_step = t.is_t ? 64 : 32, c_last = t.is_t ? cols : min(cols, ch * 128 + 128);
            // Cluster c's place.  Cluster 0 has partial tiles only where it shares a T tile; they lie in cluster 1's place, behind those of its T tile.
            auto part_of = [&](int c) {
                return P.sk_part + ((size_t)(SHARED && c == 0 ? 1 : c) * CL + crank) * kSkHalfFloats + (SHARED && c == 0 ? kRankCols * 128 : 0);
            };
            float* const part = part_of(cid) + my_tok;
            // 32 rows of one token: rounded and stored
            auto put = [&](uint16_t* dst, int left, uint32_t (&v)[32]) {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
                if (P.out_align == 32 && left >= 32) {
                    ptx::st_global_v8(dst, v);
                    ptx::st_global_v8(dst + 16, v + 8);
                } else if (P.out_align >= 16) {                 // rows are a multiple of 8
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (8 * j < left) *reinterpret_cast<uint4*>(dst + 8 * j) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < left) dst[j] = (uint16_t)(v[j >> 1] >> (16 * (j & 1)));
                }
            };
            // publish this CTA's tokens of T, resp. its half of the cluster's partial tile: the writers meet, and one thread's
            // release covers what all of them have written
            auto raise = [&](uint32_t* flag, bool withheld) {
                ptx::named_barrier_sync(1, kThreads);
                if (et == 0) {
                    ptx::fence_proxy_async_all();
                    if (!withheld) ptx::flag_release(flag, want);
                }
            };
            const bool drop = P.diag_drop_t_flags != 0;     // (diagnostic: the waits for T run out)
            // the first ranks of one token of T among v (16 or 32), scaled by s
            auto put_t = [&](int tok, int c0, int ranks, uint32_t (&v)[32]) {
                uint16_t* dst = P.mem[t.prob].T + (size_t)tok * P.rp + c0;
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = pack_bf16x2(P.s * __uint_as_float(v[2 * j]), P.s * __uint_as_float(v[2 * j + 1]));
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (8 * j < ranks) *reinterpret_cast<uint4*>(dst + 8 * j) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            };
            if (SHARED && t.shares > 1) {
                // Every cluster of a few consecutive ones has a slice of this tile, and no other piece.  Either CTA's part of the tile is
                // pieces of 32 columns (a T tile: 16) x 128 tokens; cluster k of S finishes those numbered k, k + S, ...: the others' sums of them
                // come through the scratch and the operand ring, idle by now, and are added to its own in the order of the slices.
                // What bounds it: two trips through L2 with a flag (3 us) and the SM's L2 port; with S = 4 a CTA writes 96 KB and reads 96 for every
                // 256 tokens, where the cluster of the first slice alone read 384 and the others wrote 128.  (4096 x 4096 at 128 tokens, S = 4 and T between
                // seven: 28.7 -> 26.0 us.)
                const int S = t.shares, k = t.is_t ? cid % S : (cid - P.sk_c0) % S, first = cid - k;
                const int width = t.is_t ? 16 : 32, per_half = (cols + width - 1) / width, pieces = t.nh * per_half;
                for (int h = 0; h < t.nh; ++h) {
                    const uint32_t acc = (hc + (uint32_t)h) & 1u;
                    if (!ptx::mbar_wait_warp(&bars->tmem_full[acc], ((hc + (uint32_t)h) >> 1) & 1u, abort_flag, wait_ns)) bars->abort = 1u;
                    if (agree_abort()) { failed = true; break; }
                    ptx::tc_fence_after();
                    if (t.m0 + h * kHalfT + (int)crank * 128 + my_tok - lane >= M) continue;      // (nobody in this warp has a token)
#pragma unroll 1
                    for (int c0 = c_first; c0 < c_last; c0 += c_step) {
                        const int u = h * per_half + c0 / width;
                        const bool lower = u % S != k, upper = (t.is_t ? u + 1 : u) % S != k;      // sixteen columns each
                        if (!lower && !upper) continue;
                        uint32_t v[32];
                        ptx::tmem_ld_32x32(tmem_lane + acc * (uint32_t)kPairR + (uint32_t)c0, v);
                        ptx::tmem_ld_wait();
                        float* to = part + (size_t)h * kSkAllFloats + (size_t)c0 * 128;
                        if (lower) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) __stcg(to + j * 128, __uint_as_float(v[j]));
                        }
                        if (upper) {
#pragma unroll
                            for (int j = 16; j < 32; ++j) __stcg(to + j * 128, __uint_as_float(v[j]));
                        }
                    }
                }
                if (failed) break;
                raise(P.sk_flags + cid * CL + (int)crank, false);
                const int mine = k < pieces ? (pieces - k + S - 1) / S : 0;
                if (t.m0 + (int)crank * 128 < M && mine > 0) {            // (a CTA without tokens has nothing to finish)
                    if (lane < S && !ptx::flag_wait(P.sk_flags + (first + lane) * CL + (int)crank, want, abort_flag, wait_ns)) bars->abort = 1u;
                    if (agree_abort()) { failed = true; break; }
                    // a step: two pieces, one for either warp of a lane quarter, from every other cluster
                    const int steps = (mine + 1) / 2, ahead = min(kPartSlots / (2 * (S - 1)), kPartSteps);
                    auto fetch = [&](int st) {      // one thread
                        if (st >= steps) return;
                        uint64_t* bar = &bars->part_full[st % kPartSteps];
                        const int wide = min(2, mine - 2 * st);
                        ptx::mbar_arrive_expect_tx(bar, (uint32_t)(wide * (S - 1) * width) * 512u);
                        for (int w = 0; w < wide; ++w) {
                            const int u = k + (2 * st + w) * S, h = u / per_half, c0 = (u - h * per_half) * width;
                            uint32_t to = ptx::smem_u32(x_ring) + (uint32_t)(((st % ahead) * 2 + w) * (S - 1)) * kSmemSlot;
                            for (int c = 0; c < S; ++c) {
                                if (c == k) continue;
                                ptx::bulk_copy_g2s(to, part_of(first + c) + (size_t)h * kSkAllFloats + (size_t)c0 * 128, (uint32_t)width * 512u, bar);
                                to += kSmemSlot;
                            }
                        }
                    };
                    if (et < 32) {                  // (as for the other cut tiles, below)
                        ptx::fence_proxy_async_all();
                        __syncwarp();
                        if (et == 0)
                            for (int st = 0; st < ahead; ++st) fetch(st);
                    }
                    for (int st = 0; st < steps && !failed; ++st) {
                        if (!ptx::mbar_wait_warp(&bars->part_full[st % kPartSteps], (uint32_t)(st / kPartSteps) & 1u, abort_flag, wait_ns)) bars->abort = 1u;
                        if (2 * st + ch < mine) {
                            const int u = k + (2 * st + ch) * S, h = u / per_half, c0 = (u - h * per_half) * width;
                            const int tok = t.m0 + h * kHalfT + (int)crank * 128 + my_tok;
                            const float* ring = reinterpret_cast<const float*>(x_ring) + (size_t)(((st % ahead) * 2 + ch) * (S - 1)) * (kSmemSlot / 4) + my_tok;
                            uint32_t v[32];
                            ptx::tmem_ld_32x32(tmem_lane + ((hc + (uint32_t)h) & 1u) * (uint32_t)kPairR + (uint32_t)c0, v);
                            ptx::tmem_ld_wait();
                            for (int c = 1; c < S; ++c, ring += kSmemSlot / 4) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + ring[j * 128]);
                                if (width == 32) {
#pragma unroll
                                    for (int j = 16; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + ring[j * 128]);
                                }
                            }
                            if (tok < M) {
                                if (t.is_t) put_t(tok, c0, 16, v);
                                else put(P.mem[t.prob].out + (size_t)tok * P.ld_out + r0 + c0, cols - c0, v);
                            }
                        }
                        if (st + ahead < steps) {
                            if (agree_abort()) { failed = true; break; }     // everybody has read the step's pieces: their place is filled again
                            if (et == 0) fetch(st + ahead);
                        }
                    }
                    if (!failed && agree_abort()) failed = true;
                }
                if (t.is_t && !failed && mine > 0) raise(t_flags_of(t) + k, drop);
                break;                          // (the only piece)
            }
            if (t.pre) {
                // A piece that starts a tile which other clusters finish: their partial tiles are added here.  The piece is
                // this cluster's last one; once its MMAs are complete the operand ring is idle, and the partial tiles are
                // streamed through it, several steps ahead of the warps that add them to the accumulator's values in a fixed
                // order.  (What bounds it: the SM's L2 port, 128 KB per half and contributor at 50 - 60 GB/s.  The warps meet only
                // where a place of the ring is filled again: 4096 x 4096 at 512 tokens 43.2 -> 42.0 us against meeting at every step.)
                const int c_end = contributors_end(t), nc = c_end - cid - 1;
                for (int h = 0; h < t.nh; ++h)
                    if (!ptx::mbar_wait_warp(&bars->tmem_full[(hc + (uint32_t)h) & 1u], ((hc + (uint32_t)h) >> 1) & 1u, abort_flag, wait_ns)) bars->abort = 1u;
                if (lane < nc && !ptx::flag_wait(P.sk_flags + (cid + 1 + lane) * CL + (int)crank, want, abort_flag, wait_ns)) bars->abort = 1u;
                if (agree_abort()) { failed = true; break; }
                ptx::tc_fence_after();
                const int steps = 4 * t.nh, pieces = 2 * nc, ahead = min(kPartSlots / pieces, kPartSteps);
                auto fetch = [&](int s) {       // one thread
                    if (s >= steps) return;
                    uint64_t* bar = &bars->part_full[s % kPartSteps];
                    const int h = s / 4, c0 = (s & 3) * 32;
                    ptx::mbar_arrive_expect_tx(bar, (uint32_t)pieces * kSmemSlot);
                    for (int k = 0; k < pieces; ++k) {
                        const float* src = part_of(cid + 1 + k / 2) + (size_t)h * kSkAllFloats + (size_t)((k % 2) * 128 + c0) * 128;
                        ptx::bulk_copy_g2s(ptx::smem_u32(x_ring) + (uint32_t)((s % ahead) * pieces + k) * kSmemSlot, src, kSmemSlot, bar);
                    }
                };
                if (et < 32) {                  // the warp of the thread that copies has looked at every flag
                    // the slices were written with ordinary stores by other SMs and acquired through the flags: make them
                    // visible to the copy engine (async proxy) as well
                    ptx::fence_proxy_async_all();
                    __syncwarp();
                    if (et == 0)
                        for (int s = 0; s < ahead; ++s) fetch(s);
                }
                for (int s = 0; s < steps && !failed; ++s) {
                    const int h = s / 4, c0 = ch * 128 + (s & 3) * 32;
                    const int tok = t.m0 + h * kHalfT + (int)crank * 128 + my_tok;
                    if (!ptx::mbar_wait_warp(&bars->part_full[s % kPartSteps], (uint32_t)(s / kPartSteps) & 1u, abort_flag, wait_ns)) bars->abort = 1u;
                    uint32_t v[32];
                    ptx::tmem_ld_32x32(tmem_lane + ((hc + (uint32_t)h) & 1u) * (uint32_t)kPairR + (uint32_t)c0, v);
                    ptx::tmem_ld_wait();
                    const float* ring = reinterpret_cast<const float*>(x_ring) + (size_t)((s % ahead) * pieces + ch) * (kSmemSlot / 4) + my_tok;
                    for (int c = 0; c < nc; ++c) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + ring[(size_t)(2 * c) * (kSmemSlot / 4) + j * 128]);
                    }
                    if (tok < M && c0 < cols) put(P.mem[t.prob].out + (size_t)tok * P.ld_out + r0 + c0, cols - c0, v);
                    if (s + ahead < steps) {
                        if (agree_abort()) { failed = true; break; }     // everybody has read the step's pieces: their place is filled again
                        if (et == 0) fetch(s + ahead);
                    }
                }
                if (!failed && agree_abort()) failed = true;
                break;                          // (the last piece; its accumulators are not handed on)
            }
            for (int h = 0; h < t.nh; ++h, ++hc) {
                const uint32_t acc = hc & 1u;
                const uint32_t taddr = tmem_lane + acc * (uint32_t)kPairR;
                const int tok = t.m0 + h * kHalfT + (int)crank * 128 + my_tok;
                const bool any = tok - lane < M;        // somebody in this warp has a token
                if (!ptx::mbar_wait_warp(&bars->tmem_full[acc], (hc >> 1) & 1u, abort_flag, wait_ns)) bars->abort = 1u;
                if (agree_abort()) { failed = true; break; }
                ptx::tc_fence_after();
#pragma unroll 1
                for (int c0 = c_first; c0 < c_last && any; c0 += c_step) {
                    uint32_t v[32];
                    ptx::tmem_ld_32x32(taddr + (uint32_t)c0, v);
                    ptx::tmem_ld_wait();
                    if (t.part) {
                        // fp32 sums of a slice: [row][token], so that a warp writes 128 consecutive bytes
#pragma unroll
                        for (int j = 0; j < 32; ++j) __stcg(part + (size_t)h * kSkAllFloats + (size_t)(c0 + j) * 128, __uint_as_float(v[j]));
                    } else if (tok < M) {
                        if (t.is_t) put_t(tok, c0, 32, v);
                        else put(P.mem[t.prob].out + (size_t)tok * P.ld_out + r0 + c0, cols - c0, v);
                    }
                }
                release(acc);
            }
            if (failed) break;
            if (t.part) raise(P.sk_flags + cid * CL + (int)crank, false);
            else if (t.is_t) raise(t_flags_of(t), drop);
        }
    } else if (MODE != kModeDense) {
        // ================================================================== dequant producers
        // The prologue has dealt the rows to these warps (see gemm_prep.cu).  Each thread dequantises one 64-element absmax
        // block per visit of a stage; the groups of four warps take the dequantised stages in turn.  What the next visit needs
        // is asked for right after this one's arrival, so that its latency passes while the other groups have their turn
        // (and the proxy fence, which waits for loads under way, finds none).
        // Warps with the same q carry alike loads (the forward deal gives the last 32 rows, those of most bits, to q = 3); a step on
        // from group to group puts them on the SM's four schedulers (warp mod 4), one each.  All on one scheduler they set the pace:
        // 5120 x 5120 at 60/35/5, 600 tokens, forward 70.9 us against 58.5; 13824 x 5120, 130 tokens 70.2 against 57.8.
        const int pw = warp - kFirstProducerWarp;                // 0 .. kProducerWarps - 1
        const int grp = pw >> 2, q = (pw + grp) & 3;
        constexpr int G = kProducerGroups;
        const uint32_t full0 = ptx::map_to_cta(ptx::smem_u32(&bars->full_w[0]), 0u);
        uint32_t it0 = 0;                                        // running stage number at the start of the piece
        uint32_t wi0 = 0;                                        // dequantised stages before the piece
        // Waits until the weight slot of stage `it` is free.  A parity wait tells a use of the slot from the one before it
        // only; a warp that fills every G-th stage is never further off.  T tiles and LoRA blocks run on without these
        // warps, so at the start of a piece a warp first waits until the TMA producer, which passes every stage, has found the
        // piece's first ring entry free.
        auto stage_free = [&](uint32_t it) -> bool {
            return ptx::mbar_wait_lanes(&bars->empty_w[it % SW], ((it / SW) & 1u) ^ 1u, abort_flag, wait_ns);
        };
        auto piece_open = [&](int i) -> bool {
            uint32_t ok = 1u;
            if (lane == 0) {
                const uint64_t t0 = ptx::globaltimer_ns();
                while (*reinterpret_cast<volatile uint32_t*>(&bars->seg_open) <= (uint32_t)i) {
                    __nanosleep(200);
                    if (*abort_flag != 0u || ptx::globaltimer_ns() - t0 > wait_ns) { ok = 0u; break; }
                }
            }
            return __shfl_sync(0xffffffffu, ok, 0) != 0u;
        };
        // This warp's rows of the slot are in place: one arrival on the stage's barrier in the CTA that issues the MMAs.
        auto publish = [&](uint32_t s) {
            ptx::fence_proxy_async_smem();   // the tensor core reads the rows
            __syncwarp();
            if (lane == 0) {
                if (crank == 0u) ptx::mbar_arrive(&bars->full_w[s]);
                else ptx::mbar_arrive_cluster(full0 + s * 8u);
            }
        };
        for (int i = 0; i < n_segs && !failed; ++i) {
            const Seg t = seg_at(i);
            const int n_main = t.is_t ? 0 : t.kb1 - t.kb0;
            const int r0 = t.rt * kPairR + (int)crank * kTileR;
            const Member& W = P.mem[t.prob];                    // the weight this piece belongs to
            const uint32_t itb = it0 - (uint32_t)t.kb0;         // running stage number of block kb: itb + kb
            const int kb_first = t.kb0 + (int)(((uint32_t)grp - wi0) & (uint32_t)(G - 1));   // this group's blocks, every G-th
            static_assert((G & (G - 1)) == 0, "the groups are counted with a mask");
            if (kb_first >= t.kb1 || t.is_t) {
                // nothing to dequantise for this warp
            } else if (r0 >= P.R) {
                // this CTA's rows lie past the last one: whatever the slots hold gives columns that nobody stores
                if (!piece_open(i)) { failed = true; bars->abort = 1u; break; }
                for (int kb = kb_first; kb < t.kb1; kb += G) {
                    const uint32_t it = itb + (uint32_t)kb;
                    if (!stage_free(it)) { failed = true; bars->abort = 1u; break; }
                    publish(it % SW);
                }
            } else if (MODE == kModeForward) {
                // ---------------------------------------------------------------- forward
                // The operand tile of a stage is [128 channels][64 input features], K-major: a channel's
                // 64-element absmax block is one 128-byte row.  Warp q of a group holds rows 32 q .. 32 q + 31
                // of the CTA's rows, roughly in precision order (see the deal in gemm_prep.cu).  A thread keeps its
                // channel, and the channel's levels, for the whole tile.
                const uint32_t item = __ldg(W.items + (size_t)(r0 / kTileR) * kItemStride + q * 32 + lane);
                const int cls = info_class(item), row_local = info_row(item);
                Block blk;
                const uint8_t* bits_ptr = W.packed;
                const float* absmax_ptr = W.absmax;
                int bits_stride = 0;  // packed bytes per 64-element block
                if (cls < 3) {
                    const int p = info_pos(item);
                    bits_stride = 8 << cls;
                    bits_ptr = W.packed + packed_row_offset(W.L, cls, p, r0 + row_local);
                    absmax_ptr = W.absmax + (size_t)absmax_row_of(W.L, p, r0 + row_local) * W.L.nb;
                    load_levels(blk, W.maps + (size_t)(r0 + row_local) * kTableStride, cls);
                    load_codes(blk, bits_ptr + (size_t)kb_first * bits_stride, absmax_ptr + kb_first, cls);
                }
                if (!piece_open(i)) { failed = true; bars->abort = 1u; break; }
#pragma unroll 1
                for (int kb = kb_first; kb < t.kb1; kb += G) {
                    const uint32_t it = itb + (uint32_t)kb;
                    if (!stage_free(it)) { failed = true; bars->abort = 1u; break; }
                    const uint32_t s = it % SW;
                    store_block(blk, cls, ptx::smem_u32(w_ring) + s * kSmemSlot + (uint32_t)row_local * 128u, (uint32_t)row_local & 7u);
                    publish(s);
                    const int nb = kb + G;
                    if (cls < 3 && nb < t.kb1) load_codes(blk, bits_ptr + (size_t)nb * bits_stride, absmax_ptr + nb, cls);
                }
            } else {
                // ---------------------------------------------------------------- backward
                // every stage brings 64 new channels (the contraction index); thread = one channel x 64 of
                // the CTA's 128 input features = one absmax block.  Operand tile is MN-major:
                // [feature half][64 channels][64 features], so the block is one 128-byte row.
                // The rows of a group of 64 channels have been dealt to the warps in chunks of 16 (gemm_prep.cu).
                const uint32_t half = (uint32_t)(lane >> 4) & 1u;
                const int k_first = r0 + 64 * (int)half;
                const uint4* rows = reinterpret_cast<const uint4*>(W.items) + (size_t)q * 16 + (lane & 15);   // group g: rows[g * 64]
                Block blk;
                auto fetch = [&](const uint4& rec) {
                    const int cls = (int)((rec.w >> 8) & 3u);
                    if (cls < 3) {
                        load_codes(blk, W.packed + ((size_t)rec.x << 4) + (((size_t)k_first << cls) >> 3), W.absmax + rec.y + (k_first >> 6), cls);
                        load_levels(blk, W.maps + rec.z, cls);
                    }
                };
                uint4 rec = __ldg(rows + (size_t)kb_first * kGroupRecords), next = rec;   // this visit's record, and the next one's
                if (kb_first + G < t.kb1) next = __ldg(rows + (size_t)(kb_first + G) * kGroupRecords);
                fetch(rec);
                if (!piece_open(i)) { failed = true; bars->abort = 1u; break; }
#pragma unroll 1
                for (int kb = kb_first; kb < t.kb1; kb += G) {
                    const uint32_t col = rec.w & 63u;             // channel inside the stage = contraction index of the tile
                    const uint32_t it = itb + (uint32_t)kb;
                    if (!stage_free(it)) { failed = true; bars->abort = 1u; break; }
                    const uint32_t s = it % SW;
                    store_block(blk, (int)((rec.w >> 8) & 3u), ptx::smem_u32(w_ring) + s * kSmemSlot + half * 8192u + col * 128u, col & 7u);
                    publish(s);
                    rec = next;
                    if (kb + G < t.kb1) fetch(rec);
                    if (kb + 2 * G < t.kb1) next = __ldg(rows + (size_t)(kb + 2 * G) * kGroupRecords);
                }
            }
            it0 += (uint32_t)(t.kb1 - t.kb0 + (t.lora ? LB : 0));
            wi0 += (uint32_t)n_main;
        }
    }

    if (failed) {
        atomicExch(P.status, (uint32_t)LOWRA_ERR_TIMEOUT);
        // tell the peer as well, so that the CTAs of the cluster agree below on how they leave
        ptx::st_relaxed_cluster(ptx::map_to_cta(ptx::smem_u32(&bars->abort), crank ^ 1u), 1u);
    }
    // ---------------------------------------------------------------------- teardown
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();   // the peer's copies, arrivals and MMAs no longer touch this CTA
    if (*abort_flag != 0u) {
        // Somebody gave up (the same answer in both CTAs: the flag was exchanged before the barrier).
        // Roles that were not waiting on them may have left bulk copies, TMA loads or MMAs in flight; they need
        // microseconds.  Every role has stopped issuing, so a fixed grace period covers them before shared and
        // tensor memory are given back.
        if (threadIdx.x == 0) {
            const uint64_t t0 = ptx::globaltimer_ns();
            while (ptx::globaltimer_ns() - t0 < kGraceNs) __nanosleep(1000);
        }
        __syncthreads();
        ptx::cluster_sync();
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
    }
    if (MODE != kModeDense && threadIdx.x == 0) {
        // the last CTA to leave records the call's number; every CTA has read the old one long before.  Just before
        // the numbering wraps around, it clears the flags and starts again from zero.
        __threadfence();
        if (atomicAdd(P.exits, 1u) == gridDim.x - 1u) {
            if (want == 0xFFFFFFFFu) {
                for (int i = 0; i < P.n_flags; ++i) P.flags[i] = 0u;
                want = 0u;
            }
            *P.epoch = want;
            *P.exits = 0u;
        }
    }
}

// Chooses the token tiles (256 or 512 tokens) and the schedule of a call - whole tiles, shared ones, or ranges behind so many whole weight
// tiles (see the kernel) - and returns the number of clusters to launch.  What is compared is an estimate of the call's time, in microseconds at full
// clock.  Its figures are a fit to the times of every schedule that 530 calls could take (17 to 8192 tokens, 256 to 13824 channels and features,
// ranks 16 to 128, six mixes of precisions, both directions), by the errors and by what the choice loses against the best one; estimates are within 7 %
// of the times (one standard deviation).  On 190 other calls, each in both directions, the choice is 0.5 % behind the best schedule in the mean and more
// than 5 % behind for 2 % of them.  (With the figures before, from a few shapes: 1.5 %, 10 %; most of it 512-token tiles shared at ranks above 64:
// backward 2672 x 1152, 1437 tokens, rank 128 34.7 us, now 28.4; forward 5016 x 2944, 404 tokens 36.1, now 30.8.)
static int plan_schedule(GemmParams& Q, bool may_cut, int max_clusters, float* estimate = nullptr) {
    const int blocks = Q.main_blocks + Q.lora_blocks;
    struct Choice { float us; int halves, clusters, cut, first, c0, extra, t_split, num, w_split; } best = {};
    best.us = -1.0f;
    auto tiles_of = [&](int halves) {
        int n = 0;
        for (int i = 0; i < Q.count; ++i) n += (Q.mem[i].M + halves * kHalfT - 1) / (halves * kHalfT);
        return n;
    };
    auto offer = [&](const Choice& c) { if (best.us < 0.0f || c.us < best.us) best = c; };
    // every range keeps a sixth of a tile, so that a tile has at most kMaxContributors contributors
    const int sixth = (blocks + kMaxContributors - 2) / (kMaxContributors - 1), shortest = sixth > kMinRange ? sixth : kMinRange;
    for (int halves = Q.wide_only ? 2 : 1; halves <= (Q.M > kHalfT ? 2 : 1); ++halves) {
        const float pace = halves == 1 ? 0.51f : 0.76f;         // a contraction block of a weight tile (256 tokens: the dequantising warps'; 512: the tensor core's)
        auto collect = [&](int nc) { return 4.0f * halves * (0.6f * nc > 1.57f ? 0.6f * nc : 1.57f); };    // four steps per 256 tokens
        const int super_t = tiles_of(halves), n_t = may_cut ? super_t : 0, n_w = Q.tiles_r * super_t, n = n_w + n_t;
        // when T is there: whole tiles, tiles that ts clusters share
        const float t_us = halves == 1 ? 9.4f + 0.44f * Q.main_blocks : 14.4f + 0.62f * Q.main_blocks;
        auto shared_t = [&](int ts) { return 7.0f + 0.43f * Q.main_blocks / ts + halves * (6.2f + 1.7f * (Q.lora_blocks - 1)); };
        auto single_us = [&](float n) { return 8.2f + (halves == 1 ? 0.5f : 0.76f) * n; };                // a cluster's only piece, n blocks
        {   // whole tiles
            const int clusters = n < max_clusters ? n : max_clusters, rows = (n + clusters - 1) / clusters;
            // (a second row of no more pieces than there are T tiles: they go to the clusters that had one of those, and nobody hands accumulators over)
            const float w_us = rows == 1 || (rows == 2 && n - clusters <= n_t) ? single_us(blocks * rows) : 14.9f + pace * blocks * rows;
            offer({(rows == 1 && n_t > 0 && t_us > w_us ? t_us : w_us) - 0.7f * halves, halves, clusters, 0, 0, 0, 0, 1, 0, 1});
        }
        if (!may_cut || halves > Q.part_halves || n_t > max_clusters || blocks < 2 * kMinRange) continue;
        if ((long long)n * blocks * max_clusters >= (1ll << 31)) continue;     // (32-bit arithmetic in the kernel)
        // Fewer pieces than clusters: s clusters share every weight tile, and those left over the T tiles.
        for (int s = 1; s < kMaxContributors && n_w * s + n_t <= max_clusters && blocks / s >= shortest; ++s) {
            int ts = (max_clusters - n_w * s) / n_t;
            if (ts > kMaxContributors) ts = kMaxContributors;
            if (ts > Q.main_blocks / kMinShare) ts = Q.main_blocks / kMinShare;
            if (ts < 2 || Q.main_blocks < 2 * kMinRange) ts = 1;
            if (ts == 1 && s == 1) continue;
            const float t_done = ts == 1 ? t_us : shared_t(ts), w_done = single_us((float)blocks / s);
            const float us = (t_done > w_done ? t_done : w_done) + (s == 1 ? -0.7f * halves : 3.5f + 2.5f * halves);
            // Tiles of 256 tokens between two or three clusters on (almost) all SMs are finished by the first one: the others leave while it works, and the next
            // call's CTAs come in (us, shared against this: forward 5888 x 4352, 168 tokens 32.0 -> 27.8, backward 3224 x 8832, 209 tokens 32.9 -> 28.3).  On
            // fewer SMs the two are alike at two clusters and sharing is ahead from three, by 2 to 15 %; tiles of 512 tokens are always shared (by 5 to 27 %).
            const bool by_first = halves == 1 && s <= 3 && n_t * ts + n_w * s >= 70;
            offer({us, halves, n_t * ts + n_w * s, 1, 0, n_t * ts, 0, ts, n_w * blocks, by_first ? 1 : s});
        }
        // T by clusters of its own, each tile by ts of them, and ranges over all weight tiles for the others: for few channels and many tokens, where one
        // piece in a few is a T tile that the others wait for, and for pieces that come out a little over a row (forward, us, against the
        // choices around: 1024 x 4096, 4096 / 8192 tokens 60 -> 52 / 92 -> 78; 1024 x 11008, 4096 tokens 137 -> 101; 3072 x 3072, 3000 tokens 75 -> 61;
        // 6144 x 2048, 1500 tokens 54 -> 46).  Ranges of less than half a tile gain nothing (2048 x 4096, 600 tokens 30.4 -> 33.7); nor
        // does a choice that is ahead by less than a microsecond or so (1024 x 11008, 6000 tokens 140 -> 152).
        for (int ts = 1; ts <= kMaxContributors && n_t * ts < max_clusters; ++ts) {
            if (ts > 1 && (ts > Q.main_blocks / kMinShare || Q.main_blocks < 2 * kMinRange)) break;
            const int c = max_clusters - n_t * ts;
            const float range = (float)n_w * blocks / c;
            if (range < shortest || 2.0f * range < blocks) continue;      // (longer with every ts)
            const float t_done = ts == 1 ? t_us : shared_t(ts), w_done = 12.1f + pace * range;
            offer({(t_done > w_done ? t_done : w_done) - 1.4f - 0.7f * halves + collect((int)((blocks + range) / range)), halves, max_clusters, 1, 0, n_t * ts, 0, ts, n_w * blocks, 1});
        }
        // Ranges for the last row of pieces, or for the last two.  The clusters' sweeps over the contraction fall out of step
        // inside the ranges, so the part of the token operand that is live there has to stay in L2 (ranges over all tiles of a
        // 90 MB operand: 6.5 times the DRAM reads, and no gain).
        const int rows = n / max_clusters, n_last = n - rows * max_clusters;
        const int t_cost = (int)(blocks * (halves == 1 ? 0.5f / 0.6f : 0.7f / 0.8f));   // a T tile, in blocks of a weight tile: it is paced by its loads
        for (int whole = rows; whole >= 0 && whole >= rows - 1 && n_last > 0 && rows > 0; --whole) {
            const size_t slab = (size_t)halves * kHalfT * (size_t)Q.C * 2u;   // token operand of one token tile
            const int cut_tiles = n - whole * max_clusters;
            if (whole < rows && (size_t)(cut_tiles / Q.tiles_r + 2) * slab > ((size_t)48 << 20)) continue;
            const int first = whole == 0 ? 0 : whole * max_clusters - n_t;
            if (first < 0) continue;
            const long long rest = (long long)(n_w - first) * blocks;
            int extra = whole == 0 ? t_cost : t_cost - blocks;                   // what a cluster with a T tile gets less (negative: more)
            long long num = rest + (long long)n_t * extra;
            if (extra < 0 && num / max_clusters < shortest) { extra = 0; num = rest; }
            if ((extra > 0 ? num / max_clusters - extra : num / max_clusters) < shortest) continue;
            const float range = (float)num / max_clusters;
            const int nc = (int)((blocks + range) / range);                      // contributors of a tile, about
            offer({16.7f + pace * (whole * blocks + range) + collect(nc), halves, max_clusters, 1, first, 0, extra, 1, (int)num, 1});
        }
    }
    Q.halves = best.halves;
    Q.super_total = 0;
    for (int i = 0; i < Q.count; ++i) {
        Q.mem[i].st0 = Q.super_total;
        Q.super_total += (Q.mem[i].M + Q.halves * kHalfT - 1) / (Q.halves * kHalfT);
    }
    Q.sk = best.cut;
    Q.sk_first = best.first;
    Q.sk_c0 = best.c0;
    Q.sk_extra = best.extra;
    Q.sk_num = best.num;
    Q.t_split = best.t_split;
    Q.w_split = best.w_split;
    if (estimate != nullptr) *estimate = best.us;
    return best.clusters;
}

// The estimate for a forward call of `count` members of M tokens each on a whole GPU.
float fused_estimate(int N, int K, int M, int r, int count) {
    GemmParams Q;
    memset(&Q, 0, sizeof(Q));
    float us = 0.0f;
    Q.count = count < kMaxBatch ? count : kMaxBatch;
    for (int i = 0; i < Q.count; ++i) Q.mem[i].M = M;
    Q.M = M;
    Q.C = K;
    Q.main_blocks = (K + kTileC - 1) / kTileC;
    Q.lora_blocks = (r + 63) / 64 * 64 / kTileC;
    Q.tiles_r = (N + kPairR - 1) / kPairR;
    Q.part_halves = 2;   // (tiles may be cut)
    plan_schedule(Q, true, kNumSMs / kCluster, &us);
    return us * (float)((count + kMaxBatch - 1) / kMaxBatch);
}

// The schedule of a call of `count` members on a whole GPU, its clusters returned.
int fused_schedule(bool backward, int N, int K, const int32_t* Ms, int count, int r, int* tile_tokens, int* w_split, int* t_split) {
    GemmParams Q;
    memset(&Q, 0, sizeof(Q));
    Q.count = count;
    for (int i = 0; i < count; ++i) {
        Q.mem[i].M = Ms[i];
        Q.M = Ms[i] > Q.M ? Ms[i] : Q.M;
    }
    Q.C = backward ? N : K;
    Q.main_blocks = (Q.C + kTileC - 1) / kTileC;
    Q.lora_blocks = (r + 63) / 64;
    Q.tiles_r = ((backward ? K : N) + kPairR - 1) / kPairR;
    Q.part_halves = 2;
    const int clusters = plan_schedule(Q, true, kNumSMs / kCluster);
    *tile_tokens = Q.halves * kHalfT;
    *w_split = Q.w_split;
    *t_split = Q.t_split;
    return clusters;
}

// How many clusters can be resident at once, and that the kernel may have its shared memory: once per kernel and device.
template <int MODE, int NB, bool SHARED>
static lowra_status prepare_fused(cudaLaunchConfig_t& cfg, int* max_clusters) {
    constexpr int CL = kCluster;
    static std::mutex mutex;
    static bool configured[kMaxDevices] = {false};
    static int max_clusters_of[kMaxDevices] = {0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LOWRA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mutex);
    if (!configured[dev]) {
        const int sms = device_sm_count();
        if (sms < CL) return LOWRA_ERR_CUDA;
        if (cudaFuncSetAttribute(fused_kernel<MODE, NB, SHARED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kGemmSmemBytes) != cudaSuccess)
            return LOWRA_ERR_CUDA;
        // the persistent schedule needs every cluster of the grid resident (a tile waits for T of another)
        cfg.gridDim = dim3(sms / CL * CL, 1, 1);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fused_kernel<MODE, NB, SHARED>, &cfg) != cudaSuccess || n < 1) return LOWRA_ERR_CUDA;
        max_clusters_of[dev] = n < sms / CL ? n : sms / CL;
        configured[dev] = true;
    }
    *max_clusters = max_clusters_of[dev];
    return LOWRA_OK;
}

template <int MODE, int NB>
static lowra_status launch_mode(const GemmParams& G, const BatchMaps& TM, cudaStream_t stream) {
    constexpr int CL = kCluster;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // start while the prologue kernel (the previous launch in the stream) is still running; the kernel waits for
    // it before it reads anything that kernel writes
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = kGemmSmemBytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = (MODE == kModeDense) ? 1 : 2;
    int max_clusters = 0;
    lowra_status st = prepare_fused<MODE, NB, false>(cfg, &max_clusters);
    if (st != LOWRA_OK) return st;
    if (MODE != kModeDense) {
        int n = 0;
        if ((st = prepare_fused<MODE, NB, MODE != kModeDense>(cfg, &n)) != LOWRA_OK) return st;
        max_clusters = n < max_clusters ? n : max_clusters;
    }
    GemmParams Q = G;
    const int clusters = plan_schedule(Q, MODE != kModeDense, max_clusters);
    if (Q.t_split > 1)      // (at most 36 T tiles then: their flags fit into the header)
        for (int i = 0; i < Q.count; ++i) Q.mem[i].flags = Q.flags + kSharedTFlags + Q.mem[i].st0 * CL * kTFlags;
    cfg.gridDim = dim3((unsigned)(clusters * CL), 1, 1);
    KParams<NB> QP;
    KMaps<NB> QM;
    static_cast<GemmCommon&>(QP) = static_cast<const GemmCommon&>(Q);
    for (int i = 0; i < NB; ++i) { QP.mem[i] = Q.mem[i]; QM.m[i] = TM.m[i]; }
    const bool shared = Q.t_split > 1 || Q.w_split > 1;
    const cudaError_t rc = shared ? cudaLaunchKernelEx(&cfg, fused_kernel<MODE, NB, MODE != kModeDense>, QP, QM)
                                  : cudaLaunchKernelEx(&cfg, fused_kernel<MODE, NB, false>, QP, QM);
    return rc == cudaSuccess ? LOWRA_OK : LOWRA_ERR_CUDA;
}

lowra_status launch_fused(int mode, const GemmParams& G, const BatchMaps& TM, cudaStream_t stream) {
    if (mode == kModeDense) return launch_mode<kModeDense, 1>(G, TM, stream);
    if (mode == kModeForward)
        return G.count == 1 ? launch_mode<kModeForward, 1>(G, TM, stream) : launch_mode<kModeForward, kMaxBatch>(G, TM, stream);
    return G.count == 1 ? launch_mode<kModeBackward, 1>(G, TM, stream) : launch_mode<kModeBackward, kMaxBatch>(G, TM, stream);
}

}  // namespace lowra
