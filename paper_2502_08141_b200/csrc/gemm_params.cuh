// Launch parameters shared by the prologue kernel, the fused tensor-core kernel and their host code.
#pragma once

#include <cuda.h>

#include "lowra_common.cuh"

namespace lowra {

// ---- prologue ------------------------------------------------------------------------------
constexpr int kPrepThreads = 128;
constexpr int kProducerWarps = 16;            // dequant warps of the main kernel
constexpr int kItemStride = 128;              // forward: entries per group of 128 rows in the deal table
constexpr int kGroupRecords = 64;             // backward: row records per group of 64 channels
constexpr int kCluster = 2;                   // CTAs per cluster: the pair that works on one tensor-core tile
constexpr int kMaxGroups64 = 8192;            // backward: at most this many groups of 64 output channels (N <= 524288)

struct PrepParams {
    // deal of the rows to the dequant threads of the main kernel.  Row word = row offset inside its group
    // (bits 0-6) | class (bits 7-8, 3 = row past N) | stored position (bits 9-31), all ones for "no row".
    //   forward (group 128): items[g * kItemStride + i] = i-th row of group g in precision order
    //   backward (group 64): 64 row records of 16 bytes per group, see deal_backward
    RowLayout L;
    const uint8_t* precs;
    const int32_t* inv_perm;
    uint32_t* items;      // forward: row words; backward: 16-byte row records
    int N, group;
    uint32_t* status;     // device status word, cleared (null: left alone)
    uint32_t* exits;      // the fused kernel's count of CTAs that have left, cleared (null: left alone)
    uint32_t* flags;      // [n_flags] "T of this token tile is ready" flags, cleared
    int n_flags;
    int blocks;
};

lowra_status launch_prep(const PrepParams& P, cudaStream_t stream);

// ---- fused kernel --------------------------------------------------------------------------
constexpr int kTileR = 128;       // operand rows (output channels fwd, input features bwd) per CTA ...
constexpr int kPairR = 256;       // ... and per tile: the two CTAs of a cluster form one tensor-core tile
constexpr int kHalfT = 256;       // tokens per MMA (128 in either CTA)
constexpr int kTileT = 512;       // tokens per tile at most: two MMAs' worth share every dequantised weight
constexpr int kTileC = 64;        // contraction elements per pipeline stage (= one absmax block, = 128 bytes of bf16)
// The operand ring: a stage takes one weight slot and an entry for each half of its tokens, 16 KB each.
constexpr int kSlotsW = 6, kSlotsX = 8;
// At the start and the end of a tile so many stages are worked on half by half (all of the first half's, then all of the second
// half's), so that the first half's accumulator is drained while the second half's is still being filled.
constexpr int kSkew = 4;
static_assert(kSkew <= kSlotsW && 2 * kSkew <= kSlotsX, "the ring holds the stages that are worked on half by half");
constexpr int kFirstEpilogueWarp = 2;
constexpr int kEpilogueWarps = 8;       // two per quarter of the tensor memory's lanes
constexpr int kFirstProducerWarp = kFirstEpilogueWarp + kEpilogueWarps;
constexpr int kProducerGroups = kProducerWarps / 4;   // four warps fill the weight slot of a stage, the groups take the stages in turn
constexpr int kGemmWarps = kFirstProducerWarp + kProducerWarps;
constexpr int kGemmThreads = 32 * kGemmWarps;
static_assert(kProducerGroups <= kSlotsW, "see stage_free in the kernel");
constexpr int kTmemCols = 512;    // two 128 x 256 fp32 accumulators per CTA

constexpr int kModeForward = 0, kModeBackward = 1, kModeDense = 2;

constexpr int kMaxBatch = 4;      // weights of the same shape that one launch can walk (lowra_lora_*_batch)

// One weight of a call: its quantised state, the deal of its rows, its output, its down-projected activations.
struct Member {
    RowLayout L;
    const uint8_t* packed;
    const float* absmax;
    const float* maps;
    const uint32_t* items;    // from the deal: row words (forward) or row records (backward)
    uint16_t* out;            // [M, ld_out] bf16
    uint16_t* T;              // [M, rp] bf16: s * X . A (forward) or s * dY . B^T (backward), written by the T tiles
    uint32_t* flags;          // [token tiles][kCluster] set to the call's number when a CTA's half of T is complete
    int M;                    // this member's tokens (the batch calls: the same for all; several adapters: a group's)
    int st0;                  // token tiles of the members before this one
};

// Tensor maps of one member: token operand, T, factor of the T tiles, factor of the LoRA blocks.
struct MemberMaps {
    CUtensorMap tmB, tmT, tmFt, tmFl;
};
template <int NB>
struct KMaps {
    MemberMaps m[NB];
};
using BatchMaps = KMaps<kMaxBatch>;

// What a launch needs beside its members.  (The kernel is instantiated for one member and for kMaxBatch members: a
// plain call then carries 0.7 KB of kernel parameters instead of 2.8 KB, which its launch latency shows.)
struct GemmCommon {
    int count;              // members (1 for the plain calls); all of one shape
    uint32_t* flags;        // the flags that stay in the workspace from call to call
    uint32_t* status;
    // Calls on one workspace are numbered: `epoch` holds the number of the last call that ran on it, a call's own
    // number is that + 1, and a flag is up when it holds the call's number - so flags left over from earlier calls
    // never need clearing.  The last CTA to leave (counted in `exits`) writes the call's number back.
    uint32_t* epoch;
    uint32_t* exits;
    int n_flags;            // their number, for the wrap of the numbering
    int wide_only;          // (host) token tiles of 512 only: the call's flags are counted for those
    float s;
    int rp;                 // LoRA rank rounded up to 64
    int M;                  // tokens of the largest member (host: schedule choice)
    int super_total;        // token tiles of all members
    int R;                  // A-operand rows in total: N (forward, dense) or K (backward)
    int C;                  // main contraction length: K (forward, dense) or N (backward)
    int ld_out;             // = R
    int out_align;          // what every address of a row's 32-column piece is a multiple of: 32, 16 or 2 bytes
    int main_blocks;        // ceil(C / 64)
    int lora_blocks;        // rp / 64 (0 in dense mode)
    int tiles_r;            // tiles of 256 operand rows of a member (all members have one shape)
    // schedule of the tiles that are cut between clusters (set by the launcher; sk == 0: whole tiles, dealt round-robin)
    float* sk_part;         // fp32 partial tiles: for either half of the tokens, [kCluster][256 rows][128 tokens] per cluster.  Points in front of them by
                            // the place of cluster 0, which has none of its own.
    int part_halves;        // (host) halves of a token tile that the slots have room for: 2, or 1, or 0 (no tile is cut)
    uint32_t* sk_flags;     // [clusters][kCluster] raised when a CTA's partial tile is complete
    int halves;             // token tiles of 256 (1) or 512 tokens (2)
    int t_split;            // > 1: so many clusters share a T tile, and do nothing else
    int w_split;            // > 1: so many clusters share a weight tile, from cluster sk_c0 on, and do nothing else
    int sk;
    int sk_c0;              // the first cluster that gets a range
    int sk_first;           // first weight tile of the ranges
    int sk_num;             // contraction blocks of the weight tiles behind the whole rows, plus what follows
    int sk_extra;           // blocks that a cluster with a T tile is charged (negative: credited) against its range
    unsigned long long wait_ns;   // limit of every device-side wait (lowra_set_wait_limit)
    int diag_drop_t_flags;  // diagnostic (lowra_diag_drop_t_flags): the T tiles do not raise their flags, so the waits
                            // for them run out and the call ends with LOWRA_ERR_TIMEOUT
};
template <int NB>
struct KParams : GemmCommon {
    Member mem[NB];
};
using GemmParams = KParams<kMaxBatch>;
unsigned long long wait_limit_ns();   // the process-wide limit, 1 s unless lowra_set_wait_limit changed it
constexpr int kMaxClusters = kNumSMs / kCluster;
constexpr size_t kSkHalfFloats = (size_t)kHalfT / kCluster * kPairR;   // a CTA's partial tile for every 256 tokens: its 128 of them x 256 rows
constexpr size_t kSkAllFloats = (size_t)(kMaxClusters - 1) * kCluster * kSkHalfFloats, kSkHalfBytes = kSkAllFloats * 4;   // of all clusters

constexpr uint32_t kSmemSlot = 128 * kTileC * 2;   // 16 KB: 128 operand rows or tokens of a stage
constexpr uint32_t kSmemRing = (kSlotsW + kSlotsX) * kSmemSlot;
constexpr uint32_t kSmemBarriers = 1024;
// no alignment slack: the dynamic shared memory of a kernel without static shared memory starts 1024-byte
// aligned (checked by the kernel, which the swizzled operand tiles need)
constexpr uint32_t kGemmSmemBytes = kSmemRing + kSmemBarriers;
static_assert(kGemmSmemBytes <= 232448, "227 KB of shared memory per CTA");

lowra_status launch_fused(int mode, const GemmParams& G, const BatchMaps& TM, cudaStream_t stream);
float fused_estimate(int N, int K, int M, int r, int count);
int fused_schedule(bool backward, int N, int K, const int32_t* Ms, int count, int r, int* tile_tokens, int* w_split, int* t_split);   // what a call would run (diagnostic)

// ---- forward pass for few tokens (gemm_small.cu) --------------------------------------------
constexpr int kSmallTokens = 64;    // members of up to so many tokens may take it, of 16 and fewer do
constexpr int kSmallMembers = 8;    // per launch
struct SmallMember {
    RowLayout L;
    const uint8_t* packed;
    const float* absmax;
    const float* maps;
    const uint16_t *X, *A, *B;
    uint16_t *Y, *T;          // T [M, rp]: s X A, as the fused calls leave it
    int M;
};
float small_estimate(const int32_t* n, int K, int r, int units, int most);
template <int NB>   // members the kernel's parameters have room for
struct SmallParams {
    SmallMember m[NB];
    int count, N, K, r, rp;
    float s;
    uint32_t* status;
    int clear_status;         // the call brings no deal: its status word starts from zero
    int one_weight;           // all members have the same layout, codes and absmax (several adapters)
};
lowra_status launch_small(const SmallParams<kSmallMembers>& P, cudaStream_t stream);
bool small_takes_units(const SmallParams<kSmallMembers>& P);     // whether that launch is units_kernel

// One skinny product D [R, rp] = P . Q (see gemm_grad.cu), written in bf16 as out [R, ld_out] or, transposed,
// as out [n_cols, ld_out].
struct SkinnyProduct {
    CUtensorMap tmP;  // box of [64 c][64 rows] (a_mn) or [128 rows][64 c]
    CUtensorMap tmQ;  // box of [64 c][64 columns] (b_mn) or [rp columns][64 c]
    uint16_t* out;
    int R;            // rows of D
    int C;            // length of the contraction
    int n_cols;       // columns of D that are written (a multiple of 16)
    int ld_out;
    int a_mn, b_mn;   // 1: the row (column) index of P (Q) is the contiguous one in memory
    int transposed;
    float scale;
};
// Two products that share nothing but a launch.
struct SkinnyPair {
    SkinnyProduct p[2];
    uint32_t* status;
    int rp;           // columns of D (64 or 128), of both
    int tiles0;       // row tiles of the first product (set by the launcher)
    int clear_status; // the status word starts from zero here
    unsigned long long wait_ns;   // limit of every device-side wait
};
lowra_status launch_skinny(SkinnyPair& pair, cudaStream_t stream);

}  // namespace lowra
