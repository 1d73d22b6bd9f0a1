// lowra_learn_codebooks: weighted Lloyd-Max per output channel (paper Section 5, "Weighted Lloyd's for LoRA
// Quantization", and the appendix "Weighted Lloyd-Max Algorithm"; the appendix on the learner's initialisation
// gives the initial tables, which the caller passes in).
//
// For every row, at the row's assigned precision b: the data are the row's normalised values n_i (block
// absmax normalisation exactly as in lowra_encode), each weighted by the absmax of its block; starting from the
// given levels y and thresholds t, T times: assign every value to its bucket (number of thresholds <= n),
// replace every level by the weighted mean of its bucket (an empty bucket keeps its level), set the thresholds
// to the midpoints of neighbouring levels.  Levels and thresholds in fp64, sums in 64-bit fixed point.  Output: the levels rounded to fp32 and the
// midpoints of those fp32 levels (computed in fp64, rounded to fp32), in [N, 16] tables.
//
// Three kernels.  learn_kernel adds the whole row up in every round.  ordered_learn_kernel brings every block's values into order and then searches
// them, a block per lane.  sorted_learn_kernel brings the whole row into order, after which a round takes a few hundred of its values.  The more
// thresholds and rounds, the more order pays (kernel_for).
#include <float.h>
#include <math.h>
#include <string.h>

#include "lowra_common.cuh"

namespace lowra {


struct LearnParams {
    RowLayout L;
    const float* W;       // [N, K] original order
    float* maps;          // [N, 16] original order ([3][N][16] in the three-precision form: plane c = 2^c bits)
    float* thresholds;    // likewise
    int iterations;
    int N, K;             // the three-precision form has no layout: every row is learnt at 1, 2 and 4 bits
    int row0;             // this launch's rows: stored rows row0 .. row0 + grid - 1
    int turn;             // see enter()
    int bins;             // sorted rows: cells
    int one;              // 1, which the compiler does not know
    unsigned near_zero;   // see too_coarse
    double init_y[3][16];  // initial levels per class (1, 2, 4 bits)
    double init_t[3][16];  // initial thresholds per class
};

// The rows of one call may go to several launches, which know nothing of each other's rows.  turn 1, the first of them, lets the next one
// begin once everything before the call is complete; turn 2 does not wait for the launch before it to begin but to end, so that
// what comes after it may rely on all.  turn 0: a launch by itself.
__device__ __forceinline__ void enter(int turn) {
    if (turn != 2) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void leave(int turn) {
    if (turn == 2) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// NV sums per lane (NV = 4, 8 or 16) added up over the warp: instead of NV butterflies over all 32 lanes, every step
// hands half of a lane's values to its partner and adds the partner's other half to its own, so that the number of
// values halves with the distance; once a lane holds one value the remaining steps are plain butterflies.  Afterwards
// the lanes whose low bits are zero hold the totals: value number lane / (32 / NV) in v[0].  A fixed order of additions.
template <int NV>
__device__ __forceinline__ void warp_sums(long long (&v)[NV], int lane) {
    int d = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, d >>= 1) {
        const bool upper = (lane & d) != 0;
#pragma unroll
        for (int k = 0; k < n / 2; ++k) {
            const long long send = upper ? v[k] : v[k + n / 2];
            const long long keep = upper ? v[k + n / 2] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
    }
#pragma unroll
    for (; d >= 1; d >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
}

// ---------------------------------------------------------------------------------------------------------------------------------
// The arithmetic of all kernels.  A bucket's sums of w and of w * n are formed on a grid, so that they do not depend on the order
// of the additions: results are reproducible, and the same whichever kernel takes the row.  Let the row's largest weight be below
// 2^e.  fp64 numbers from 64 * 2^e to 128 * 2^e are multiples of u = 2^(e - 46), and adding to g = 96 * 2^e takes w (to nearest) and w * n
// (down) to that grid: s + w * n, one fused multiply-add rounding down, is s plus w * n taken down, whatever s is, so that a
// run of sixteen elements is a chain of these.  The sums are whole numbers of u, added up in 64-bit integers.  An element of a bucket costs its
// sum less than u, K of them less than 2^-24 of a sum of 2^24 K u, a rounding to fp32.  A bucket whose sum is nearer to zero (light elements only,
// or a mean next to zero) is added up again with what the grid leaves over.
__device__ __forceinline__ double grid_of(float most) {   // g
    return 96.0 * (most > 0.0f && most < INFINITY ? ldexp(1.0, ilogbf(most) + 1) : 1.0);
}
__device__ __forceinline__ unsigned long long grid_bits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ long long grid_product(double n, double w, double g) { return (long long)(grid_bits(__fma_rd(n, w, g)) - grid_bits(g)); }
__device__ __forceinline__ long long grid_weight(double w, double g) { return (long long)(grid_bits(w + g) - grid_bits(g)); }
// A block's weight in multiples of 2^e (for the grid 96), where that is kept instead of the absmax; what is positive stays positive.
constexpr double kGrid = 96.0;
__device__ __forceinline__ float weight_scale(float row_most) {
    return row_most > 0.0f && row_most < INFINITY ? (float)ldexp(1.0, -ilogbf(row_most) - 1) : 0.0f;
}
__device__ __forceinline__ float scaled_weight(float m, float scale) { return m > 0.0f && scale > 0.0f ? fmaxf(__fmul_rn(m, scale), FLT_MIN) : 0.0f; }
// the larger one; NaN if one is NaN (a row that holds a NaN, an infinity or a block whose reciprocal overflows has no mean: its
// levels come out as NaN)
__device__ __forceinline__ float max_nan(float a, float b) {
    float m;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
    return m;
}

// Whether a bucket's sum of w n is not enough: below 2^24 K u (near_zero: the upper half of that as an fp64 number, K rounded down to a power of two).  Exactly zero is
// the sum of zeros.  But an empty bucket and one of weights below u look alike: rows that have such weights (zero_too = 1) are looked through for
// them.  (Rows of a few different values have many empty buckets, and took up to 40 times as long when all were looked through for them.)
__device__ __forceinline__ bool too_coarse(double sn, unsigned near_zero, unsigned zero_too) {
    return ((unsigned)__double2hiint(sn) & 0x7fffffffu) - 1u + zero_too < near_zero;
}
constexpr float kVanishing = 0x1p-44f;   // scaled weights from here on are above u
// A bucket added up again, by all threads that call this (element(p): value and scaled weight number p of p0, p0 + step, ... below p1): on the grid
// kGrid, or, where its weights vanish there, on one of its own.  wn and w in multiples of u, the others in multiples of 2^-46 u.
struct Fine {
    long long wn, wn_lo, w, w_lo;
};
__device__ __forceinline__ void add_up(Fine& f) {       // over the warp
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        f.wn += __shfl_xor_sync(0xffffffffu, f.wn, d);
        f.wn_lo += __shfl_xor_sync(0xffffffffu, f.wn_lo, d);
        f.w += __shfl_xor_sync(0xffffffffu, f.w, d);
        f.w_lo += __shfl_xor_sync(0xffffffffu, f.w_lo, d);
    }
}
template <int UNROLL, typename F>
__device__ __forceinline__ Fine fine_sums(F element, int p0, int p1, int step, float t_lo, float t_hi, double g) {
    const double g2 = g * 0x1p-46;
    Fine f = {0, 0, 0, 0};
#pragma unroll UNROLL
    for (int p = p0; p < p1; p += step) {
        const float2 e = element(p);
        const bool in = t_lo <= e.x && e.x < t_hi;
        const double n = in ? (double)e.x : 0.0, w = in ? (double)e.y : 0.0;
        const double a = __fma_rd(n, w, g), b = __dadd_rn(w, g);           // what they leave over is exact
        f.wn += (long long)(grid_bits(a) - grid_bits(g));
        f.w += (long long)(grid_bits(b) - grid_bits(g));
        f.wn_lo += (long long)(grid_bits(__dadd_rd(__fma_rn(n, w, -__dsub_rn(a, g)), g2)) - grid_bits(g2));
        f.w_lo += (long long)(grid_bits(__dadd_rn(__dsub_rn(w, __dsub_rn(b, g)), g2)) - grid_bits(g2));
    }
    add_up(f);
    return f;
}
template <typename F>
__device__ __forceinline__ float largest_weight(F element, int p0, int p1, int step, float t_lo, float t_hi) {
    float most = 0.0f;
    for (int p = p0; p < p1; p += step) {
        const float2 e = element(p);
        if (t_lo <= e.x && e.x < t_hi) most = fmaxf(most, e.y);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, d));
    return most;
}
__device__ __forceinline__ double fine_mean(const Fine& f) {
    return ((double)f.wn + 0x1p-46 * (double)f.wn_lo) / ((double)f.w + 0x1p-46 * (double)f.w_lo);
}

// number of thresholds <= x among t[0 .. L-2] (sorted): branch-free binary search, L = 2, 4 or 16.
// x is an fp32 value and tf[j] is the least fp32 number >= the fp64 threshold t[j], so "t[j] <= x" (in fp64) and
// "tf[j] <= x" (in fp32) are the same statement.
template <int B>
__device__ __forceinline__ int bucket_of(float x, const float* tf) {
    if (B == 1) return tf[0] <= x ? 1 : 0;
    if (B == 2) {
        const int hi = tf[1] <= x ? 2 : 0;
        return hi + (tf[hi] <= x ? 1 : 0);
    }
    int c = tf[7] <= x ? 8 : 0;
    c += tf[c + 3] <= x ? 4 : 0;
    c += tf[c + 1] <= x ? 2 : 0;
    c += tf[c] <= x ? 1 : 0;
    return c;
}

// Where group of four elements number q of a row lies in shared memory (in units of 16 bytes).  The rounds read the row
// sixteen elements = four groups per thread at a time (eight in the 4-bit rounds); with the groups of every set of four
// exchanged among themselves by the number of the pair of sets they are in, the eight lanes that share a shared-memory
// wavefront fall into eight different 16-byte columns, in the rounds' reads and in the loader's writes alike.
__device__ __forceinline__ int quad_slot(int q) { return q ^ ((q >> 3) & 3); }

// The row: asynchronous coalesced 128-bit copies, all of them in flight together; then every thread normalises sixteen elements at a
// time where they lie (as in lowra_encode: reciprocal rounded to nearest, one multiplication): the four lanes that hold a
// 64-element block between them find its absmax in two shuffles.  Returns the row's largest absmax and its smallest but zero.  Ends with a
// barrier.
template <int THREADS>
__device__ float2 load_row(const LearnParams& P, int r, float* xs, float* ws, float* most_of) {
    const int K = P.K;
    const int tid = threadIdx.x;
    const float* wrow = P.W + (size_t)r * K;
    for (int i = 4 * tid; i < K; i += 4 * THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(xs + 4 * quad_slot(i >> 2))), "l"(wrow + i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float most = 0.0f, least = INFINITY;
    for (int run = tid; run < (K / 16 + 31) / 32 * 32; run += THREADS) {   // (a warp stays together)
        float4 v[4];
        float m = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = run < K / 16 ? *reinterpret_cast<const float4*>(xs + 4 * quad_slot(4 * run + q)) : make_float4(0.f, 0.f, 0.f, 0.f);
            m = max_nan(max_nan(m, max_nan(fabsf(v[q].x), fabsf(v[q].y))), max_nan(fabsf(v[q].z), fabsf(v[q].w)));
        }
        m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const float inv = (m == 0.0f) ? 0.0f : __frcp_rn(m);
        most = max_nan(max_nan(most, m), __fmul_rn(inv, 0.0f));
        if (m > 0.0f) least = fminf(least, m);
        if (run < K / 16) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<float4*>(xs + 4 * quad_slot(4 * run + q)) =
                    make_float4(__fmul_rn(v[q].x, inv), __fmul_rn(v[q].y, inv), __fmul_rn(v[q].z, inv), __fmul_rn(v[q].w, inv));
            if ((run & 3) == 0) ws[run >> 2] = m;
        }
    }
#pragma unroll
    for (int d = 4; d < 32; d <<= 1) {
        most = max_nan(most, __shfl_xor_sync(0xffffffffu, most, d));
        least = fminf(least, __shfl_xor_sync(0xffffffffu, least, d));
    }
    if ((tid & 31) == 0) { most_of[2 * (tid >> 5)] = most; most_of[2 * (tid >> 5) + 1] = least; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) { most = max_nan(most, most_of[2 * w]); least = fminf(least, most_of[2 * w + 1]); }
    return make_float2(most, least);
}

// learn_kernel.  One CTA per row: the row is read from HBM once, normalised on its way into shared memory; the T passes run out of
// shared memory.  Every thread keeps private sums per bucket: in registers for 1 and 2 bits, in a bank-conflict-free
// slice of shared memory for 4 bits; they are added up by a halving exchange inside a warp, then across warps.  One barrier
// per round; every warp forms the new levels and thresholds itself; a row whose thresholds have settled (as fp32 numbers) skips its
// remaining rounds.
//
// The mean of the bucket [t_lo, t_hi) by the whole CTA; y if it weighs nothing (vanished: nothing on the row's grid).  scratch: five words per warp
// that nobody reads, free again at the end.
template <int THREADS>
__device__ __noinline__ double fine_mean_row(const float* xs, const float* ws, float row_most, int K, float t_lo, float t_hi, bool vanished,
                                             double y, long long* scratch) {
    constexpr int kWarps = THREADS / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float scale = weight_scale(row_most);
    auto element = [&](int p) { return make_float2(xs[4 * quad_slot(p >> 2) + (p & 3)], scaled_weight(ws[p / kBlock], scale)); };
    double g = kGrid;
    if (vanished) {
        float* most_of = reinterpret_cast<float*>(scratch + 4 * kWarps);
        float most = largest_weight(element, tid, K, THREADS, t_lo, t_hi);
        if (lane == 0) most_of[warp] = most;
        __syncthreads();
        for (int w = 0; w < kWarps; ++w) most = fmaxf(most, most_of[w]);
        g = grid_of(most);
        if (!(most > 0.0f)) {
            __syncthreads();
            return y;
        }
    }
    Fine f = fine_sums<2>(element, tid, K, THREADS, t_lo, t_hi, g);
    if (lane == 0) { scratch[4 * warp] = f.wn; scratch[4 * warp + 1] = f.wn_lo; scratch[4 * warp + 2] = f.w; scratch[4 * warp + 3] = f.w_lo; }
    __syncthreads();
    f = Fine{0, 0, 0, 0};
    for (int w = 0; w < kWarps; ++w) { f.wn += scratch[4 * w]; f.wn_lo += scratch[4 * w + 1]; f.w += scratch[4 * w + 2]; f.w_lo += scratch[4 * w + 3]; }
    __syncthreads();
    return fine_mean(f);
}

// One pass at 1 or 2 bits: this thread's sums over the elements at or above threshold j - 1 (j >= 1) and, if ALL, over all (j = 0).
template <int B, int THREADS, bool ALL>
__device__ __forceinline__ void few_buckets(const float* xs, const float* ws, int K, double g, const float* th, unsigned long long* cn, long long* cw) {
    constexpr int Lv = 1 << B, j0 = ALL ? 0 : 1;
#pragma unroll
    for (int j = j0; j < Lv; ++j) { cn[j] = 0ull; cw[j] = 0; }
    for (int run = threadIdx.x; run < K / 16; run += THREADS) {   // elements 16 run .. 16 run + 15, all in block run / 4
        const float4 xa = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(4 * run));
        const float4 xb = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(4 * run + 1));
        const float4 xc = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(4 * run + 2));
        const float4 xd = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(4 * run + 3));
        const double w = (double)ws[run >> 2];
        const float xf[16] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w, xc.x, xc.y, xc.z, xc.w, xd.x, xd.y, xd.z, xd.w};
        double s[Lv];
        int cq[Lv];
#pragma unroll
        for (int j = j0; j < Lv; ++j) { s[j] = g; cq[j] = 0; }
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const double x = (double)xf[u];
            if (ALL) s[0] = __fma_rd(x, w, s[0]);
#pragma unroll
            for (int j = 1; j < Lv; ++j) {
                int hi;
                asm("{\n\t.reg .pred p;\n\tsetp.le.f32 p, %2, %3;\n\tselp.b32 %0, %4, 0, p;\n\t@p add.s32 %1, %1, 1;\n\t}"
                    : "=r"(hi), "+r"(cq[j]) : "f"(th[j - 1]), "f"(xf[u]), "r"(__double2hiint(x)));
                s[j] = __fma_rd(__hiloint2double(hi, __double2loint(x)), w, s[j]);
            }
        }
        const long long wg = grid_weight(w, g);
        if (ALL) cq[0] = 16;
#pragma unroll
        for (int j = j0; j < Lv; ++j) {
            cn[j] += grid_bits(s[j]) - grid_bits(g);
            cw[j] += cq[j] * wg;
        }
    }
}

// T rounds on the row parked in shared memory, at B bits; tables to maps_out / thr_out ([16] each).
// One barrier per round: the warps leave their partial sums in shared memory (two buffers, used in turn), meet once, and
// then EVERY warp forms the new levels and thresholds for itself - lane j holds level j and threshold j in registers, the
// same numbers in every warp since they come from the same sums - so nobody waits for a first warp to publish them.
template <int B, int THREADS>
__device__ void learn_row(const LearnParams& P, const float* xs, const float* ws, float row_most, unsigned zero_too, long long* acc, long long* red2,
                          float* tfw_all, int iterations, float* maps_out, float* thr_out) {
    constexpr int kLearnThreads = THREADS, kLearnWarps = THREADS / 32;
    constexpr int Lv = 1 << B;      // levels
    constexpr int c = B >> 1;       // class index
    const int K = P.K;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* tf = tfw_all + warp * 16;                      // 4 bits: this warp's copy of the thresholds (bucket search by index)
    double ylane = lane < Lv ? P.init_y[c][lane] : 0.0;   // level `lane`
    float tlane = lane + 1 < Lv ? __double2float_ru(P.init_t[c][lane]) : 0.0f;   // threshold `lane`: the least fp32 number >= it
    float th[B <= 2 ? Lv - 1 : 1];                        // 1 and 2 bits: all thresholds in registers
    if (B <= 2) {
#pragma unroll
        for (int j = 0; j < Lv - 1; ++j) th[j] = __double2float_ru(P.init_t[c][j]);
    } else {
        __syncthreads();   // (a row's first tenant of this space was its absmax)
        if (lane < 16) tf[lane] = tlane;
        __syncwarp();
    }

    unsigned long long all_n = 0ull;
    long long all_w = 0;
    const double g = grid_of(row_most);
    const bool bad = !(row_most < INFINITY) && iterations > 0;
    for (int it = 0; it < iterations; ++it) {
        long long* red = red2 + (it & 1) * (2 * 16 * kLearnWarps);
        // ---- one pass: private sums of w * n and w per bucket.  The weight is the same for the sixteen elements a thread
        // takes at a time (a quarter of a 64-element block): the elements are counted per bucket, and the weight's sum follows.
        if (B <= 2) {
            // Few buckets: no bucket index at all.  cn[0] / cw[0] take all elements, cn[j] / cw[j] (j >= 1) those at or above
            // threshold j - 1, and a bucket's sums are the difference of two neighbours.  An element that is out becomes
            // a tiny positive number (the upper half of the fp64 number zero), which rounding down leaves without effect: one
            // selection instead of a conditional addition (1 bit, 4096 x 4096: 8.2 against 10 us a round).
            // (The first round forms cn[0] for all.)
            unsigned long long cn[Lv];
            long long cw[Lv];
            if (it == 0) few_buckets<B, THREADS, true>(xs, ws, K, g, th, cn, cw);
            else few_buckets<B, THREADS, false>(xs, ws, K, g, th, cn, cw);
            if (it == 0) { all_n = cn[0]; all_w = cw[0]; }
            cn[0] = all_n;
            cw[0] = all_w;
            long long v[2 * Lv];
#pragma unroll
            for (int j = 0; j < Lv; ++j) {
                v[2 * j] = (long long)(j == Lv - 1 ? cn[j] : cn[j] - cn[j + 1]);
                v[2 * j + 1] = j == Lv - 1 ? cw[j] : cw[j] - cw[j + 1];
            }
            warp_sums<2 * Lv>(v, lane);
            if ((lane & (32 / (2 * Lv) - 1)) == 0) red[(lane / (32 / (2 * Lv))) * kLearnWarps + warp] = v[0];
        } else {
            // 16 buckets: the sums live in shared memory, one (w n, w) pair per thread and bucket; eight elements at a
            // time, their bucket searches side by side
            longlong2* acc2 = reinterpret_cast<longlong2*>(acc);
#pragma unroll
            for (int j = 0; j < Lv; ++j) acc2[j * kLearnThreads + tid] = make_longlong2(0, 0);
            for (int run = tid; run < K / 8; run += kLearnThreads) {
                const float4 xa = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(2 * run));
                const float4 xb = *reinterpret_cast<const float4*>(xs + 4 * quad_slot(2 * run + 1));
                const double w = (double)ws[run >> 3];
                const long long wg = grid_weight(w, g);
                const float xf[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
                int b[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) b[u] = bucket_of<B>(xf[u], tf);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    longlong2 a = acc2[b[u] * kLearnThreads + tid];
                    a.x += grid_product((double)xf[u], w, g);
                    a.y += wg;
                    acc2[b[u] * kLearnThreads + tid] = a;
                }
            }
#pragma unroll
            for (int half = 0; half < 2; ++half) {   // eight buckets = sixteen sums at a time
                long long v[16];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const longlong2 a = acc2[(8 * half + j) * kLearnThreads + tid];
                    v[2 * j] = a.x;
                    v[2 * j + 1] = a.y;
                }
                warp_sums<16>(v, lane);
                if ((lane & 1) == 0) red[(16 * half + lane / 2) * kLearnWarps + warp] = v[0];
            }
        }
        __syncthreads();
        // ---- new levels, then midpoints with a shuffle in between: every warp
        bool coarse = false, vanished = false;
        if (lane < Lv) {
            long long sn = 0, sd = 0;
#pragma unroll
            for (int w2 = 0; w2 < kLearnWarps; ++w2) { sn += red[(2 * lane) * kLearnWarps + w2]; sd += red[(2 * lane + 1) * kLearnWarps + w2]; }
            vanished = sd <= 0;
            coarse = too_coarse((double)sn, P.near_zero, zero_too);
            if (!vanished) ylane = (double)sn / (double)sd;
        }
        for (unsigned left = __ballot_sync(0xffffffffu, coarse); left != 0u; left &= left - 1u) {     // (the same in every warp)
            const int k = __ffs(left) - 1;
            const float t_lo = __shfl_sync(0xffffffffu, tlane, max(k - 1, 0)), t_hi = __shfl_sync(0xffffffffu, tlane, k);
            const double mean = fine_mean_row<THREADS>(xs, ws, row_most, K, k > 0 ? t_lo : -INFINITY, k < Lv - 1 ? t_hi : INFINITY,
                                                       __shfl_sync(0xffffffffu, (int)vanished, k) != 0, __shfl_sync(0xffffffffu, ylane, k),
                                                       red2 + ((it & 1) ^ 1) * (2 * 16 * kLearnWarps));
            if (lane == k) ylane = mean;
        }
        const double yn = __shfl_down_sync(0xffffffffu, ylane, 1);
        bool same = true;
        if (lane + 1 < Lv) {
            const float tn = __double2float_ru((ylane + yn) * 0.5);
            same = tn == tlane;
            tlane = tn;
        }
        if (B <= 2) {
#pragma unroll
            for (int j = 0; j < Lv - 1; ++j) th[j] = __shfl_sync(0xffffffffu, tlane, j);
        } else {
            if (lane < 16) tf[lane] = tlane;
            __syncwarp();
        }
        // thresholds that have not moved (as the fp32 numbers the elements are compared with) assign every element
        // as before: the next round would form the same sums and change nothing, nor any later one
        if (__all_sync(0xffffffffu, same)) break;
    }

    // ---- tables: fp32 levels, midpoints of the fp32 levels; unused levels 0, unused thresholds +inf
    if (warp == 0) {
        const float m = (lane < Lv) ? (bad ? __int_as_float(0x7fc00000) : (float)ylane) : 0.0f;
        const float mn = __shfl_down_sync(0xffffffffu, m, 1);
        if (lane < kTableStride) {
            maps_out[lane] = m;
            thr_out[lane] = (lane + 1 < Lv) ? (float)(((double)m + (double)mn) * 0.5) : __int_as_float(0x7f800000);
        }
    }
    __syncthreads();   // the sums in shared memory are reused by the next run, the row buffer by the next row
}

// FOUR: with rounds at 4 bits.  Only these need the 32 KB of per-thread bucket sums in shared memory, and the rounds of a row are a
// chain of short phases between barriers, so what hides their latency is the number of CTAs per SM: without those 32 KB three times
// as many fit (all-1-bit rows: 0.52 -> 0.34 ms on 4096 x 11008 at ten rounds).
// THREADS: short rows take fewer, which all have work, and pay less for the end of a round (1-bit rows, T = 2, 4096 of them: 20.5 ->
// 13.5 us at K = 1024, 29 -> 26 us at K = 4096; at K = 11008 the other way round: 86 against 72).
// What bounds it: instruction issue, five per element, round and threshold.  Together with the row's way in, 4096 x 4096, T = 2: 27.4 ->
// 24.5 us at 1 bit and 41.6 -> 37 at 2; 4096 x 11008: 78 -> 69 and 112 -> 101; without rounds 50 -> 38 there.
template <bool ALL3, bool FOUR, int THREADS>
__global__ void __launch_bounds__(THREADS) learn_kernel(const __grid_constant__ LearnParams P) {
    extern __shared__ __align__(16) unsigned char learn_smem[];
    constexpr int kWarps = THREADS / 32;
    // [2 x 2 * 16 * warps partial sums][FOUR: 2 * 16 * threads sums][K floats][nb floats][warps x 16 floats]
    long long* red2 = reinterpret_cast<long long*>(learn_smem);
    long long* acc = red2 + 2 * 2 * 16 * kWarps;
    float* xs = reinterpret_cast<float*>(acc + (FOUR ? 2 * 16 * THREADS : 0));
    float* ws = xs + P.K;
    float* tfw = ws + P.K / kBlock;   // 4-bit runs: a copy of the thresholds (fp32 upper neighbours) per warp
    enter(P.turn);
    // with a layout: stored rows from the last to the first, i.e. the longer 2-bit rows (4-bit rows) are handed out first and the
    // short 1-bit rows fill the gaps at the end
    const int i = P.row0 + (int)(gridDim.x - 1 - blockIdx.x);
    const int r = ALL3 ? i : P.L.perm[i];
    const float2 scale = load_row<THREADS>(P, r, xs, ws, tfw);
    const float most = scale.x;
    // (scaled_weight of the smallest against kVanishing, without the scaling: the largest lies between this power of two and the next)
    const unsigned zero_too = scale.y < __uint_as_float(__float_as_uint(most) & 0x7f800000u) * (2.0f * kVanishing) ? 1u : 0u;
    float* m = P.maps + (size_t)r * kTableStride;
    float* h = P.thresholds + (size_t)r * kTableStride;
    if (ALL3) {
        // the row under every precision, from the one copy in shared memory
        const size_t plane = (size_t)P.N * kTableStride;
        learn_row<1, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, P.iterations, m, h);
        learn_row<2, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, P.iterations, m + plane, h + plane);
        learn_row<4, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, FOUR ? P.iterations : 0, m + 2 * plane, h + 2 * plane);
    } else {
        const int b = P.L.precs[r];
        if (b == 1) learn_row<1, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, P.iterations, m, h);
        else if (b == 2) learn_row<2, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, P.iterations, m, h);
        else learn_row<4, THREADS>(P, xs, ws, most, zero_too, acc, red2, tfw, FOUR ? P.iterations : 0, m, h);
    }
    leave(P.turn);
}

// ---------------------------------------------------------------------------------------------------------------------------------
// Rounds on a sorted row.  A round needs, for every threshold, the weighted sums over the values below it.  With the row in
// (nearly) sorted order and running sums of it, that is one look-up and a short scan per threshold, whatever the number of
// rounds, levels and precisions - where a pass over the row costs about 13 thread instructions per element, half of them on the fp64
// and conversion pipes, and six times that at 4 bits.  One CTA per row:
//   - the row comes asynchronously into shared memory and from there, normalised (as in lowra_encode), into registers; bins_of(K)
//     equal cells of [-1, 1] are counted and their counts added up; then every value and its weight go to their place, a cell's
//     places being handed out by an atomic;
//   - running sums over every sixteen places;
//   - T rounds by one warp (in the three-precision form a warp per precision): threshold t lies in cell b; everything before cell b
//     is below it, so its sums are the running sums up to the last multiple of sixteen before the cell plus the values from there
//     to the end of the cell that are below t.
// The order inside a cell is that in which the atomics arrive, which integer sums do not see.
// What bounds it: shared-memory wavefronts (two atomics and an 8-byte store per element at random places: 24 wavefronts for 32
// elements, the pipe 77 % busy at T = 0) and, in the rounds, the latency of one warp's steps (about 1000 cycles each, hidden by the
// other rows of the SM).  For 4-bit rows and the three-precision form: 4096 x 4096 of 4 bits, T = 10, 109 us (ordered blocks 140, a pass over the row per
// round 415); three precisions 127 (181, 624).
constexpr int kSortedMaxK = 16384;         // 10 to 11 bytes of shared memory per element
int bins_of(int K) { int n = 256; while (n < K / 6) n *= 2; return n; }

struct Sums {
    long long wn, w;     // multiples of 2^-46
};

// Where place p lies in shared memory (in units of 8 bytes): the 16-byte pairs of every 16 places are exchanged among
// themselves, so that the eight lanes of a wavefront, which read 128 bytes apart, meet different banks.
__device__ __forceinline__ int sorted_slot(int p) { return p ^ ((p >> 3) & 14); }

// Cell of x among `bins`: monotone in x, so a value in an earlier cell than a threshold is below it.  Normalised values lie in
// [-1, 1] up to a rounding, thresholds anywhere; adding 2^23 rounds to a whole number in the low bits (the mask: NaN lands
// somewhere, but inside).
__device__ __forceinline__ int cell_of(float x, int bins) {
    return __float_as_int(fmaf(x, (float)(bins / 2 - 1), (float)(bins / 2) + 8388608.0f)) & (bins - 1);
}
__device__ __forceinline__ int cell_of_threshold(float t, int bins) { return cell_of(fminf(fmaxf(t, -1.0000005f), 1.0000005f), bins); }
__device__ __forceinline__ Sums shfl_xor_sums(const Sums& s, int d) {
    return Sums{__shfl_xor_sync(0xffffffffu, s.wn, d), __shfl_xor_sync(0xffffffffu, s.w, d)};
}

// The same by a warp; the bucket lies somewhere in places p0 .. p1 - 1.
__device__ __noinline__ double fine_mean_sorted(const float2* sorted, int p0, int p1, float t_lo, float t_hi, bool vanished, double y) {
    const int lane = threadIdx.x & 31;
    auto element = [&](int p) { return sorted[sorted_slot(p)]; };
    double g = kGrid;
    if (vanished) {
        const float most = largest_weight(element, p0 + lane, p1, 32, t_lo, t_hi);
        if (!(most > 0.0f)) return y;
        g = grid_of(most);
    }
    return fine_mean(fine_sums<1>(element, p0 + lane, p1, 32, t_lo, t_hi, g));
}

constexpr int kMany = 32 * 4;
// Sums of places p0 .. p1 - 1 whose values are below t, by a warp.
__device__ __noinline__ Sums sums_below(const float2* sorted, int p0, int p1, float t) {
    Sums s = {0, 0};
#pragma unroll 4
    for (int p = p0 + (int)(threadIdx.x & 31); p < p1; p += 32) {
        const float2 e = sorted[sorted_slot(p)];
        const double n = e.x < t ? (double)e.x : 0.0, w = e.x < t ? (double)e.y : 0.0;
        s.wn += grid_product(n, w, kGrid);
        s.w += grid_weight(w, kGrid);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const Sums o = shfl_xor_sums(s, d);
        s.wn += o.wn; s.w += o.w;
    }
    return s;
}

// One more value in cell c for every lane that is in; the lanes that share a cell add together, for one by one their additions wait for one another
// (not so where nobody asks for the place: the hardware adds up ones).  Returns the lane's place.
__device__ __forceinline__ int add_to_cell(uint32_t* cells, int c, bool in) {
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, in ? c : -1 - lane);
    const int leader = __ffs(peers) - 1;
    uint32_t before = 0u;
    if (in && lane == leader) before = atomicAdd(&cells[c], (uint32_t)__popc(peers));
    return (int)__shfl_sync(0xffffffffu, before, leader) + __popc(peers & ((1u << lane) - 1u));
}

// T rounds at B bits by one warp; tables to maps_out / thr_out ([16] each).  first[b]: places before cell b; run[i]: sums over
// the first 16 i places.  The G lanes of group j look after level j and the threshold above it (the last group: everything), all with
// the same values; what bounds a round is the length of this chain, so it has few shuffles.
template <int B, bool CROWDED>
__device__ __forceinline__ void learn_sorted(const LearnParams& P, const float2* sorted, const uint32_t* first, const Sums* run, int bins, float row_most,
                             float* maps_out, float* thr_out) {
    constexpr int Lv = 1 << B, c = B >> 1;
    constexpr int G = B == 4 ? 2 : 8;
    const int lane = threadIdx.x & 31, j = lane / G, K = P.K;
    const bool top = j >= Lv - 1;                          // no threshold above
    double y = j < Lv ? P.init_y[c][j] : 0.0;
    float t = !top ? __double2float_ru(P.init_t[c][j]) : INFINITY;   // the least fp32 number >= the threshold
    for (int it = 0; it < P.iterations; ++it) {
        const unsigned zero_too = *reinterpret_cast<const volatile uint32_t*>(first - 1);     // (not worth a register)
        const int b = cell_of_threshold(t, bins);
        const int p1 = top ? K : (int)first[b + 1], p0 = top ? K : (int)first[b] & ~15;
        const Sums base = run[p0 >> 4];
        Sums s = {0, 0};
        // (crowded rows: a cell of many places is the whole warp's work, below)
        for (int p = p0 + lane % G, end = CROWDED && p1 - p0 > kMany ? p0 : p1; p < end; p += G) {
            const float2 e = sorted[sorted_slot(p)];
            if (e.x < t) {
                s.wn += grid_product((double)e.x, (double)e.y, kGrid);
                s.w += grid_weight((double)e.y, kGrid);
            }
        }
        __syncwarp();
#pragma unroll
        for (int d = G / 2; d >= 1; d >>= 1) {
            const Sums o = shfl_xor_sums(s, d);
            s.wn += o.wn; s.w += o.w;
        }
        if (CROWDED) {
            for (unsigned left = __ballot_sync(0xffffffffu, p1 - p0 > kMany); left != 0u;) {
                const int k = (__ffs(left) - 1) / G;
                left &= ~(((1u << G) - 1u) << (k * G));
                const Sums all = sums_below(sorted, __shfl_sync(0xffffffffu, p0, k * G), __shfl_sync(0xffffffffu, p1, k * G), __shfl_sync(0xffffffffu, t, k * G));
                if (j == k) s = all;
            }
        }
        s.wn += base.wn; s.w += base.w;
        // the bucket: what lies below its upper threshold less what lies below its lower one
        Sums low = {__shfl_up_sync(0xffffffffu, s.wn, G), __shfl_up_sync(0xffffffffu, s.w, G)};
        if (j == 0) low.wn = low.w = 0;
        const double sn = (double)(s.wn - low.wn);
        const long long sw = s.w - low.w;
        if (j < Lv && sw > 0) y = sn / (double)sw;
        for (unsigned left = __ballot_sync(0xffffffffu, j < Lv && too_coarse(sn, P.near_zero, zero_too)); left != 0u;) {
            const int k = (__ffs(left) - 1) / G;
            left &= ~(((1u << G) - 1u) << (k * G));
            const float t_lo = k > 0 ? __shfl_sync(0xffffffffu, t, max(k - 1, 0) * G) : -INFINITY;
            const float t_hi = __shfl_sync(0xffffffffu, t, k * G);
            const int q0 = k > 0 ? (int)first[cell_of_threshold(t_lo, bins)] : 0, q1 = k < Lv - 1 ? (int)first[cell_of_threshold(t_hi, bins) + 1] : K;
            const double mean = fine_mean_sorted(sorted, q0, q1, t_lo, t_hi, __shfl_sync(0xffffffffu, (int)(sw <= 0), k * G) != 0,
                                                 __shfl_sync(0xffffffffu, y, k * G));
            if (j == k) y = mean;
        }
        const double yn = __shfl_down_sync(0xffffffffu, y, G);
        const float tn = !top ? __double2float_ru((y + yn) * 0.5) : INFINITY;
        // thresholds that have not moved (as the fp32 numbers the elements are compared with) assign every element as
        // before: the next round would form the same sums and change nothing, nor any later one
        const bool same = tn == t;
        t = tn;
        if (__all_sync(0xffffffffu, same)) break;
    }
    // tables: fp32 levels, midpoints of the fp32 levels; unused levels 0, unused thresholds +inf
    const double yl = __shfl_sync(0xffffffffu, y, min(lane, Lv - 1) * G);
    const float m = (lane < Lv) ? (row_most < INFINITY ? (float)yl : __int_as_float(0x7fc00000)) : 0.0f;
    const float mn = __shfl_down_sync(0xffffffffu, m, 1);
    if (lane < kTableStride) {
        maps_out[lane] = m;
        thr_out[lane] = (lane + 1 < Lv) ? (float)(((double)m + (double)mn) * 0.5) : __int_as_float(0x7f800000);
    }
}

// All rounds of row r.  Crowded rows by a function of their own, which leaves the others' registers alone.
template <bool ALL3, bool CROWDED>
__device__ __forceinline__ void learn_rounds(const LearnParams& P, const float2* sorted, const uint32_t* first, const Sums* run, float row_most, int r) {
    const int warp = threadIdx.x >> 5, bins = P.bins;
    float* y = P.maps + (size_t)r * kTableStride;
    float* h = P.thresholds + (size_t)r * kTableStride;
    if (ALL3) {   // a warp per precision
        const size_t plane = (size_t)P.N * kTableStride;
        for (int c = warp; c < 3; c += blockDim.x >> 5) {
            if (c == 0) learn_sorted<4, CROWDED>(P, sorted, first, run, bins, row_most, y + 2 * plane, h + 2 * plane);
            else if (c == 1) learn_sorted<2, CROWDED>(P, sorted, first, run, bins, row_most, y + plane, h + plane);
            else learn_sorted<1, CROWDED>(P, sorted, first, run, bins, row_most, y, h);
        }
    } else if (warp == 0) {
        learn_sorted<4, CROWDED>(P, sorted, first, run, bins, row_most, y, h);
    }
}
template <bool ALL3>
__device__ __noinline__ void learn_rounds_crowded(const LearnParams& P, const float2* sorted, const uint32_t* first, const Sums* run, float row_most, int r) {
    learn_rounds<ALL3, true>(P, sorted, first, run, row_most, r);
}

// Exclusive sums of v[0 .. NV-1] over the threads of the CTA (scratch: NV entries per warp).  Ends with a barrier.
template <int NV, typename T>
__device__ __forceinline__ void block_exclusive(T (&v)[NV], T (*scratch)[NV]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) incl[k] = v[k];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const T o = __shfl_up_sync(0xffffffffu, incl[k], d);
            if (lane >= d) incl[k] += o;
        }
    }
    if (lane == 31) {
#pragma unroll
        for (int k = 0; k < NV; ++k) scratch[warp][k] = incl[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = incl[k] - v[k];
    for (int w = 0; w < warp; ++w) {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] += scratch[w][k];
    }
    __syncthreads();
}

// THREADS threads at most, PER elements each, CTAS of them per SM.
template <bool ALL3, int THREADS, int PER, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) sorted_learn_kernel(const __grid_constant__ LearnParams P) {
    extern __shared__ __align__(16) unsigned char sorted_smem[];
    const int K = P.K, bins = P.bins, tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, n_warps = nt >> 5;
    // [K float2 values and weights in order; before that, the row][K / 16 + 1 Sums][32 x 2 long long][32 floats][0, crowded, zero_too, 0][cells]
    float2* sorted = reinterpret_cast<float2*>(sorted_smem);
    Sums* run = reinterpret_cast<Sums*>(sorted + K);
    long long(*scratch)[2] = reinterpret_cast<long long(*)[2]>(run + K / 16 + 1);
    float* most_of = reinterpret_cast<float*>(scratch + 32);
    uint32_t* cells = reinterpret_cast<uint32_t*>(most_of + 32) + 4;
    enter(P.turn);
    // stored rows from the last to the first: the 4-bit rows, whose rounds are a little longer, go out first
    const int i0 = P.row0 + (int)(gridDim.x - 1 - blockIdx.x);
    const int r = ALL3 ? i0 : P.L.perm[i0];
    const float* wrow = P.W + (size_t)r * K;
    const bool in = tid * PER < K;
#pragma unroll
    for (int u = 0; u < PER / 4; ++u) {
        const int i = 4 * (u * nt + tid);
        if (i < K)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sorted_smem + 4 * i)), "l"(wrow + i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int i = tid - 1; i < bins / 4; i += nt) *reinterpret_cast<uint4*>(cells + 4 * i) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- this thread's part of a block, its 16-byte pieces in an order that spreads the lanes over the banks
    float x[PER];
    float m = 0.0f;
#pragma unroll
    for (int j = 0; j < PER / 4; ++j) {
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) f = *reinterpret_cast<const float4*>(sorted_smem + 4 * PER * tid + 16 * (j ^ ((tid * PER / 32) & (PER / 4 - 1))));
        x[4 * j] = f.x; x[4 * j + 1] = f.y; x[4 * j + 2] = f.z; x[4 * j + 3] = f.w;
        m = max_nan(max_nan(m, max_nan(fabsf(f.x), fabsf(f.y))), max_nan(fabsf(f.z), fabsf(f.w)));
    }
    for (int d = 1; d < kBlock / PER; d <<= 1) m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, d));
    const float inv = (m == 0.0f) ? 0.0f : __frcp_rn(m);
    float most = max_nan(m, __fmul_rn(inv, 0.0f));
#pragma unroll
    for (int d = 16; d >= kBlock / PER; d >>= 1) most = max_nan(most, __shfl_xor_sync(0xffffffffu, most, d));
    if ((tid & 31) == 0) most_of[warp] = most;
    // ---- count the cells
#pragma unroll
    for (int e = 0; e < PER; ++e) x[e] = __fmul_rn(x[e], inv);
    // Crowded (for a warp): neighbours are equal in one lane of eight - a row of a few different values.
    const bool crowded = __popc(__ballot_sync(0xffffffffu, in && x[0] == x[1])) >= 4;
    if (crowded) cells[-3] = 1u;
    if (in) {
#pragma unroll
        for (int e = 0; e < PER; ++e) atomicAdd(&cells[cell_of(x[e], bins)], 1u);
    }
    __syncthreads();
    // ---- counts -> places before the cell
    {
        const int per = (bins / 4 + nt - 1) / nt, c0 = tid * per, c1 = min(c0 + per, bins / 4);
        uint32_t before[1] = {0u};
        for (int i = c0; i < c1; ++i) {
            const uint4 n = *reinterpret_cast<const uint4*>(cells + 4 * i);
            before[0] += n.x + n.y + n.z + n.w;
        }
        block_exclusive<1, uint32_t>(before, reinterpret_cast<uint32_t(*)[1]>(scratch));
        uint32_t b = before[0];
        for (int i = c0; i < c1; ++i) {
            const uint4 n = *reinterpret_cast<const uint4*>(cells + 4 * i);
            *reinterpret_cast<uint4*>(cells + 4 * i) = make_uint4(b, b + n.x, b + n.x + n.y, b + n.x + n.y + n.z);
            b += n.x + n.y + n.z + n.w;
        }
    }
    float row_most = 0.0f;
    for (int w = 0; w < n_warps; ++w) row_most = max_nan(row_most, most_of[w]);
    const float weight = scaled_weight(m, weight_scale(row_most));
    if (weight > 0.0f && weight < kVanishing) cells[-2] = 1u;
    __syncthreads();
    // ---- every value and its weight to their place; afterwards a cell's entry is the place where it ends
    if (crowded) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int place = add_to_cell(cells, cell_of(x[e], bins), in);
            if (in) sorted[sorted_slot(place)] = make_float2(x[e], weight);
        }
    } else if (in) {
#pragma unroll
        for (int e = 0; e < PER; ++e)
            sorted[sorted_slot((int)atomicAdd(&cells[cell_of(x[e], bins)], 1u))] = make_float2(x[e], weight);
    }
    __syncthreads();
    // ---- running sums: this thread's places, sixteen at a time
    {
        unsigned long long part[PER / 16][2], all[2] = {0ull, 0ull};     // (modulo 2^64)
#pragma unroll
        for (int q = 0; q < PER / 16; ++q) {
            part[q][0] = all[0]; part[q][1] = all[1];
            if (in) {
#pragma unroll
                for (int p = 0; p < 16; p += 2) {
                    const float4 e = *reinterpret_cast<const float4*>(sorted + sorted_slot(tid * PER + q * 16 + p));
                    all[0] += grid_bits(__fma_rd((double)e.x, (double)e.y, kGrid)) + grid_bits(__fma_rd((double)e.z, (double)e.w, kGrid));
                    all[1] += grid_bits((double)e.y + kGrid) + grid_bits((double)e.w + kGrid);
                }
                all[0] -= 16ull * grid_bits(kGrid);
                all[1] -= 16ull * grid_bits(kGrid);
            }
        }
        unsigned long long before[2] = {all[0], all[1]};
        block_exclusive<2, unsigned long long>(before, reinterpret_cast<unsigned long long(*)[2]>(scratch));
        if (in) {
#pragma unroll
            for (int q = 0; q < PER / 16; ++q)
                run[tid * (PER / 16) + q] = Sums{(long long)(before[0] + part[q][0]), (long long)(before[1] + part[q][1])};
        }
        if (tid == K / PER - 1) run[K / 16] = Sums{(long long)(before[0] + all[0]), (long long)(before[1] + all[1])};
    }
    __syncthreads();
    // ---- rounds
    const uint32_t* first = cells - 1;   // first[b]: the places before cell b
    if (first[-2] != 0u) learn_rounds_crowded<ALL3>(P, sorted, first, run, row_most, r);
    else learn_rounds<ALL3, false>(P, sorted, first, run, row_most, r);
    leave(P.turn);
}

// ---------------------------------------------------------------------------------------------------------------------------------
// Rounds on blocks in order.  A lane takes one absmax block (of short rows a half or a quarter), so that all its values have one weight and order is a matter
// of its registers alone: a sorting network, no atomics, no scattered stores (the order of a whole row costs 24 shared-memory wavefronts for 32
// elements, above).  The values lie in shared memory as [place][lane], with the sums of w * n before every fourth place; a lane finds a threshold's
// place in its block by bisection, every look-up free of bank conflicts, adds the few values of the last four below it, and the warp's sums are
// added up by a halving exchange.  The same sums on the same grid as in the other kernels, hence the same tables bit for bit.
// What bounds it: instruction issue (60 to 73 % of the slots, with the 16 warps that an SM's shared memory takes): 2400 instructions a warp until the first
// round, 1360 of them in the network, then 62 for a threshold and 150 for a round.  Against rounds through
// the row and the whole row's order, 4096 x 4096, T = 10: 80 -> 57 us at 60/35/5 % of 1/2/4 bits (70 -> 45 at 1 bit, 86 -> 56 at 2); three precisions, T = 2: 65.5 -> 54.1.
// Rows with one block 10^6 times heavier, nearly every bucket of which is added up again (fine_mean_ordered): 81 us, 121 with every block walked through for every bucket.
// Not taken: two blocks a lane in turn (49 -> 55 us at 1 bit, T = 10: half the warps); rows one after the other in a persistent grid, the next one's load
// in flight (66: five rows to an SM instead of eight); halves of blocks (a fifth less network, but every threshold twice: 61 -> 70 at 2 bits).
//
// Batcher's odd-even merge sort ("Sorting networks and their applications", 1968): layer (p, k), then those after it.  Both a minimum and a maximum go to
// the half-rate pipe, which bounds the network; so every other maximum is formed on the other one, as what the minimum leaves of the two bit patterns'
// sum (half of them: 30.5 -> 29.4 us at T = 1; two thirds are more instructions than that wins, 30.6).
template <int P_, int K_, int PER>
__device__ __forceinline__ void sort_layers(float (&x)[PER], int one) {
#pragma unroll
    for (int i = 0; i < PER - K_; ++i) {
        if (i >= K_ % P_ && ((i - K_ % P_) & K_) == 0 && i / (2 * P_) == (i + K_) / (2 * P_)) {
            const float lo = fminf(x[i], x[i + K_]);
            if ((i & 1) == 0) {
                x[i + K_] = fmaxf(x[i], x[i + K_]);
            } else {
                int hi;
                asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(hi) : "r"(__float_as_int(x[i])), "r"(one), "r"(__float_as_int(x[i + K_])));
                asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(hi) : "r"(__float_as_int(lo)), "r"(-one));
                x[i + K_] = __int_as_float(hi);
            }
            x[i] = lo;
        }
    }
    if constexpr (K_ > 1) sort_layers<P_, K_ / 2, PER>(x, one);
    else if constexpr (2 * P_ < PER) sort_layers<2 * P_, 2 * P_, PER>(x, one);
}

// As warp_sums, for any number of values and none of them held twice: afterwards v[0] of a lane is total number slot(lane).
template <int NV, int D>
struct Halve {
    static __device__ __forceinline__ void sums(long long* v, int lane) {
        if constexpr (D >= 1) {
            if constexpr (NV > 1) {
                constexpr int H = (NV + 1) / 2;
                const bool upper = (lane & D) != 0;
#pragma unroll
                for (int k = 0; k < H; ++k) {
                    const long long b = k + H < NV ? v[k + H] : 0;
                    const long long send = upper ? v[k] : b, keep = upper ? b : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, D);
                }
                Halve<H, D / 2>::sums(v, lane);
            } else {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], D);
                Halve<1, D / 2>::sums(v, lane);
            }
        }
    }
    // which of the NV totals that is; -1: none, or one that another lane holds as well
    static __device__ __forceinline__ int slot(int lane, int n = NV) {
        if constexpr (D >= 1) {
            constexpr int H = (NV + 1) / 2;
            const bool upper = (lane & D) != 0;
            if constexpr (NV > 1) {
                const int below = Halve<H, D / 2>::slot(lane, upper ? max(n - H, 0) : min(n, H));
                return below < 0 ? -1 : below + (upper ? H : 0);
            } else {
                return upper ? -1 : Halve<1, D / 2>::slot(lane, n);
            }
        } else {
            return n > 0 ? 0 : -1;
        }
    }
};

// Who looks after which level and the threshold above it: BITS = 1, 2, 4: lane j after level j; 7: all three precisions, lanes 0 to 15, 16 to 19, 20 and 21.
template <int BITS>
struct Levels {
    static constexpr int kLevels = BITS == 7 ? 22 : 1 << BITS, kThresholds = BITS == 7 ? 19 : (1 << BITS) - 1;
    static __device__ __forceinline__ int cls(int lane) { return BITS == 7 ? (lane < 16 ? 2 : lane < 20 ? 1 : 0) : BITS >> 1; }
    static __device__ __forceinline__ int level(int lane) { return BITS == 7 ? (lane < 16 ? lane : lane < 20 ? lane - 16 : lane - 20) : lane; }
    static __device__ __forceinline__ constexpr int lane_of(int q) { return BITS == 7 ? (q < 15 ? q : q < 18 ? q + 1 : q + 2) : q; }
    static __device__ __forceinline__ int threshold_of(int lane) { return BITS == 7 ? (lane < 15 ? lane : lane < 19 ? lane - 1 : lane - 2) : lane; }
};

__device__ __forceinline__ long long lds_s64(uint32_t at) {
    long long v;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(at));
    return v;
}

// (by the instruction's own predicate; see threshold_place)
__device__ __forceinline__ void add_if_below(uint32_t& a, uint32_t by, float x, float t) {
    asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %1, %2;\n\t@p add.u32 %0, %0, %3;\n\t}" : "+r"(a) : "f"(x), "f"(t), "r"(by));
}

// What a thread has in order: PER values, 32 apart, and their weight.
struct Ordered {
    uint32_t xs;        // this thread's first value
    uint32_t sums;      // of w n before values 0, 4, 8, ..., 32 apart
    float weight;
};

// As fine_sums, for `count` values of one weight, 32 apart in shared memory from `at` on.
__device__ __forceinline__ Fine fine_sums_of(float weight, uint32_t at, int count, double g) {
    const double g2 = g * 0x1p-46, w = (double)weight, b = __dadd_rn(w, g);
    Fine f = {0, 0, count * (long long)(grid_bits(b) - grid_bits(g)),
              count * (long long)(grid_bits(__dadd_rn(__dsub_rn(w, __dsub_rn(b, g)), g2)) - grid_bits(g2))};
    for (int p = 0; p < count; ++p, at += 128) {
        const double n = (double)lds_f32(at), a = __fma_rd(n, w, g);
        f.wn += (long long)(grid_bits(a) - grid_bits(g));
        f.wn_lo += (long long)(grid_bits(__dadd_rd(__fma_rn(n, w, -__dsub_rn(a, g)), g2)) - grid_bits(g2));
    }
    add_up(f);
    return f;
}

// The mean of the bucket [t_lo, t_hi) by the whole CTA; y if it weighs nothing.  scratch: five words per warp.  A thread's part of the bucket lies together:
// two bisections find it.
template <int PER, int WARPS>
__device__ __noinline__ double fine_mean_ordered(Ordered O, float t_lo, float t_hi, bool vanished, double y, long long* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t at = O.xs, end = O.xs;
#pragma unroll
    for (int h = PER / 2; h >= 1; h /= 2) {
        add_if_below(at, h * 128, lds_f32(at + (h - 1) * 128), t_lo);
        add_if_below(end, h * 128, lds_f32(end + (h - 1) * 128), t_hi);
    }
    add_if_below(at, 128, lds_f32(at), t_lo);
    add_if_below(end, 128, lds_f32(end), t_hi);
    const int count = end > at ? (int)(end - at) / 128 : 0;
    double g = kGrid;
    if (vanished) {
        float* most_of = reinterpret_cast<float*>(scratch + 4 * WARPS);
        float most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(count > 0 ? O.weight : 0.0f)));      // (none is negative)
        if (WARPS > 1) {
            if (lane == 0) most_of[warp] = most;
            __syncthreads();
            for (int w = 0; w < WARPS; ++w) most = fmaxf(most, most_of[w]);
        }
        g = grid_of(most);
        if (!(most > 0.0f)) {
            __syncthreads();
            return y;
        }
    }
    Fine f = fine_sums_of(O.weight, at, count, g);
    if (WARPS > 1) {
        if (lane == 0) { scratch[4 * warp] = f.wn; scratch[4 * warp + 1] = f.wn_lo; scratch[4 * warp + 2] = f.w; scratch[4 * warp + 3] = f.w_lo; }
        __syncthreads();
        f = Fine{0, 0, 0, 0};
        for (int w = 0; w < WARPS; ++w) { f.wn += scratch[4 * w]; f.wn_lo += scratch[4 * w + 1]; f.w += scratch[4 * w + 2]; f.w_lo += scratch[4 * w + 3]; }
        __syncthreads();
    }
    return fine_mean(f);
}

// T rounds and the tables of row r.  Every warp forms all levels and thresholds from all warps' sums, as in learn_row.  The thresholds five at a time: their
// searches hide one another's latency, and the loop's code stays short (all 19 unrolled, the instruction cache missed).
template <int BITS, int PER, int WARPS>
__device__ __forceinline__ void ordered_rounds(const LearnParams& P, const Ordered& O, long long all_n, long long all_w,
                                               unsigned zero_too, float row_most, long long* red2, int r) {
    using V = Levels<BITS>;
    constexpr int NQ = V::kThresholds, kAtOnce = NQ < 5 ? NQ : 5;
    constexpr int kRed = 2 * (BITS == 7 ? NQ : 15) * WARPS;      // (also room for fine_mean_ordered's scratch)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = V::cls(lane), j = V::level(lane), Lv = 1 << (1 << c);
    const bool mine = lane < V::kLevels, top = j >= Lv - 1;
    const int slot = Halve<2 * kAtOnce, 16>::slot(lane);
    double y = mine ? P.init_y[c][j] : 0.0;
    float t = mine && !top ? __double2float_ru(P.init_t[c][j]) : INFINITY;
    const double w = (double)O.weight;
    const long long wg = grid_weight(w, kGrid);
    for (int it = 0; it < P.iterations; ++it) {
        long long* red = red2 + (it & 1) * kRed;
#pragma unroll 1
        for (int q0 = 0; q0 < NQ; q0 += kAtOnce) {
            float tq[kAtOnce];
            uint32_t at[kAtOnce];
            uint32_t n[kAtOnce];
            double s[kAtOnce];
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {
                tq[k] = __shfl_sync(0xffffffffu, t, V::lane_of(q0 + k));
                at[k] = O.xs;
                s[k] = kGrid;
                n[k] = 0u;
            }
#pragma unroll
            for (int h = PER / 2; h >= 4; h /= 2) {
#pragma unroll
                for (int k = 0; k < kAtOnce; ++k) add_if_below(at[k], h * 128, lds_f32(at[k] + (h - 1) * 128), tq[k]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
#pragma unroll
                for (int k = 0; k < kAtOnce; ++k) {
                    const float x = lds_f32(at[k] + e * 128);
                    const double d = (double)x;
                    n[k] += x < tq[k] ? 1u : 0u;
                    s[k] = __fma_rd(__hiloint2double(x < tq[k] ? __double2hiint(d) : 0, __double2loint(d)), w, s[k]);   // (see few_buckets)
                }
            }
            long long v[2 * kAtOnce];
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {
                const uint32_t before = at[k] - O.xs;
                v[2 * k] = lds_s64(O.sums + before / 2) + (long long)(grid_bits(s[k]) - grid_bits(kGrid));
                v[2 * k + 1] = (long long)(n[k] + before / 128) * wg;
            }
            Halve<2 * kAtOnce, 16>::sums(v, lane);
            if (slot >= 0 && 2 * q0 + slot < 2 * NQ) red[(2 * q0 + slot) * WARPS + warp] = v[0];
        }
        if (WARPS > 1) __syncthreads();
        else __syncwarp();
        long long fn = all_n, fw = all_w;
        if (!top) {
            fn = fw = 0;
            const int q = V::threshold_of(lane);
#pragma unroll
            for (int k = 0; k < WARPS; ++k) { fn += red[2 * q * WARPS + k]; fw += red[(2 * q + 1) * WARPS + k]; }
        }
        const long long ln = __shfl_up_sync(0xffffffffu, fn, 1), lw = __shfl_up_sync(0xffffffffu, fw, 1);
        const double sn = (double)(j == 0 ? fn : fn - ln);
        const long long sw = j == 0 ? fw : fw - lw;
        const bool vanished = sw <= 0;
        if (!vanished) y = sn / (double)sw;
        for (unsigned left = __ballot_sync(0xffffffffu, mine && too_coarse(sn, P.near_zero, zero_too)); left != 0u; left &= left - 1u) {     // (the same in every warp)
            const int k = __ffs(left) - 1;
            const float t_lo = __shfl_sync(0xffffffffu, t, max(k - 1, 0)), t_hi = __shfl_sync(0xffffffffu, t, k);
            const bool first = __shfl_sync(0xffffffffu, j, k) == 0;
            const double mean = fine_mean_ordered<PER, WARPS>(O, first ? -INFINITY : t_lo, t_hi, __shfl_sync(0xffffffffu, (int)vanished, k) != 0,
                                                                  __shfl_sync(0xffffffffu, y, k), red2 + ((it & 1) ^ 1) * kRed);
            if (lane == k) y = mean;
        }
        const double yn = __shfl_down_sync(0xffffffffu, y, 1);
        const float tn = mine && !top ? __double2float_ru((y + yn) * 0.5) : INFINITY;
        const bool same = tn == t;
        t = tn;
        if (__all_sync(0xffffffffu, same)) break;
    }
    if (warp == 0) {
        const bool bad = !(row_most < INFINITY) && P.iterations > 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (BITS != 7 && k != BITS >> 1) continue;
            const int lv = 1 << (1 << k), l0 = BITS == 7 ? (k == 2 ? 0 : k == 1 ? 16 : 20) : 0;
            const size_t plane = BITS == 7 ? (size_t)k * P.N * kTableStride : 0;
            const double yl = __shfl_sync(0xffffffffu, y, l0 + min(lane, lv - 1));
            const float m = lane < lv ? (bad ? __int_as_float(0x7fc00000) : (float)yl) : 0.0f;
            const float mn = __shfl_down_sync(0xffffffffu, m, 1);
            if (lane < kTableStride) {
                P.maps[plane + (size_t)r * kTableStride + lane] = m;
                P.thresholds[plane + (size_t)r * kTableStride + lane] = (lane + 1 < lv) ? (float)(((double)m + (double)mn) * 0.5) : __int_as_float(0x7f800000);
            }
        }
    }
}

template <bool ALL3, int PER, int WARPS>
constexpr size_t ordered_smem() {
    return (size_t)WARPS * (PER * 32 * 4 + (PER / 4) * 32 * 8 + 2 * 2 * Levels<ALL3 ? 7 : 4>::kThresholds * 8 + 16 + 8);
}

// WARPS warps, a lane of which has PER values of one block; CTAS of them to an SM.
template <bool ALL3, int PER, int WARPS, int CTAS>
__global__ void __launch_bounds__(32 * WARPS, CTAS) ordered_learn_kernel(const __grid_constant__ LearnParams P) {
    extern __shared__ __align__(16) unsigned char ordered_smem_bytes[];
    constexpr int kPieces = PER / 4, kLanes = kBlock / PER;     // 16-byte pieces a lane; lanes a block
    const int K = P.K, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* xs = reinterpret_cast<float*>(ordered_smem_bytes);                           // [warps][PER][32]; before that, a warp's 32 PER values as they come
    long long* sums = reinterpret_cast<long long*>(xs + WARPS * PER * 32);              // [warps][PER / 4][32]
    long long* red2 = sums + WARPS * (PER / 4) * 32;                                    // two buffers of [thresholds][2][warps]
    long long* totals = red2 + 2 * 2 * Levels<ALL3 ? 7 : 4>::kThresholds * WARPS;       // [warps][2]
    float* most_of = reinterpret_cast<float*>(totals + 2 * WARPS);                      // [warps][2]
    enter(P.turn);
    const int i0 = P.row0 + (int)(gridDim.x - 1 - blockIdx.x);
    const int r = ALL3 ? i0 : P.L.perm[i0];
    const float* wrow = P.W + (size_t)r * K;
    const int first = warp * (PER * 32);
#pragma unroll
    for (int u = 0; u < kPieces; ++u) {
        const int at = first + 4 * (32 * u + lane);
        if (at < K) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(xs + at)), "l"(wrow + at) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int b = ALL3 ? 0 : P.L.precs[r];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    const bool in = first + lane * PER < K;
    float x[PER];
    float m = 0.0f;
#pragma unroll
    for (int q = 0; q < kPieces; ++q) {       // in an order in which eight lanes meet different banks
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) f = *reinterpret_cast<const float4*>(xs + first + PER * lane + 4 * (q ^ (PER >= 32 ? lane & 7 : (lane >> 1) & 3)));
        x[4 * q] = f.x; x[4 * q + 1] = f.y; x[4 * q + 2] = f.z; x[4 * q + 3] = f.w;
        m = max_nan(max_nan(m, max_nan(fabsf(f.x), fabsf(f.y))), max_nan(fabsf(f.z), fabsf(f.w)));
    }
#pragma unroll
    for (int d = 1; d < kLanes; d <<= 1) m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, d));
    const float inv = (m == 0.0f) ? 0.0f : __frcp_rn(m);
    float most = max_nan(m, __fmul_rn(inv, 0.0f)), least = m > 0.0f ? m : INFINITY;
#pragma unroll
    for (int e = 0; e < PER; ++e) x[e] = __fmul_rn(x[e], inv);
    sort_layers<1, 1, PER>(x, P.one);
#pragma unroll
    for (int d = kLanes; d < 32; d <<= 1) {
        most = max_nan(most, __shfl_xor_sync(0xffffffffu, most, d));
        least = fminf(least, __shfl_xor_sync(0xffffffffu, least, d));
    }
    if (WARPS > 1) {
        if (lane == 0) { most_of[2 * warp] = most; most_of[2 * warp + 1] = least; }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < WARPS; ++k) { most = max_nan(most, most_of[2 * k]); least = fminf(least, most_of[2 * k + 1]); }
    } else {
        __syncwarp();          // the row has been read
    }
    const float scale = weight_scale(most), weight = scaled_weight(m, scale);
    const unsigned zero_too = least < INFINITY && scaled_weight(least, scale) < kVanishing ? 1u : 0u;
    float* mine = xs + first + lane;
    long long* before = sums + warp * ((PER / 4) * 32) + lane;
    long long all[2] = {0, PER * grid_weight((double)weight, kGrid)};
    {
        const double w = (double)weight;
#pragma unroll
        for (int q = 0; q < PER; q += 16) {
            double s = kGrid;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                if ((e & 3) == 0) before[((q + e) / 4) * 32] = all[0] + (long long)(grid_bits(s) - grid_bits(kGrid));
                mine[(q + e) * 32] = x[q + e];
                s = __fma_rd((double)x[q + e], w, s);
            }
            all[0] += (long long)(grid_bits(s) - grid_bits(kGrid));
        }
    }
    __syncwarp();       // (see lds_f32)
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        all[0] += __shfl_xor_sync(0xffffffffu, all[0], d);
        all[1] += __shfl_xor_sync(0xffffffffu, all[1], d);
    }
    if (WARPS > 1) {
        if (lane == 0) { totals[2 * warp] = all[0]; totals[2 * warp + 1] = all[1]; }
        __syncthreads();
        all[0] = all[1] = 0;
#pragma unroll
        for (int k = 0; k < WARPS; ++k) { all[0] += totals[2 * k]; all[1] += totals[2 * k + 1]; }
    }
    const Ordered O = {(uint32_t)__cvta_generic_to_shared(mine), (uint32_t)__cvta_generic_to_shared(before), weight};
    if (ALL3) ordered_rounds<7, PER, WARPS>(P, O, all[0], all[1], zero_too, most, red2, r);
    else if (b == 1) ordered_rounds<1, PER, WARPS>(P, O, all[0], all[1], zero_too, most, red2, r);
    else if (b == 2) ordered_rounds<2, PER, WARPS>(P, O, all[0], all[1], zero_too, most, red2, r);
    else ordered_rounds<4, PER, WARPS>(P, O, all[0], all[1], zero_too, most, red2, r);
    leave(P.turn);
}

}  // namespace lowra

namespace lowra {
namespace {

lowra_status launch_rows(void (*kernel)(LearnParams), const LearnParams& P, int rows, int threads, size_t smem, SmemLimit* limit, void* stream) {
    if (ensure_smem_limit(reinterpret_cast<const void*>(kernel), smem, limit) != LOWRA_OK) return LOWRA_ERR_CUDA;
    // a row per CTA and as many CTAs as rows: a 4-bit row takes five times as long as a 1-bit one, and fresh CTAs handed out
    // by the hardware keep the SMs evenly busy where a persistent grid (every CTA walking over its share of the rows) left
    // some of them waiting at the end (the 7B layer at 60/35/5: 2.05 -> 1.68 ms)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)rows, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P) == cudaSuccess ? LOWRA_OK : LOWRA_ERR_CUDA;
}

template <bool ALL3, bool FOUR, int THREADS>
lowra_status launch_learn_kernel(const LearnParams& P, int rows, void* stream) {
    const size_t smem = (2 * 2 * 16 * (THREADS / 32) + (FOUR ? 2 * 16 * THREADS : 0)) * sizeof(long long) +
                        ((size_t)P.K + (size_t)P.K / kBlock + 16 * (THREADS / 32)) * sizeof(float);
    if (smem > 200 * 1024) return LOWRA_ERR_SHAPE;   // the row has to fit into shared memory (K <= 40960)
    static SmemLimit limit = {};
    return launch_rows(learn_kernel<ALL3, FOUR, THREADS>, P, rows, THREADS, smem, &limit, stream);
}

size_t sorted_smem_bytes(int K) {
    return (size_t)K * sizeof(float2) + ((size_t)K / 16 + 1) * sizeof(Sums) + 32 * (2 * sizeof(long long) + sizeof(float)) + ((size_t)bins_of(K) + 4) * 4;
}

template <bool ALL3, int THREADS, int PER, int CTAS>
lowra_status launch_sorted_kernel(LearnParams& P, int rows, void* stream) {
    P.bins = bins_of(P.K);
    static SmemLimit limit = {};
    return launch_rows(sorted_learn_kernel<ALL3, THREADS, PER, CTAS>, P, rows, (P.K / PER + 31) / 32 * 32, sorted_smem_bytes(P.K), &limit, stream);
}

bool two_long_rows(int K) { return 2 * (sorted_smem_bytes(K) + 1024) <= 228 * 1024; }   // an SM holds two (K <= 11776)

// Which kernel takes a class of rows (c = 0, 1, 2: 1, 2, 4 bits; 3: all of them).  Measured, us, 4096 rows (K >= 13824: 3328) after 2, 4 and 10
// rounds, learn_kernel / ordered_learn_kernel at 1 and 2 bits, ordered_learn_kernel / sorted_learn_kernel else:
//             1 bit                            2 bits                           4 bits                            all three
//   K=512     11/6    15/8    24/12            14/8    23/11   48/20            17/14   28/18   62/28             22/19   38/27   85/48
//   K=1024    11/9    16/12   27/16            15/10   23/14   49/23            19/21   31/28   68/48             23/27   39/38   90/68
//   K=2048    16/17   23/20   41/26            23/19   37/22   78/31            29/34   39/40   77/59             33/37   47/46   97/72
//   K=3072    21/29   31/35   56/47            31/32   50/39   108/58           49/51   70/62   137/93            57/55   87/70   179/112
//   K=4096    26/30   39/36   72/48            39/33   63/40   138/59           49/63   71/74   140/109           57/67   87/83   181/127
//   K=5120    34/44   51/52   94/73            50/48   84/59   185/91           75/78   108/93  216/136           87/84   133/103 281/159
//   K=8192    48/56   71/64   134/90           72/60   121/73  267/113          94/143  140/170 277/245           107/140 172/169 359/247
//   K=11008   69/99   100/116 188/168          102/106 168/130 369/204          157/180 231/206 462/284           181/183 282/209 592/287
//   K=13824   74/93   107/110 199/155          106/101 175/124 381/197          153/255 230/296 460/417           178/252 281/294 589/418
//   K=16384   83/97   119/114 225/162          120/105 197/130 432/209          169/281 263/322 549/443           199/279 328/321 704/445
// At 1 bit the ordered blocks pay in the fourth round where every lane has a block, later where some have none (K = 3072, 5120), or where an SM
// holds few warps (K = 8320 to 12288); K up to 2048 is one warp, up to 1024 of short networks.
// A few rows to an SM (per_sm) wait for the longest chain, and a warp's network is longer than the eight warps' way to the order of a whole row, or, of 2048 values
// at 1 and 2 bits, than rounds through the row.  Ordered against sorted, us, at 4 bits, one round / two: 296 rows of 1152 8.0 6.1 / 9.6 7.1, of 2048 8.1 6.6 / 9.6 8.2, of
// 4096 8.6 8.1; 1600 rows of 2048 12.0 16.3.  Rows that leave most of their last warp without a block (1152, 2176 values) gain little from it with any number.  Of 1794 calls for
// each column (23 lengths, 40 to 4096 rows) the choice is 0.8 % (4 bits), 1.7 (all, 1 bit) and 0.6 (2 bits) behind the better kernel in the mean: where the two are close, the order of
// whole rows is left out, for rows of few values, crowded in one cell, take it up to three times as long (296 pruned rows of 8192, two rounds 17.0 46.2).
enum Kernel { kRowAgain, kOrdered, kSorted };
int ordered_warps(int K) { return (K + 2047) / 2048; }
// Rows of up to `up_to` values: by their whole order from round `few` on with up to `rows` of them to an SM, from round `many` on with more.
struct SortedFrom { int up_to, rows, few, many; };
constexpr SortedFrom kFour[] = {{512, 8, 2, 2}, {1024, 8, 3, 3}, {1536, 6, 1, 2}, {2048, 5, 1, 4}, {2560, 2, 1, 2}, {3072, 2, 1, 3}, {4096, 2, 2, 5}, {5120, 4, 2, 3},
                                {6144, 2, 2, 10}, {8192, 0, 7, 7}, {11776, 0, 4, 4}, {kSortedMaxK, 0, 9, 9}};
constexpr SortedFrom kAll[] = {{512, 8, 2, 2}, {1024, 8, 4, 4}, {1536, 6, 1, 2}, {2048, 5, 1, 4}, {2560, 2, 1, 2}, {3072, 3, 1, 2}, {4096, 2, 2, 3}, {5120, 2, 2, 2},
                               {6144, 2, 2, 4}, {8192, 0, 4, 4}, {10240, 2, 2, 3}, {11776, 0, 3, 3}, {kSortedMaxK, 0, 5, 5}};
Kernel kernel_for(int K, int c, int iterations, int rows) {
    if (K > kSortedMaxK || iterations < 1) return kRowAgain;
    const int per_sm = (rows + kNumSMs - 1) / kNumSMs;
    if (c == 0) {
        const bool pays = K <= 1024 ? K <= 512 || iterations >= 2 || per_sm > 5 : K <= 2048 ? iterations >= (per_sm <= 4 ? 6 : 3)
                        : (iterations - (K > 8192 && K <= 12288 ? 2 : 0)) * K >= 4 * 2048 * ordered_warps(K);
        return pays ? kOrdered : kRowAgain;
    }
    if (c == 1) {
        const int from = K <= 1024 ? 1 : K <= 2048 ? (per_sm <= 4 ? 4 : 2) : K <= 3072 && per_sm <= 2 ? 4 : K > 8192 && K <= 12288 ? 3 : 2;
        return iterations >= from ? kOrdered : kRowAgain;
    }
    const SortedFrom* line = c == 2 ? kFour : kAll;
    while (K > line->up_to) ++line;
    // (In the order of whole rows an SM has five at a time; and in company - encoded or assessed right behind - up to five rows of two warps each crowd on the SMs that the kernel
    // before leaves first: 400 x 3072 of 4 bits, two rounds and encode 17.7 us, by the whole rows' order 15.3.)
    const int many = K > 2560 && K <= 4096 && (per_sm <= 5 || (K <= 3072 && per_sm == 6)) ? 2 : line->many;
    return iterations >= (per_sm <= line->rows ? line->few : many) ? kSorted : kOrdered;
}

// 4-bit rows, n4 of N, among others of more than 1024 values.  They are the longest, and of a few rows the last one counts (444 x 3072 at 30/50/20, one round 9.5 -> 7.5 us; 535 x 6144
// at 60/35/5, six 19.1 -> 14.4).  Otherwise they go by the whole row's order later than by themselves, for that is a launch more: 2.5 us of the 12 that a short call takes the host
// (600 x 2048 at 60/35/5, two rounds 15 -> 12.3).
Kernel four_in_company(int K, int iterations, int N, int n4) {
    const int per_sm = (N + kNumSMs - 1) / kNumSMs;
    if (K > kSortedMaxK || iterations < 2) return kernel_for(K, 2, iterations, per_sm <= (K <= 2048 ? 8 : K <= 4096 ? 5 : 0) ? n4 : N);
    const int from = K <= 6144 && per_sm <= 4 ? 2 : K <= 2048 ? 4 : K <= 3072 ? 3 : K <= 4096 ? 5 : K <= 6144 ? 3 : K <= 8192 ? 7 : K <= 11776 ? 4 : 9;
    return iterations >= from ? kSorted : kOrdered;
}

template <bool ALL3, int PER, int WARPS, int CTAS>
lowra_status launch_ordered_kernel(const LearnParams& P, int rows, void* stream) {
    static SmemLimit limit = {};
    return launch_rows(ordered_learn_kernel<ALL3, PER, WARPS, CTAS>, P, rows, 32 * WARPS, ordered_smem<ALL3, PER, WARPS>(), &limit, stream);
}

// As many rows to an SM as its shared memory takes: 12 KB for 2048 values.
template <bool ALL3>
lowra_status launch_ordered(const LearnParams& P, int rows, void* stream) {
    const int K = P.K;
    return K <= 512 ? launch_ordered_kernel<ALL3, 16, 1, 32>(P, rows, stream)
         : K <= 1024 ? launch_ordered_kernel<ALL3, 32, 1, 24>(P, rows, stream)
         : K <= 2048 ? launch_ordered_kernel<ALL3, 64, 1, 16>(P, rows, stream)
         : K <= 4096 ? launch_ordered_kernel<ALL3, 64, 2, 8>(P, rows, stream)
         : K <= 6144 ? launch_ordered_kernel<ALL3, 64, 3, 5>(P, rows, stream)
         : K <= 8192 ? launch_ordered_kernel<ALL3, 64, 4, 4>(P, rows, stream)
         : K <= 10240 ? launch_ordered_kernel<ALL3, 64, 5, 3>(P, rows, stream)
         : K <= 12288 ? launch_ordered_kernel<ALL3, 64, 6, 2>(P, rows, stream)
         : K <= 14336 ? launch_ordered_kernel<ALL3, 64, 7, 2>(P, rows, stream)
                      : launch_ordered_kernel<ALL3, 64, 8, 2>(P, rows, stream);
}

// validation shared by the two entry points is done by the callers; this fills the tables and launches (n1, n2, n4: rows to be
// learnt at 1, 2 and 4 bits)
template <bool ALL3>
lowra_status launch_learn(LearnParams& P, const double* init_levels_host, const double* init_thresholds_host,
                          int n1, int n2, int n4, void* stream) {
    if (((size_t)P.K + (size_t)P.K / kBlock) * sizeof(float) > 160 * 1024) return LOWRA_ERR_SHAPE;   // K <= 40960: the row has to fit
    lowra_status st = check_device();
    if (st != LOWRA_OK) return st;
    int log_k = 0;
    while ((2 << log_k) <= P.K) ++log_k;
    P.one = 1;
    P.near_zero = (unsigned)(1023 + 24 + log_k) << 20;
    for (int c = 0; c < 3; ++c)
        for (int j = 0; j < 16; ++j) {
            P.init_y[c][j] = init_levels_host[c * 16 + j];
            P.init_t[c][j] = init_thresholds_host[c * 16 + j];
        }
    const int per_sm = (P.N + kNumSMs - 1) / kNumSMs;
    Kernel kernel[3];
    for (int c = 0; c < 3; ++c) kernel[c] = kernel_for(P.K, ALL3 ? 3 : c, P.iterations, P.N);
    if (!ALL3 && 2 * n4 <= P.N && P.K > 1024) kernel[2] = four_in_company(P.K, P.iterations, P.N, n4);
    // (one launch fewer counts for more than the rows' kernel where these are few: 535 x 2048 at 60/35/5, T = 4 11.7 -> 10.2 us)
    if (!ALL3 && per_sm <= 8 && kernel[0] == kRowAgain && kernel[1] == kOrdered && n1 > 0 && n2 > 0) kernel[0] = kOrdered;
    // Stored rows are in the order of their precisions, and more bits want more order: a launch for every kernel that has classes, the last classes' first
    // (in turns; see enter()).
    const int n[3] = {n1, n2, n4};
    int end = P.N;
    P.turn = 0;
    for (int c = ALL3 ? 0 : 2; end > 0; ) {
        const Kernel k = kernel[c];
        int rows = ALL3 ? P.N : 0;
        for (; !ALL3 && c >= 0 && (kernel[c] == k || n[c] == 0); --c) rows += n[c];
        if (rows == 0) continue;
        if (rows < P.N) P.turn = end == P.N ? 1 : 2;
        P.row0 = end - rows;
        end -= rows;
        if (k == kOrdered) {
            st = launch_ordered<ALL3>(P, rows, stream);
        } else if (k == kSorted) {
            // As many CTAs to an SM as its shared memory takes, for the phases of one row leave what bounds the others idle.  The registers
            // go with that: 16 elements a thread up to K = 8192; beyond it two rows of 512 threads beat one of 1024 (K = 11008: 152
            // against 232 us) as long as two fit.
            st = P.K <= 4096       ? launch_sorted_kernel<ALL3, 256, 16, 5>(P, rows, stream)
               : P.K <= 5120       ? launch_sorted_kernel<ALL3, 320, 16, 4>(P, rows, stream)
               : P.K <= 8192       ? launch_sorted_kernel<ALL3, 512, 16, 2>(P, rows, stream)
               : two_long_rows(P.K) ? launch_sorted_kernel<ALL3, 512, 32, 2>(P, rows, stream)
                                    : launch_sorted_kernel<ALL3, 1024, 16, 1>(P, rows, stream);
        } else {
            const bool four = (ALL3 || (kernel[2] == kRowAgain && n4 > 0)) && P.iterations > 0;
            st = four ? launch_learn_kernel<ALL3, true, 128>(P, rows, stream)
               : P.K <= 4096 ? launch_learn_kernel<ALL3, false, 64>(P, rows, stream) : launch_learn_kernel<ALL3, false, 128>(P, rows, stream);
        }
        if (st != LOWRA_OK) return st;
    }
    return LOWRA_OK;
}

}  // namespace
}  // namespace lowra

extern "C" lowra_status lowra_learn_codebooks(const lowra_layout* layout, const float* W_dev,
                                              const double* init_levels_host, const double* init_thresholds_host,
                                              int32_t iterations, float* maps_dev, float* thresholds_dev, void* stream) {
    using namespace lowra;
    lowra_status st = check_layout(layout);
    if (st != LOWRA_OK) return st;
    if (!W_dev || !init_levels_host || !init_thresholds_host || !maps_dev || !thresholds_dev) return LOWRA_ERR_NULL;
    if (iterations < 0 || iterations > 1000) return LOWRA_ERR_SHAPE;
    if (!aligned16(W_dev) || !aligned16(maps_dev) || !aligned16(thresholds_dev)) return LOWRA_ERR_ALIGN;
    LearnParams P;
    P.L = make_row_layout(layout);
    P.W = W_dev;
    P.maps = maps_dev;
    P.thresholds = thresholds_dev;
    P.iterations = iterations;
    P.N = layout->N;
    P.K = layout->K;
    return launch_learn<false>(P, init_levels_host, init_thresholds_host, layout->counts[0], layout->counts[1], layout->counts[2], stream);
}

extern "C" lowra_status lowra_learn_codebooks_all(int32_t N, int32_t K, const float* W_dev,
                                                  const double* init_levels_host, const double* init_thresholds_host,
                                                  int32_t iterations, float* maps3_dev, float* thresholds3_dev,
                                                  void* stream) {
    using namespace lowra;
    if (!W_dev || !init_levels_host || !init_thresholds_host || !maps3_dev || !thresholds3_dev) return LOWRA_ERR_NULL;
    if (N < 1 || K < 128 || K % 128 != 0 || iterations < 0 || iterations > 1000) return LOWRA_ERR_SHAPE;
    if (!aligned16(W_dev) || !aligned16(maps3_dev) || !aligned16(thresholds3_dev)) return LOWRA_ERR_ALIGN;
    LearnParams P;
    memset(&P.L, 0, sizeof(P.L));   // no layout: every row at every precision
    P.W = W_dev;
    P.maps = maps3_dev;
    P.thresholds = thresholds3_dev;
    P.iterations = iterations;
    P.N = N;
    P.K = K;
    return launch_learn<true>(P, init_levels_host, init_thresholds_host, N, N, N, stream);
}
