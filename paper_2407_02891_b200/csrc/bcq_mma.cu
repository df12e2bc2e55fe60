// Small-batch BCQ product (2 <= B <= 16 columns, tiled layout) for sm_100a: every weight tile is
// read from HBM once and serves all columns.
//
//   Y[b] = sum_g ( sum_i alpha_i (B_i X[b])_g + z (sum X[b])_g )          (Eq. bcw + Eq. fuse_step3)
//
// With several columns the product is a (thin) dense contraction, so the sums go through the tensor cores: mma.sp
// m16n8k32, fp16 operands, fp32 accumulators, operands in registers, the weight bits as sparsity metadata (see
// bcq_mma_core.cuh).  One MMA = 16 weight rows -- two row units, i.e. two tiles of the same window -- x 16 weights x 8
// columns of X (9 .. 16 columns: a second MMA with the same metadata).  The 128 weights of a scaling unit
// are 8 MMAs per plane; their sum is scaled in fp32 by the row's alpha.
// (The shared-memory-operand tensor path, tcgen05, would need the expanded weights -- 16 times the packed bytes --
// written to shared or tensor memory first; with at most 16 columns that costs more than the MMAs themselves.)
//
// A block owns a range of row units (in pairs) and a range of windows of K.  Its (pair, window) jobs, pair after pair,
// are dealt to 16 warps in contiguous runs of equal length, so that no warp idles whatever the number of pairs; a pair
// that two or more warps share is put together through shared memory in a fixed order.  All of the block's x is staged
// before the first job.  (A decomposition whose x does not fit runs in phases of as many windows as do, whole pairs per
// warp, sums kept in shared memory between phases.)  Every warp keeps its own ring of slots (one slot = one tile pair =
// one contiguous piece of memory) filled with bulk async copies.
//
// Split K: as in the batch-1 kernel, every output owns one 64-bit word of the workspace, to which a split adds its
// fixed-point sum and an arrival; whoever completes a word stores y and clears the word.  A sum that the word cannot hold
// (infinite, not a number, very large) arrives as such, and the warp that completes the word computes that output over all of K.
// The result does not depend on the order of arrival.  (fp32 sums per split, added up by the last to arrive, take a fence and
// two more round trips to L2, and leave the adding to the last block: 8192 x 8192, 8 columns, 4 splits 21.6 us against 19.5;
// 2048 x 8192, 16 splits 14.6 against 6.9.)  All waits are bounded.
//
// Bound: dispatch of the tensor instruction (9 cycles) and of the half-rate instructions around it (2.5 per MMA: metadata,
// signs of x, half-words of planes): 16 cycles per MMA and SM sub-partition at up to 8 columns, 13 at 16; then the fixed
// 4 - 5 us of a launch (x, split-K atomics).  28672 x 8192, q = 3, groups of 128: 71 - 79 us at 8 columns and 103 - 113 at
// 16 with bits expanded to +-alpha by two instructions per register and whole pairs per warp; 47 and 80 us so.
#include "bcq_mma_core.cuh"

namespace bcq {

constexpr int kMmaThreads = kMmaWarps * 32;
constexpr int kMmaSmemBytes = 232448;    // 227 KB: the per-block opt-in maximum
constexpr int kMmaFixedBytes = 1024;     // barriers and flags
constexpr int kMmaMaxSlotsPerWarp = 4;

static_assert(8 * kMmaWarps * kMmaMaxSlotsPerWarp + 4 * (1 + kMmaWarps) <= kMmaFixedBytes, "barrier area");

// Split-K words: arrivals in the top bits, below them the arrivals whose sum is not in the word, then the sum of the
// biased fixed-point partial sums.  The widths follow from the number of arrivals.  The unit is 2^-36, so that
// even 31 roundings to it are at most 2^-32, a 128th of half a step of fp16's subnormal numbers; what is left is the
// limit of a partial sum: 2^19 for 4 splits, 2^16 for 8, 2^15 for up to 15, 2^13 for 16, 2^12 for up to 31.
constexpr int kMmaUnit = 36;
struct SplitFormat {
    int count_shift, odd_shift;
    long long bias;
    float limit;   // a power of two; sums whose magnitude is not below it are not in the word
    int arrivals;
};
inline SplitFormat split_format(int arrivals)
{
    int cb = 1, lb = 0;
    while ((1 << cb) <= arrivals) ++cb;
    while ((1 << lb) < arrivals) ++lb;
    SplitFormat f;
    f.count_shift = 64 - cb, f.odd_shift = 64 - 2 * cb;
    f.bias = 1ll << (f.odd_shift - lb - 1);
    f.limit = float(double(f.bias) / double(1ll << kMmaUnit));
    f.arrivals = arrivals;
    return f;
}
__device__ __forceinline__ unsigned long long split_encode(float v, const SplitFormat &f)
{
    const bool in = fabsf(v) < f.limit;
    const long long fixed = __float2ll_rn(in ? v * float(1ll << kMmaUnit) : 0.f);   // the product is exact
    return (1ull << f.count_shift) + (in ? 0ull : 1ull << f.odd_shift) + (unsigned long long)(fixed + f.bias);
}
__device__ __forceinline__ bool split_complete(unsigned long long before, const SplitFormat &f) { return int(before >> f.count_shift) == f.arrivals - 1; }
__device__ __forceinline__ bool split_odd(unsigned long long w, const SplitFormat &f) { return ((w & ((1ull << f.count_shift) - 1)) >> f.odd_shift) != 0; }
__device__ __forceinline__ __half split_decode(unsigned long long w, const SplitFormat &f)
{
    const long long s = (long long)(w & ((1ull << f.odd_shift) - 1)) - (long long)f.arrivals * f.bias;
    return __double2half(double(s) * (1.0 / double(1ll << kMmaUnit)));
}

__device__ int g_mma_status = 0;  // 0, or the code of the wait that ran out (sticky until taken)

struct MmaParams {
    const uint8_t *tiles;
    const uint16_t *alpha;   // per-row scales only: [u][i][r]
    const uint16_t *z;       // per-row scales only: [u][r]
    const __half *X;         // [B][K]
    __half *Y;               // [B][N]
    unsigned long long *accum;   // [B][N] split-K words, all zero between launches; k_splits > 1 only
    int N, K, B;
    int u_base, u_rem, w_base, w_rem;   // even partitions: part r starts at r * base + min(r, rem), base + (r < rem) items
    int split;               // k_splits > 1
    int phase_windows;       // windows whose x is staged at a time
    int depth;               // ring slots per warp
    int x_at, sum_at, ring_at;   // shared memory: constants and x; sums between phases; rings
    uint32_t ones;           // (1, 1) in fp16: a value known to the compiler would be put into registers again at every use
    SplitFormat fmt;
};

enum { kMmaWaitFull = 11, kMmaWaitDrain = 14 };

struct MmaOnes {   // every non-zero is 1
    uint32_t v[4];
    __device__ const uint32_t (&operator()(int, int) const)[4] { return v; }
};

// Outputs whose sum did not fit their split-K words: one warp computes the pair of row units at ua (units from u1 on belong to
// other blocks) over all of K, segment by segment as the kernel does, the segments in fp64, and stores this lane's outputs in
// `which` (bit e: row unit ua + (e / 2) % 2, column as in the kernel).  The warp's ring, free by then, holds eight columns of a
// segment of x.  Ends early once all of the outputs are NaN: a column of NaN costs 3 us at 8192 x 8192, 8 columns (1.8 ms with a
// scalar product per output).
template <int Q, bool GROUPED, bool WIDE>
__device__ __forceinline__ void mma_whole_pair(const MmaParams &p, int ua, int u1, unsigned which)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int T = Q * 512 + (GROUPED ? Q * 64 + 64 : 0), HALVES = WIDE ? 2 : 1, NA = 4 * HALVES;
    const int lane = threadIdx.x & 31, m = lane >> 2, t = lane & 3, U = p.N / kUnitRows;
    const int next_unit = ua + 1 < u1 ? 1 : 0;   // (an odd block's last unit stands in for the one it does not have)
    const int half_lo = m * 16 + 2 * ((2 * t - m) & 7), half_hi = m * 16 + 2 * ((2 * t + 1 - m) & 7);
    unsigned char *buf = smem + p.ring_at + int(threadIdx.x >> 5) * p.depth * 2 * T;
    const MmaOnes unit = {{p.ones, p.ones, p.ones, p.ones}};
    double acc[NA];
#pragma unroll
    for (int e = 0; e < NA; ++e) acc[e] = 0.0;
    for (int seg = 0; seg < p.K / 128; ++seg) {
        const unsigned char *tile = p.tiles + (size_t(seg >> 2) * U + ua) * T;
        uint4 raw[HALVES][4];   // lane = (column of eight, word): 32 activations
#pragma unroll
        for (int half = 0; half < HALVES; ++half) {
            const int b = 8 * half + m;
            const uint4 *src = reinterpret_cast<const uint4 *>(p.X + size_t(b) * p.K + 128 * size_t(seg) + 32 * t);
#pragma unroll
            for (int j = 0; j < 4; ++j) raw[half][j] = b < p.B ? __ldg(src + j) : make_uint4(0u, 0u, 0u, 0u);
        }
        uint32_t bits[Q][2];
        __half scale[2][Q + 1];
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned char *at = tile + i * 512 + 128 * (seg & 3) + (h ? half_hi : half_lo);
                bits[i][h] = __byte_perm(__ldg(reinterpret_cast<const uint16_t *>(at)), __ldg(reinterpret_cast<const uint16_t *>(at + next_unit * T)), 0x5410u);
            }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i <= Q; ++i) {
                const int u = ua + h * next_unit;
                const uint16_t *at;
                if constexpr (GROUPED)
                    at = reinterpret_cast<const uint16_t *>(tile + h * next_unit * T + Q * 512) + (8 * (seg & 3) + m) * (Q + 1) + i;
                else
                    at = i < Q ? p.alpha + (size_t(u) * Q + i) * kUnitRows + m : p.z + size_t(u) * kUnitRows + m;
                scale[h][i] = __ushort_as_half(__ldg(at));
            }
#pragma unroll
        for (int half = 0; half < HALVES; ++half) {
            __syncwarp();   // the staged columns have been read
            float x = stage_word(raw[half], buf + m * kXSegBytes, t);
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            const float sums[2] = {__shfl_sync(0xffffffffu, x, 8 * t), __shfl_sync(0xffffffffu, x, 8 * t + 4)};   // of columns 2 t, 2 t + 1
            __syncwarp();
            float c[Q][4], none[1][4];
            segment_sums<Q, false, true>(bits, buf + m * kXSegBytes + t * 16, buf, unit, c, none);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                double v = double(__half2float(scale[e >> 1][Q])) * double(sums[e & 1]);
#pragma unroll
                for (int i = 0; i < Q; ++i) v = fma(double(__half2float(scale[e >> 1][i])), double(c[i][e]), v);
                acc[4 * half + e] += v;
            }
        }
        bool open = false;
#pragma unroll
        for (int e = 0; e < NA; ++e) open = open || (((which >> e) & 1u) && acc[e] == acc[e]);
        if (!__any_sync(0xffffffffu, open)) break;
    }
#pragma unroll
    for (int e = 0; e < NA; ++e)
        if ((which >> e) & 1u)
            p.Y[size_t(8 * (e >> 2) + 2 * t + (e & 1)) * p.N + size_t(ua + ((e >> 1) & 1)) * kUnitRows + m] = __double2half(acc[e]);
    __syncwarp();
}

// An output that is to be computed over all of K keeps the mark of the warp that completed its split-K word in it until the end
// of the kernel, which has no registers to spare for a list, nor for what is found again here: the block's row units and
// windows and the warp's pairs, as in the kernel.
__device__ __forceinline__ unsigned mma_mark() { return blockIdx.y * kMmaWarps + (threadIdx.x >> 5) + 1; }
template <int Q, bool GROUPED, bool WIDE>
__device__ __noinline__ void mma_marked_outputs(const MmaParams &p)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = lane >> 2, t = lane & 3;
    const int rbi = blockIdx.x, u0 = rbi * p.u_base + min(rbi, p.u_rem), u1 = u0 + p.u_base + (rbi < p.u_rem ? 1 : 0);
    const int nwin = p.w_base + (int(blockIdx.y) < p.w_rem ? 1 : 0), P = (u1 - u0 + 1) >> 1;
    const bool whole = nwin <= p.phase_windows;
    const int run = (warp & 3) * (kMmaWarps / 4) + (warp >> 2), j0 = run * P * nwin / kMmaWarps, j1 = (run + 1) * P * nwin / kMmaWarps;
    const int last = whole ? (j1 - 1) / nwin : P - 1;
    for (int pair = whole ? j0 / nwin : warp; pair <= last; pair += whole ? 1 : kMmaWarps) {
        const int ua = u0 + 2 * pair;
        unsigned which = 0;
        for (int e = 0; e < (WIDE ? 8 : 4); ++e) {
            const int h = (e >> 1) & 1, b = 8 * (e >> 2) + 2 * t + (e & 1);
            unsigned long long *word = p.accum + size_t(b) * p.N + size_t(ua + h) * kUnitRows + m;
            if (ua + h < u1 && b < p.B && *word == mma_mark()) which |= 1u << e, *word = 0;
        }
        if (__any_sync(0xffffffffu, which != 0)) mma_whole_pair<Q, GROUPED, WIDE>(p, ua, u1, which);
    }
}

// Q planes; GROUPED: scales per (row, group of 128) inside the tiles, else per row in arrays;
// WIDE: 9..16 columns (two MMAs per step), else at most 8.
template <int Q, bool GROUPED, bool WIDE>
__global__ void __launch_bounds__(kMmaThreads, 1) mma_gemm_kernel(const __grid_constant__ MmaParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int T = Q * 512 + (GROUPED ? Q * 64 + 64 : 0);   // bytes of one tile
    constexpr int kSlotBytes = 2 * T;
    constexpr int BR = WIDE ? 16 : 8;
    constexpr int NA = WIDE ? 8 : 4;                           // accumulators per lane and pair
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int rbi = blockIdx.x, ks = blockIdx.y, U = p.N / kUnitRows;
    const int u0 = rbi * p.u_base + min(rbi, p.u_rem), w0 = ks * p.w_base + min(ks, p.w_rem);
    const int V = p.u_base + (rbi < p.u_rem ? 1 : 0), nwin = p.w_base + (ks < p.w_rem ? 1 : 0);
    const int u1 = u0 + V, P = (V + 1) >> 1;   // row units and unit pairs of this block
    const bool whole = nwin <= p.phase_windows;   // all of x at once
    const int D = p.depth;

    // ---- shared memory: [barriers | shared pairs' sums | group sums of x | x operands | sums between phases | rings] ----
    unsigned char *part = smem + kMmaFixedBytes;                               // [run][lane][NA] fp32
    float *xconst = reinterpret_cast<float *>(smem + p.x_at);                  // [window][segment][column]: sum of x
    unsigned char *xs = smem + p.x_at + size_t(min(nwin, p.phase_windows)) * 4 * BR * sizeof(float);   // [window][column]
    unsigned char *between = smem + p.sum_at;                                  // [pair][lane][NA] fp32
    unsigned char *ring = smem + p.ring_at + warp * D * kSlotBytes;
    const uint32_t full0 = smem_u32(smem) + 8 * kMmaMaxSlotsPerWarp * warp;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + 8 * kMmaWarps * kMmaMaxSlotsPerWarp);

    // ---- jobs of this warp: (pair, window) from (pair0, win0) on -----------------------------------------------
    // Run r belongs to warp (r mod 4) * 4 + r / 4: the runs that get one job more than the others (or the only jobs, where
    // there are fewer than warps) come at regular distances and would otherwise share a sub-partition's tensor pipe.
    const int run = (warp & 3) * (kMmaWarps / 4) + (warp >> 2);
    int total, pair0, win0 = 0;
    if (whole) {
        const int jobs = P * nwin, j0 = run * jobs / kMmaWarps;
        total = (run + 1) * jobs / kMmaWarps - j0, pair0 = j0 / nwin, win0 = j0 - pair0 * nwin;
    } else {
        total = warp < P ? (P - warp + kMmaWarps - 1) / kMmaWarps * nwin : 0;
        pair0 = warp;
    }
    struct Cursor {
        int pair, win, lo, hi;   // lo .. hi - 1: the windows of the current phase
    };
    Cursor next = {pair0, win0, 0, whole ? nwin : p.phase_windows};
    auto advance = [&](Cursor &c) {
        if (++c.win == c.hi) {
            c.win = c.lo;
            c.pair += whole ? 1 : kMmaWarps;
            if (!whole && c.pair >= P) {
                c.pair = warp, c.lo = c.hi, c.hi = min(c.hi + p.phase_windows, nwin);
                c.win = c.lo;
            }
        }
    };
    int issued = 0, consumed = 0;
    auto issue_next = [&](int slot) {   // lane 0 only
        if (issued < total) {
            const int ua = u0 + 2 * next.pair;
            const size_t tile = size_t(w0 + next.win) * U + ua;
            const uint32_t bytes = (ua + 1 < u1) ? kSlotBytes : T;   // the last pair of an odd block is one tile
            mbar_expect_tx(full0 + 8 * slot, bytes);
            bulk_g2s(smem_u32(ring + slot * kSlotBytes), p.tiles + tile * T, bytes, full0 + 8 * slot);
            ++issued;
            advance(next);
        }
    };
    if (lane == 0) {
        for (int s = 0; s < D; ++s) mbar_init(full0 + 8 * s, 1);
        if (tid == 0) *abort_flag = 0;
        abort_flag[1 + warp] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // weights are constants and may be fetched before the previous kernel in the stream has finished
        for (int s = 0; s < D; ++s) issue_next(s);
    }
    // Programmatic dependent launch, as in the batch-1 kernel.  X, the split-K words and Y wait for the predecessor.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int m = lane >> 2, t = lane & 3;
    const MmaOnes unit = {{p.ones, p.ones, p.ones, p.ones}};
    // chunk pairs 2 t and 2 t + 1 of row m's segment: the tile stores the segment's 16 chunks rotated by 2 m, so they sit
    // at half-words (2 t - m) mod 8 and (2 t + 1 - m) mod 8 of the row's 16 bytes
    const int half_lo = m * 16 + 2 * ((2 * t - m) & 7), half_hi = m * 16 + 2 * ((2 * t + 1 - m) & 7);
    // columns beyond B read a staged column (their accumulators are not stored)
    const unsigned char *xa0 = xs + (m < p.B ? m : 0) * kXColBytes + t * 16;
    const unsigned char *xb0 = xs + (m + 8 < p.B ? m + 8 : 0) * kXColBytes + t * 16;

    float acc[NA];
#pragma unroll
    for (int e = 0; e < NA; ++e) acc[e] = 0.f;

    // outputs of one finished pair: rows m of both units, columns 2 t, 2 t + 1 (and 8 + those)
    auto emit = [&](int pair) {
        const int ua = u0 + 2 * pair;
        unsigned long long before[NA], mine[NA];
#pragma unroll
        for (int e = 0; e < NA; ++e) {   // all adds on their way before the first answer is looked at
            const int h = (e >> 1) & 1, b = 8 * (e >> 2) + 2 * t + (e & 1);
            const size_t at = size_t(b) * p.N + size_t(ua + h) * kUnitRows + m;
            before[e] = mine[e] = 0;
            if (ua + h < u1 && b < p.B) {
                if (p.split) {
                    mine[e] = split_encode(acc[e], p.fmt);
                    before[e] = atomicAdd(p.accum + at, mine[e]);
                } else {
                    p.Y[at] = __float2half_rn(acc[e]);
                }
            }
        }
        if (p.split) {
#pragma unroll
            for (int e = 0; e < NA; ++e) {
                const int h = (e >> 1) & 1, b = 8 * (e >> 2) + 2 * t + (e & 1);
                const size_t at = size_t(b) * p.N + size_t(ua + h) * kUnitRows + m;
                if (ua + h < u1 && b < p.B && split_complete(before[e], p.fmt)) {
                    const bool odd = split_odd(before[e] + mine[e], p.fmt);
                    if (!odd) p.Y[at] = split_decode(before[e] + mine[e], p.fmt);
                    p.accum[at] = odd ? mma_mark() : 0;
                    if (odd) abort_flag[1 + warp] = 1;   // some of the warp's outputs carry its mark
                }
            }
        }
    };

    bool alive = true;
    int slot = 0, fill = 0, done = 0;
    Cursor cur = {pair0, win0, 0, whole ? nwin : p.phase_windows};
    bool began = win0 == 0;   // this warp has the current pair from its first window on
    for (int lo = 0; lo < nwin; lo += p.phase_windows) {
        const int nw = min(p.phase_windows, nwin - lo);
        // ---- stage x of the windows lo .. lo + nw - 1: four threads per (window, column, segment) ----------------
        if (lo > 0) __syncthreads();   // nobody reads the previous windows' x any more
#pragma unroll 2
        for (int base = warp * 32; base < nw * p.B * 16; base += kMmaThreads) {
            const int task = min(base + lane, nw * p.B * 16 - 1);   // (the count is a multiple of 16)
            const int st = task & 3, sg = (task >> 2) & 3, wb = task >> 4, w = wb / p.B, b = wb - w * p.B;
            const uint4 *src = reinterpret_cast<const uint4 *>(p.X + size_t(b) * p.K + size_t(w0 + lo + w) * kWindow + 128 * sg + 32 * st);
            const uint4 raw[4] = {__ldg(src), __ldg(src + 1), __ldg(src + 2), __ldg(src + 3)};
            float s = stage_word(raw, xs + size_t(w * p.B + b) * kXColBytes + sg * kXSegBytes, st);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (st == 0) xconst[(w * 4 + sg) * BR + b] = s;
        }
        __syncthreads();

        while (done < total && cur.lo == lo) {
            if (alive) alive = __all_sync(0xffffffffu, mbar_wait(full0 + 8 * slot, fill & 1, abort_flag, kMmaWaitFull, &g_mma_status));
            if (!alive) break;
            ++consumed;
            if (done > 0 && cur.win == cur.lo) {   // a new pair (this phase)
#pragma unroll
                for (int e = 0; e < NA; ++e) acc[e] = 0.f;
                began = true;
            }
            if (lo > 0 && cur.win == lo) {
                const float *from = reinterpret_cast<const float *>(between) + (cur.pair * 32 + lane) * NA;
#pragma unroll
                for (int e = 0; e < NA; ++e) acc[e] = from[e];
            }
            const unsigned char *tile = ring + slot * kSlotBytes;
            const int wl = cur.win - lo;
            const unsigned char *xa = xa0 + size_t(wl * p.B) * kXColBytes, *xb = xb0 + size_t(wl * p.B) * kXColBytes;
            const float *xc = xconst + wl * 4 * BR + 2 * t;
            // (an odd block's last pair has one tile: what the slot holds behind it is read, but rows m + 8 are not stored)
            [[maybe_unused]] float row_scale[2][Q + 1];
            if constexpr (!GROUPED) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int u = min(u0 + 2 * cur.pair + h, u1 - 1);
#pragma unroll
                    for (int i = 0; i < Q; ++i)
                        row_scale[h][i] = __half2float(__ushort_as_half(__ldg(p.alpha + (size_t(u) * Q + i) * kUnitRows + m)));
                    row_scale[h][Q] = __half2float(__ushort_as_half(__ldg(p.z + size_t(u) * kUnitRows + m)));
                }
            }
            float c[Q][4], ch[WIDE ? Q : 1][4];
            float2 k0 = make_float2(0.f, 0.f), k1 = k0;   // sums of x of columns 2t, 2t + 1; of 8 + those
            if constexpr (!GROUPED) {
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float2 a = *reinterpret_cast<const float2 *>(xc + g * BR);
                    k0.x += a.x, k0.y += a.y;
                    if constexpr (WIDE) {
                        const float2 b = *reinterpret_cast<const float2 *>(xc + g * BR + 8);
                        k1.x += b.x, k1.y += b.y;
                    }
                }
            }
            // acc += scale times the sums of plane i, or z times the sums of x, for the rows of unit h
            auto scaled = [&](int h, float a, const float (&lo4)[4], const float (&hi4)[4]) {
                acc[2 * h] = fmaf(a, lo4[2 * h], acc[2 * h]);
                acc[2 * h + 1] = fmaf(a, lo4[2 * h + 1], acc[2 * h + 1]);
                if constexpr (WIDE) {
                    acc[4 + 2 * h] = fmaf(a, hi4[2 * h], acc[4 + 2 * h]);
                    acc[5 + 2 * h] = fmaf(a, hi4[2 * h + 1], acc[5 + 2 * h]);
                }
            };
            if constexpr (!GROUPED) {
#pragma unroll
                for (int i = 0; i < Q; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        c[i][e] = 0.f;
                        if constexpr (WIDE) ch[i][e] = 0.f;
                    }
            }
            // (wide, one copy of the body: four are more than the instruction caches hold for 16 warps at different places,
            // 84.5 -> 87.8 us at 28672 x 8192; up to 8 columns four copies fit and save 2 %)
#pragma unroll (WIDE ? 1 : 4)
            for (int g = 0; g < 4; ++g) {
                uint32_t bits[Q][2];
#pragma unroll
                for (int i = 0; i < Q; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const unsigned char *base = tile + i * 512 + g * 128 + (h ? half_hi : half_lo);
                        const uint32_t a = *reinterpret_cast<const uint16_t *>(base), b = *reinterpret_cast<const uint16_t *>(base + T);
                        bits[i][h] = __byte_perm(a, b, 0x5410u);
                    }
                if constexpr (GROUPED) {
                    k0 = *reinterpret_cast<const float2 *>(xc + g * BR);
                    if constexpr (WIDE) k1 = *reinterpret_cast<const float2 *>(xc + g * BR + 8);
                    segment_sums<Q, WIDE, true>(bits, xa + g * kXSegBytes, xb + g * kXSegBytes, unit, c, ch);
                    // the unit's scales: alpha_i times the signed sums, z times the sum of x
                    const float zx[4] = {k0.x, k0.y, k0.x, k0.y}, zxh[4] = {k1.x, k1.y, k1.x, k1.y};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const unsigned char *sp = tile + h * T + Q * 512 + (8 * g + m) * (2 * (Q + 1));
                        __align__(8) __half sc[Q + 1];
                        if constexpr (Q == 3) {
                            *reinterpret_cast<uint2 *>(sc) = *reinterpret_cast<const uint2 *>(sp);
                        } else if constexpr (Q == 1) {
                            *reinterpret_cast<uint32_t *>(sc) = *reinterpret_cast<const uint32_t *>(sp);
                        } else {
#pragma unroll
                            for (int i = 0; i <= Q; ++i) sc[i] = reinterpret_cast<const __half *>(sp)[i];
                        }
                        scaled(h, __half2float(sc[Q]), zx, zxh);
#pragma unroll
                        for (int i = 0; i < Q; ++i) scaled(h, __half2float(sc[i]), c[i], ch[WIDE ? i : 0]);
                    }
                } else {
                    segment_sums<Q, WIDE, false>(bits, xa + g * kXSegBytes, xb + g * kXSegBytes, unit, c, ch);
                }
            }
            if constexpr (!GROUPED) {
                const float zx[4] = {k0.x, k0.y, k0.x, k0.y}, zxh[4] = {k1.x, k1.y, k1.x, k1.y};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    scaled(h, row_scale[h][Q], zx, zxh);
#pragma unroll
                    for (int i = 0; i < Q; ++i) scaled(h, row_scale[h][i], c[i], ch[WIDE ? i : 0]);
                }
            }
            // the slot has been read: order those reads before the next copy into it, then refill it
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) issue_next(slot);
            if (++slot == D) {
                slot = 0;
                ++fill;
            }
            ++done;
            if (cur.win == nwin - 1) {
                if (began) {
                    emit(cur.pair);
                } else {   // the end of a pair that an earlier warp began
                    float *to = reinterpret_cast<float *>(part) + (run * 32 + lane) * NA;
#pragma unroll
                    for (int e = 0; e < NA; ++e) to[e] = acc[e];
                }
            } else if (!whole && cur.win == lo + nw - 1) {   // more windows of the pair in a later phase
                float *to = reinterpret_cast<float *>(between) + (cur.pair * 32 + lane) * NA;
#pragma unroll
                for (int e = 0; e < NA; ++e) to[e] = acc[e];
            }
            advance(cur);
        }
    }

    // ---- pairs that several warps share: the warp with the first window adds the others' sums up, in the runs' order ----
    if (whole) {
        const bool open = done == total && total > 0 && cur.win != 0;   // this warp's last pair is not finished
        if (alive && open && !began) {
            float *to = reinterpret_cast<float *>(part) + (run * 32 + lane) * NA;
#pragma unroll
            for (int e = 0; e < NA; ++e) to[e] = acc[e];
        }
        __syncthreads();
        if (alive && open && began) {
            const int jobs = P * nwin, end = (cur.pair + 1) * nwin;
            for (int c = run + 1; c < kMmaWarps; ++c) {
                const int s = c * jobs / kMmaWarps, e1 = (c + 1) * jobs / kMmaWarps;
                if (s >= end) break;
                if (s == e1) continue;
                const float *from = reinterpret_cast<const float *>(part) + (c * 32 + lane) * NA;
#pragma unroll
                for (int e = 0; e < NA; ++e) acc[e] += from[e];
            }
            if (!*abort_flag) emit(cur.pair);
        }
    }

    __syncwarp();
    if (alive && abort_flag[1 + warp]) mma_marked_outputs<Q, GROUPED, WIDE>(p);   // (the warp's ring is free now)

    // Gave up on a wait: copies this warp started may still be in flight.  See them land (bounded)
    // before the block's shared memory can be handed to another block.
    if (!alive && lane == 0) {
        for (int j = consumed; j < issued; ++j) {
            bool landed = false;
            for (int itr = 0; itr < kSpinLimit && !landed; ++itr) {
                landed = mbar_test_wait(full0 + 8 * (j % D), uint32_t((j / D) & 1));
                if (!landed) __nanosleep(32);
            }
            if (!landed) atomicExch(&g_mma_status, int(kMmaWaitDrain));
        }
    }
}

// Shared memory of one launch: where things lie, how many windows' x is staged at a time and how deep the rings are.
struct MmaLayout {
    int phase_windows, depth, x_at, sum_at, ring_at;
};
static MmaLayout mma_layout(int q, bool grouped, int B, int windows, int pairs)
{
    const int slot = 2 * (q * 512 + (grouped ? (q + 1) * 64 : 0)), wide = B > 8, acc_bytes = wide ? 32 : 16, br = wide ? 16 : 8;
    const int x_window = B * kXColBytes + 4 * br * int(sizeof(float));
    MmaLayout l;
    l.x_at = kMmaFixedBytes + kMmaWarps * 32 * acc_bytes;
    const int room = kMmaSmemBytes - l.x_at - 128;   // (the rings start at a multiple of 128)
    const int fit = (room - 2 * kMmaWarps * slot) / x_window;   // two slots per warp at least
    int sums = 0;
    if (windows <= fit) {
        l.phase_windows = windows;
    } else {   // phases: the pairs' sums between them, and one slot per warp if two leave no room for x
        sums = pairs * 32 * acc_bytes;
        int x_room = room - sums - 2 * kMmaWarps * slot;
        if (x_room < x_window) x_room = room - sums - kMmaWarps * slot;
        l.phase_windows = x_room / x_window;
        if (l.phase_windows > windows - 1) l.phase_windows = windows - 1;   // (phases and pairs shared by warps exclude each other)
    }
    l.sum_at = l.x_at + l.phase_windows * x_window;
    l.ring_at = (l.sum_at + sums + 127) / 128 * 128;
    l.depth = (kMmaSmemBytes - l.ring_at) / (kMmaWarps * slot);
    if (l.depth > kMmaMaxSlotsPerWarp) l.depth = kMmaMaxSlotsPerWarp;
    return l;
}
int mma_windows_at_once(int q, bool grouped, int B)
{
    int w = 1;
    while (w < kMaxWindowsPerBlock && mma_layout(q, grouped, B, w + 1, 1).phase_windows == w + 1) ++w;
    return w;
}

template <int Q, bool GROUPED, bool WIDE>
static cudaError_t launch_mma_q(const MmaParams &prm, dim3 grid, cudaStream_t st)
{
    static bool configured[64] = {};   // the shared-memory opt-in is per function and per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(mma_gemm_kernel<Q, GROUPED, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaSmemBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kMmaThreads);
    cfg.dynamicSmemBytes = kMmaSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see griddepcontrol in the kernel
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, mma_gemm_kernel<Q, GROUPED, WIDE>, prm);
}

template <int Q>
static cudaError_t launch_mma_sel(const MmaParams &prm, bool grouped, dim3 grid, cudaStream_t st)
{
    const bool wide = prm.B > 8;
    if (grouped) return wide ? launch_mma_q<Q, true, true>(prm, grid, st) : launch_mma_q<Q, true, false>(prm, grid, st);
    return wide ? launch_mma_q<Q, false, true>(prm, grid, st) : launch_mma_q<Q, false, false>(prm, grid, st);
}

cudaError_t launch_mma_gemm(const bcq_desc &d, const bcq_plan &plan, const void *packed, const uint16_t *alpha,
                            const uint16_t *z, const uint16_t *X, uint16_t *Y, int B, void *workspace, cudaStream_t st)
{
    MmaParams prm = {};
    prm.tiles = static_cast<const uint8_t *>(packed);
    prm.alpha = alpha;   // used with per-row scales only
    prm.z = z;
    prm.X = reinterpret_cast<const __half *>(X);
    prm.Y = reinterpret_cast<__half *>(Y);
    prm.accum = static_cast<unsigned long long *>(workspace);
    prm.N = d.N;
    prm.K = d.K;
    prm.B = B;
    const int U = d.N / kUnitRows, W = d.K / kWindow;
    const int splits = plan.k_splits < kMmaMaxSplits ? plan.k_splits : kMmaMaxSplits;
    prm.u_base = U / plan.row_blocks, prm.u_rem = U % plan.row_blocks;
    prm.w_base = W / splits, prm.w_rem = W % splits;
    prm.ones = 0x3C003C00u;
    prm.split = splits > 1;
    prm.fmt = split_format(splits);
    const bool grouped = d.group != 0;
    const int windows = prm.w_base + (prm.w_rem ? 1 : 0), pairs = (prm.u_base + (prm.u_rem ? 1 : 0) + 1) / 2;
    const MmaLayout l = mma_layout(d.q, grouped, B, windows, pairs);   // (a warp's ring is at least 2 KB: mma_whole_pair)
    if (l.phase_windows < 1 || l.depth < 1) return cudaErrorInvalidValue;
    prm.phase_windows = l.phase_windows, prm.depth = l.depth;
    prm.x_at = l.x_at, prm.sum_at = l.sum_at, prm.ring_at = l.ring_at;
    const dim3 grid(plan.row_blocks, splits);
    switch (d.q) {
        case 1: return launch_mma_sel<1>(prm, grouped, grid, st);
        case 2: return launch_mma_sel<2>(prm, grouped, grid, st);
        case 3: return launch_mma_sel<3>(prm, grouped, grid, st);
        case 4: return launch_mma_sel<4>(prm, grouped, grid, st);
    }
    return cudaErrorInvalidValue;
}

// Read and clear the device status word (synchronises with the device).
cudaError_t mma_status_take(int *status)
{
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_mma_status, sizeof(int));
    if (e != cudaSuccess) return e;
    if (v != 0) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_mma_status, &zero, sizeof(int));
    }
    *status = v;
    return e;
}

}  // namespace bcq
