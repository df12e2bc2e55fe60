// Output error of the candidates of the GPTQT search (Eq. gptqt step 2; Eq. reexplore) on tcgen05.
//
// For one re-explored scale (W_int, S, qbias of step 1 are given) and a set of BCchoice candidates p:
//
//     err[p][n] = sum_t ( sum_k ( S lut_p[W_int[n][k]] + qbias - W[n][k] ) X[t][k] )^2
//
// lut_p[v] = the integer of BCchoice p nearest to v (Eq. round).  The inner sum is a dense contraction
// dW_p (N x K) times X^T (K x T): here the tensor cores are the right unit.  A block owns 128 rows of W
// and up to four candidates; per 64-wide slice of K its threads form the four dW_p tiles in fp16 (dW_p = S step_p[v] + r:
// step_p[v] = lut_p[v] - v, one shared-memory word per element holds it for all four candidates; r = S v + qbias - W, the
// residual of step 1, fp32 and rounded to fp16 once; one fp16 fused multiply-add per pair of elements and candidate)
// straight into shared memory in the 128-byte-swizzled K-major
// operand layout, and a warp of its own issues tcgen05.mma (M = 128, N = T, K = 16, fp16 x fp16 -> fp32) into
// one accumulator per candidate in tensor memory.  The slices of X (same layout), r and W_int arrive by tensor-map
// copies that one thread starts (r and W_int of all scale factors are written by one pass over W, launch_step_one): thousands of 16-byte loads per slice would hold the forming warps at the load
// queue.  Two operand stages: the 16 forming warps publish a stage on its "full" mbarrier, the issuing warp hands it
// back by tcgen05.commit on its "free" mbarrier, so the tensor cores work on one slice while the next is formed
// (issuing 16 MMAs holds a thread for about a microsecond: a forming thread cannot do it).  At the end every row's
// T outputs are read back with tcgen05.ld, squared and summed.  Several scale factors share a launch (grid z).
//
// All waits are bounded; a wait that runs out sets a device status word (see search_status_take), the
// block still frees its tensor memory and returns.
#include <cuda.h>   // CUtensorMap and its enumerations (types only: the encoder is taken from the runtime)

#include "bcq_async.cuh"
#include "bcq_internal.cuh"

namespace bcq {

constexpr int kSearchThreads = 512;      // 16 warps form the operand tiles (latency-bound with fewer)
constexpr int kSearchFormers = kSearchThreads / 32;
constexpr int kSearchBlock = kSearchThreads + 64;   // + the warp that issues the MMAs and the one that starts the copies
constexpr int kSearchRows = 128;        // rows of W per block = M of the MMA
constexpr int kSearchKTile = 64;        // weights along K per stage: 128 bytes of fp16, one swizzle row
constexpr int kSearchMaxCand = 4;       // candidates (accumulators) per block
constexpr int kSearchATile = kSearchRows * kSearchKTile * 2;   // 16 KB
constexpr int kSearchMaxT = 256;
constexpr int kSearchWTile = kSearchRows * kSearchKTile * 2;   // a slice of the residuals: 16 KB
constexpr int kSearchITile = kSearchRows * kSearchKTile;       // a slice of W_int: 8 KB
constexpr int kSearchSpin = 1 << 22;

static __device__ int g_search_status = 0;

struct SearchParams {
    const __half *S;        // [N][G] per scale factor, scale_stride elements apart
    size_t scale_stride;
    const __half *X;        // [T][K]
    float *err_rows;        // [scale factor][P][N]
    int N, K, G, L;         // N: rows of this launch; L = weights per scaling unit (K when one per row)
    int err_stride;         // rows of err_rows per candidate
    int T, P;               // T: tokens of this launch (a piece of at most 256 of the call's)
    int accumulate;         // add to err_rows instead of writing it (every piece but the first)
    int cand_per_block;     // 1..4, so that cand_per_block * T <= 512 columns of tensor memory
    int tmem_cols;          // power of two >= 32 covering cand_per_block accumulators of acc_cols columns
    int tokens_first;       // the MMAs' roles (see search_tokens_first)
    int lut_size;           // 2^n_bits <= 64
    const float *lut;       // [P][64]: lut[p][v] = the integer of BCchoice p nearest to v
    const int *order;       // [P]: the candidates as the blocks take them (see search_step_is_byte)
};

__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    // K-major operand, 128-byte swizzle: rows of 128 bytes, groups of 8 rows 1024 bytes apart
    uint64_t d = 0;
    d |= uint64_t((addr & 0x3FFFFu) >> 4);        // start address, 16-byte units
    d |= uint64_t(1) << 16;                        // leading byte offset (unused with a swizzled K-major tile)
    d |= uint64_t(1024 >> 4) << 32;                // stride byte offset: 8 rows further on
    d |= uint64_t(1) << 46;                        // descriptor version of this architecture
    d |= uint64_t(2) << 61;                        // 128-byte swizzle
    return d;
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool search_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int code)
{
    for (int it = 0; it < kSearchSpin; ++it) {
        if (mbar_test_wait(bar, parity)) return true;
        if (it >= 8) __nanosleep(64);
        if ((it & 255) == 255 && *abort_flag) return false;
    }
    *abort_flag = 1;
    atomicExch(&g_search_status, code);
    return false;
}

// one box of a tiled tensor map into shared memory, completion counted in bytes on an mbarrier (x: the
// innermost coordinate in elements, a multiple of 64 here: 64- or 128-byte aligned)
__device__ __forceinline__ void tma_box_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
                 "l"(map), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}
// a copy this block has started must have landed before the block's shared memory is given up
__device__ __forceinline__ void search_drain(uint32_t bar, uint32_t parity)
{
    for (int it = 0; it < kSearchSpin; ++it) {
        if (mbar_test_wait(bar, parity)) return;
        __nanosleep(64);
    }
}

// grid (row tiles of 128, groups of cand_per_block candidates, scale factors); dynamic shared memory: 2 stages x
// (cand_per_block x 16 KB of dW tiles | X's slice, T x 128 bytes rounded up to 1 KB | the residual's slice 16 KB | W_int's 8 KB),
// 1024-byte aligned.
__global__ void __launch_bounds__(kSearchBlock, 1)
    search_error_kernel(const SearchParams p, const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
                        const __grid_constant__ CUtensorMap imap)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // stage 0 free, stage 1 free, all done, stage 0/1 full, X of stage 0/1 landed, residuals and W_int of stage 0/1 landed
    __shared__ __align__(8) unsigned long long bars[9];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    // per value v of W_int one word: byte c stands for lut_c[v] - v, the step from v to the nearest integer of the block's
    // candidate c (between -63 and 63): the upper byte of the step as fp16 if that is all of it for every step of the block,
    // else 128 + step.  One lookup per operand element serves the four candidates.
    __shared__ uint32_t step_s[64];
    __shared__ float part[4][kSearchMaxCand][kSearchRows];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cand0 = blockIdx.y * p.cand_per_block;
    const int ncand = min(p.cand_per_block, p.P - cand0);
    const int T = p.T;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_bytes = uint32_t(p.cand_per_block) * kSearchATile, x_bytes = (uint32_t(T) * 128u + 1023u) & ~1023u;
    const uint32_t stage_bytes = a_bytes + x_bytes + kSearchWTile + kSearchITile;   // dW tiles | X | residuals | W_int
    const uint32_t bar0 = smem_u32(&bars[0]);
    volatile int *abort_flag = &abort_s;

    int cand[kSearchMaxCand];   // the block's candidates
#pragma unroll
    for (int c = 0; c < kSearchMaxCand; ++c) cand[c] = p.order[cand0 + min(c, ncand - 1)];
    bool fits = true;
    for (int v = tid; v < p.lut_size; v += kSearchBlock)
        for (int c = 0; c < ncand; ++c) fits = fits && search_step_is_byte(int(p.lut[size_t(cand[c]) * 64 + v]) - v);
    const bool byte_steps = __syncthreads_and(fits ? 1 : 0) != 0;
    for (int v = tid; v < p.lut_size; v += kSearchBlock) {
        uint32_t word = byte_steps ? 0u : 0x80808080u;   // candidates the block does not have: step 0
        for (int c = 0; c < ncand; ++c) {
            const int step = int(p.lut[size_t(cand[c]) * 64 + v]) - v;   // the table holds integers
            const uint32_t code = byte_steps ? uint32_t(__half_as_ushort(__int2half_rn(step))) >> 8 : uint32_t(128 + step);
            word = (word & ~(0xffu << (8 * c))) | (code << (8 * c));
        }
        step_s[v] = word;
    }
    if (tid == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        mbar_init(bar0 + 16, 1);
        mbar_init(bar0 + 24, kSearchFormers);
        mbar_init(bar0 + 32, kSearchFormers);
        for (int i = 5; i < 9; ++i) mbar_init(bar0 + 8 * i, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {   // one warp allocates the accumulators' columns of tensor memory
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(uint32_t(p.tmem_cols)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_s;

    // instruction descriptor: fp32 accumulate, fp16 A and B, both K-major, M = 128; N: tokens, or the rows of one or two
    // candidates
    const uint32_t idesc = (1u << 4) | (uint32_t(kSearchRows >> 4) << 24);
    const uint32_t idesc_n = uint32_t((p.tokens_first ? kSearchRows : T) >> 3) << 17;

    const int ktiles = p.K / kSearchKTile;
    bool alive = true;
    if (warp == kSearchFormers) {
        // ---- the issuing warp: per slice, wait until the stage is full, issue the slice's MMAs, hand the stage back ----
        for (int kt = 0; kt < ktiles && alive; ++kt) {
            const int s = kt & 1;
            if (!search_wait(bar0 + 24 + 8 * s, uint32_t((kt >> 1) & 1), abort_flag, 3) ||
                !search_wait(bar0 + 40 + 8 * s, uint32_t((kt >> 1) & 1), abort_flag, 4)) {
                alive = false;
                break;
            }
            if (lane == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t st_base = base + uint32_t(s) * stage_bytes;
                const uint64_t xdesc = smem_desc_sw128(st_base + a_bytes);
                if (p.tokens_first) {
                    for (int c = 0; c < ncand; c += 2) {   // two candidates' tiles lie one behind the other: 256 rows
                        const uint64_t wdesc = smem_desc_sw128(st_base + uint32_t(c) * kSearchATile);
                        const uint32_t both = idesc + (c + 1 < ncand ? 2u * idesc_n : idesc_n);
#pragma unroll
                        for (int j = 0; j < kSearchKTile / 16; ++j)   // 16 weights = 32 bytes further along the row
                            umma_f16(tmem_base + uint32_t(c * kSearchRows), xdesc + uint64_t(2 * j), wdesc + uint64_t(2 * j), both, (kt > 0 || j > 0) ? 1u : 0u);
                    }
                } else {
                    for (int c = 0; c < ncand; ++c) {
                        const uint64_t wdesc = smem_desc_sw128(st_base + uint32_t(c) * kSearchATile);
#pragma unroll
                        for (int j = 0; j < kSearchKTile / 16; ++j)
                            umma_f16(tmem_base + uint32_t(c * T), wdesc + uint64_t(2 * j), xdesc + uint64_t(2 * j), idesc + idesc_n, (kt > 0 || j > 0) ? 1u : 0u);
                    }
                }
                umma_commit(bar0 + 8 * s);
                if (kt == ktiles - 1) umma_commit(bar0 + 16);
            }
            __syncwarp();
        }
    } else if (warp == kSearchFormers + 1) {
        // ---- the copying warp: residuals and W_int a slice ahead (their stage is read again when every forming warp has finished the
        // slice before), X as soon as the tensor cores have let go of the stage ----
        if (lane == 0) {
            const int irow0 = int(blockIdx.z) * p.N + int(blockIdx.x) * kSearchRows;   // the scale factors' matrices as one of gridDim.z * N rows
            int x_started = -1, w_started = -1;
            auto start_w = [&](int kt) {
                const uint32_t to = base + uint32_t(kt & 1) * stage_bytes + a_bytes + x_bytes, bar = bar0 + 56 + 8 * (kt & 1);
                mbar_expect_tx(bar, kSearchWTile + kSearchITile);
                tma_box_2d(to, &wmap, kt * kSearchKTile, irow0, bar);
                tma_box_2d(to + kSearchWTile, &imap, kt * kSearchKTile, irow0, bar);
                w_started = kt;
            };
            start_w(0);
            for (int kt = 0; kt < ktiles && alive; ++kt) {
                if (kt + 1 < ktiles) {
                    if (kt > 0 && !search_wait(bar0 + 24 + 8 * ((kt - 1) & 1), uint32_t(((kt - 1) >> 1) & 1), abort_flag, 6)) {
                        alive = false;
                        break;
                    }
                    start_w(kt + 1);
                }
                if (kt >= 2 && !search_wait(bar0 + 8 * (kt & 1), uint32_t(((kt >> 1) - 1) & 1), abort_flag, 7)) {
                    alive = false;
                    break;
                }
                mbar_expect_tx(bar0 + 40 + 8 * (kt & 1), uint32_t(T) * 128u);
                tma_box_2d(base + uint32_t(kt & 1) * stage_bytes + a_bytes, &xmap, kt * kSearchKTile, 0, bar0 + 40 + 8 * (kt & 1));
                x_started = kt;
            }
            // whatever was started lands before the block's shared memory is given up (long ago, unless the block gives up)
            for (int j = x_started; j >= 0 && j > x_started - 2; --j) search_drain(bar0 + 40 + 8 * (j & 1), uint32_t((j >> 1) & 1));
            for (int j = w_started; j >= 0 && j > w_started - 2; --j) search_drain(bar0 + 56 + 8 * (j & 1), uint32_t((j >> 1) & 1));
        }
    } else {
        // this thread's part of a dW tile: row r of the block, 16 consecutive weights (2 pieces of 16 bytes)
        const int r = tid >> 2, quart = tid & 3;
        const int n = blockIdx.x * kSearchRows + r;
        const bool row_ok = n < p.N;
        const uint32_t a_row_off = uint32_t(r) * 128u;
        // W's slice lands with the 128-byte swizzle (16-byte piece ^ row & 7: a warp's loads then spread over
        // all banks), W_int's as it is
        const uint32_t w_off0 = a_bytes + x_bytes + uint32_t(r) * 128u + uint32_t(((2 * quart) ^ (r & 7)) << 4);
        const uint32_t w_off1 = a_bytes + x_bytes + uint32_t(r) * 128u + uint32_t(((2 * quart + 1) ^ (r & 7)) << 4);
        const uint32_t i_off = a_bytes + x_bytes + kSearchWTile + uint32_t(r) * 64u + uint32_t(quart << 4);

        // scale of (row, scaling unit): loaded one slice before the unit starts (rows beyond N keep 0)
        const int slices_per_unit = p.L / kSearchKTile;
        const size_t s_at = size_t(blockIdx.z) * p.scale_stride + size_t(row_ok ? n : 0) * p.G;
        const __half *srow = p.S + s_at;
        __half s_next = __float2half_rn(0.f);
        if (row_ok) s_next = __ldg(srow);
        __half Sh = s_next;
        int unit = 0, left = 0;   // slices left in the current scaling unit

        // The forming warps do not wait for one another: each waits for the stage (the MMAs that read it two slices ago) and for
        // W, and publishes its part; a block-wide barrier per slice kept all of them in step, loads, arithmetic and stores one
        // after the other.
        for (int kt = 0; kt < ktiles; ++kt) {
            const int s = kt & 1;
            const uint32_t st_base = base + uint32_t(s) * stage_bytes;
            bool ok = kt < 2 || search_wait(bar0 + 8 * s, uint32_t(((kt >> 1) - 1) & 1), abort_flag, 1);
            ok = ok && search_wait(bar0 + 56 + 8 * s, uint32_t((kt >> 1) & 1), abort_flag, 5);
            if (!__all_sync(0xffffffffu, ok)) {
                alive = false;
                break;
            }

            uint4 wcur0, wcur1, icur;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(wcur0.x), "=r"(wcur0.y), "=r"(wcur0.z), "=r"(wcur0.w) : "r"(st_base + w_off0));
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(wcur1.x), "=r"(wcur1.y), "=r"(wcur1.z), "=r"(wcur1.w) : "r"(st_base + w_off1));
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(icur.x), "=r"(icur.y), "=r"(icur.z), "=r"(icur.w) : "r"(st_base + i_off));
            if (left == 0) {
                Sh = s_next;
                left = slices_per_unit;
                ++unit;
                if (row_ok && unit < p.G) s_next = __ldg(srow + unit);
            }
            --left;

            // dW_p = S lut_p[v] + qbias - W = S (lut_p[v] - v) + r with r = S v + qbias - W, the residual of step 1, which comes
            // ready (fp32, rounded to fp16 once for all candidates).  Per candidate the step comes
            // out of the lookup's byte as the fp16 number itself, or as 1024 + byte (bit pattern 0x6400 | byte), minus 1152; one
            // fp16 fused multiply-add on a pair of weights then is the operand as it is stored (rounded once).
            // (rows beyond N hold zeros or the next scale factor's first rows: they are formed like the others and their
            // outputs are not stored)
            const uint32_t resid[8] = {wcur0.x, wcur0.y, wcur0.z, wcur0.w, wcur1.x, wcur1.y, wcur1.z, wcur1.w};   // of weights (2 j, 2 j + 1)
            const uint32_t i4[4] = {icur.x, icur.y, icur.z, icur.w};   // 4 W_int: byte offsets into the words
            const __half2 S2 = __half2half2(Sh);
            auto form = [&](auto BYTES) {
                constexpr bool bytes = decltype(BYTES)::value;
                const __half2 bias2 = __half2half2(__float2half_rn(-1152.f));
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    uint32_t e[8];   // the words of weights 8 i .. 8 i + 7
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        e[j] = *reinterpret_cast<const uint32_t *>(reinterpret_cast<const unsigned char *>(step_s) +
                                                                   __byte_perm(i4[2 * i + (j >> 2)], 0u, 0x4440u + (j & 3)));
                    uint32_t pair01[4], pair23[4];   // bytes: candidates (0, 1) resp. (2, 3) of weights (2 j, 2 j + 1)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        pair01[j] = __byte_perm(e[2 * j], e[2 * j + 1], 0x5140u);
                        pair23[j] = __byte_perm(e[2 * j], e[2 * j + 1], 0x7362u);
                    }
                    const int piece = 2 * quart + i;
                    const uint32_t dst = st_base + a_row_off + uint32_t((piece ^ (r & 7)) << 4);
                    static_for<0, kSearchMaxCand>([&](auto C) {
                        constexpr int c = decltype(C)::value;
                        if (c < ncand) {
                            uint32_t packed[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t pair = c < 2 ? pair01[j] : pair23[j];
                                const uint32_t raw = bytes ? __byte_perm(pair, 0u, (c & 1) ? 0x3424u : 0x1404u)
                                                           : __byte_perm(pair, 0x64646464u, (c & 1) ? 0x4342u : 0x4140u);
                                __half2 step = *reinterpret_cast<const __half2 *>(&raw);
                                if constexpr (!bytes) step = __hadd2(step, bias2);
                                const __half2 h = __hfma2(S2, step, *reinterpret_cast<const __half2 *>(&resid[4 * i + j]));
                                packed[j] = *reinterpret_cast<const uint32_t *>(&h);
                            }
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + uint32_t(c) * kSearchATile), "r"(packed[0]), "r"(packed[1]), "r"(packed[2]), "r"(packed[3]) : "memory");
                        }
                    });
                }
            };
            if (byte_steps)
                form(std::true_type{});
            else
                form(std::false_type{});
            // the tiles are read by the tensor cores' proxy, and W's slice is overwritten by the copies' proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 24 + 8 * s);    // this warp's part of the stage is full
        }
    }

    // ---- the accumulators are complete: every row's squared outputs ------------------------------------
    alive = __syncthreads_and((alive && search_wait(bar0 + 16, 0u, abort_flag, 2)) ? 1 : 0) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int quarter = warp & 3, colpart = warp >> 2;   // a warp reads the 32 lanes of its quarter
    auto read16 = [&](int col, float (&v)[16]) {
        uint32_t w[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
            : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]),
              "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
            : "r"(tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(col)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(w[j]);
    };
    if (alive && warp < kSearchFormers) {
        for (int c = 0; c < ncand; ++c) {
            if (p.tokens_first) {
                // lane = token, column = row: 32 rows per warp, squared, then added up over the 32 tokens; every exchange
                // halves the rows a lane keeps, lane l ends up with row l (lanes beyond T hold whatever lay behind X)
                float sq[32];
                const bool token = quarter * 32 + lane < T;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float v[16];
                    read16(c * kSearchRows + colpart * 32 + half * 16, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) sq[half * 16 + j] = token ? v[j] * v[j] : 0.f;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int j = 0; j < o; ++j) {
                        const float send = up ? sq[j] : sq[j + o], keep = up ? sq[j + o] : sq[j];
                        sq[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                }
                part[quarter][c][colpart * 32 + lane] = sq[0];
            } else {   // lane = row, column = token: every fourth piece of 16 columns
                float sum = 0.f;
                for (int ch = colpart; ch < T / 16; ch += 4) {
                    float v[16];
                    read16(c * T + ch * 16, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum = fmaf(v[j], v[j], sum);
                }
                part[colpart][c][quarter * 32 + lane] = sum;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (alive && tid < kSearchRows) {
        const int row = blockIdx.x * kSearchRows + tid;
        if (row < p.N)
            for (int c = 0; c < ncand; ++c) {
                float *out = p.err_rows + (size_t(blockIdx.z) * p.P + size_t(p.order[cand0 + c])) * p.err_stride + row;
                const float sum = (part[0][c][tid] + part[1][c][tid]) + (part[2][c][tid] + part[3][c][tid]);
                *out = p.accumulate ? *out + sum : sum;   // pieces of tokens run one after the other on the stream
            }
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(uint32_t(p.tmem_cols)) : "memory");
    }
}

// err[c] = sum over rows of err_rows[c][.] in a fixed order (fp64), one block per candidate
__global__ void __launch_bounds__(256) search_sum_kernel(const float *__restrict__ err_rows, int N, double *__restrict__ err)
{
    __shared__ double sh[256];
    const float *src = err_rows + size_t(blockIdx.x) * N;
    double s = 0.0;
    for (int i = threadIdx.x; i < N; i += 256) s += double(src[i]);
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) err[blockIdx.x] = sh[0];
}

// the first candidate, in order, whose error is below all earlier ones
__global__ void search_argmin_kernel(const double *__restrict__ err, int count, int P, int *__restrict__ best)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int at = 0;
    double lowest = err[0];
    for (int i = 1; i < count; ++i)
        if (err[i] < lowest) lowest = err[i], at = i;
    best[0] = at / P;
    best[1] = at % P;
}

// Which operand the MMAs take as A.  Weights: 128 rows of one candidate against T tokens.  Tokens: up to 128 of them
// against the rows of two candidates at once, which reads 12 instead of 16 KB of shared memory per 16 weights and pair of
// candidates at 128 tokens (the pipe that bounds the kernel), but not less from 64 tokens down, and more than 128 do not fit.
bool search_tokens_first(int T) { return T > 64 && T <= kSearchRows; }
int search_cand_per_block(int T)
{
    int c = 512 / T;
    return c > kSearchMaxCand ? kSearchMaxCand : c;
}

// tokens per launch: pieces of about equal size, multiples of 16
static int search_piece(int T)
{
    const int pieces = (T + kSearchMaxT - 1) / kSearchMaxT;
    return ((T + pieces - 1) / pieces + 15) / 16 * 16;
}
// Rows per launch where only `most` rows' step 1 (a multiple of 128) fit the workspace: the multiple of 128 with the fewest
// rounds of blocks, one per SM (4096 x 4096, 25 candidates, 8 factors, 128 tokens: 32 tiles of rows are 1792 blocks, 13 rounds,
// in launches of 10 tiles still 13, of 11 14).  Every launch also waits for its last blocks and for its step 1: a quarter of a round.
int search_rows_per_launch(int N, int most, int T, int P, int scales, int sms)
{
    if (most >= N || most < kSearchRows) return most;
    const int piece = search_piece(T), per_block = search_cand_per_block(piece);
    const long long per_tile = (long long)((P + per_block - 1) / per_block) * scales;
    const int tiles = (N + kSearchRows - 1) / kSearchRows;
    auto rounds = [&](int t) { return (t * per_tile + sms - 1) / sms; };
    long long best = -1;
    int rows = kSearchRows;
    for (int t = most / kSearchRows; t >= 1; --t) {
        const long long quarters = 4 * (tiles / t * rounds(t) + (tiles % t ? rounds(tiles % t) : 0)) + (tiles + t - 1) / t;
        if (best < 0 || quarters < best) best = quarters, rows = t * kSearchRows;
    }
    return rows;
}

// two stages of (dW tiles | X | residuals | W_int), each part a multiple of 1024 bytes, + room to align the first
size_t search_smem_bytes(int T)
{
    const size_t x_bytes = (size_t(T) * 128 + 1023) / 1024 * 1024;
    return 2 * (size_t(search_cand_per_block(T)) * kSearchATile + x_bytes + kSearchWTile + kSearchITile) + 1024;
}

// Tensor map of a row-major matrix [rows][cols] for boxes of 64 columns x box_rows rows.  The encoder is a
// driver function; the runtime hands out its address, so the library links against the runtime only.
static cudaError_t search_tensor_map(CUtensorMap *map, const void *ptr, bool bytes, uint64_t rows, uint64_t cols, uint32_t box_rows,
                                     bool swizzle)
{
    using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &found);
        if (e != cudaSuccess) return e;
        if (found != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<Encode>(fn);
    }
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * (bytes ? 1u : 2u)};
    const cuuint32_t box[2] = {uint32_t(kSearchKTile), box_rows};
    const cuuint32_t steps[2] = {1u, 1u};
    const CUresult r = encode(map, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(ptr), dims,
                              strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_search_errors(const uint16_t *resid, const uint8_t *offsets, const uint16_t *S, size_t scale_stride, const uint16_t *X,
                                 int rows, int N, int K, int group, int T, int n_bits, const float *lut_dev /*[P][64]*/, const int *order_dev /*[P]*/,
                                 int P, int scales, float *err_rows /*[scales][P][N], from the first of these rows on*/, cudaStream_t st)
{
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    SearchParams p = {};
    p.S = reinterpret_cast<const __half *>(S), p.scale_stride = scale_stride;
    p.X = reinterpret_cast<const __half *>(X), p.err_rows = err_rows;
    p.N = rows, p.err_stride = N, p.K = K, p.L = group == 0 ? K : group, p.G = K / p.L, p.P = P;
    p.lut_size = 1 << n_bits;
    p.lut = lut_dev, p.order = order_dev;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        size_t most = 0;
        for (int t = 16; t <= kSearchMaxT; t += 16) most = search_smem_bytes(t) > most ? search_smem_bytes(t) : most;
        e = cudaFuncSetAttribute(search_error_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    // the slices of the residuals and of W_int (the scale factors' matrices as one of scales * rows rows)
    CUtensorMap xmap, wmap, imap;
    const uint64_t all = uint64_t(scales) * uint64_t(rows);
    if ((e = search_tensor_map(&wmap, resid, false, all, uint64_t(K), uint32_t(kSearchRows), true)) != cudaSuccess) return e;
    if ((e = search_tensor_map(&imap, offsets, true, all, uint64_t(K), uint32_t(kSearchRows), false)) != cudaSuccess) return e;
    const unsigned row_tiles = unsigned((rows + kSearchRows - 1) / kSearchRows);
    // the error is a sum over tokens: pieces of at most 256 tokens, one launch each, the later ones adding to err_rows
    const int piece = search_piece(T);
    for (int t0 = 0; t0 < T; t0 += piece) {
        const int Tp = T - t0 < piece ? T - t0 : piece;
        p.X = reinterpret_cast<const __half *>(X) + size_t(t0) * K;
        p.T = Tp, p.accumulate = t0 > 0 ? 1 : 0;
        p.cand_per_block = search_cand_per_block(Tp);
        p.tokens_first = search_tokens_first(Tp) ? 1 : 0;
        int cols = 32;
        while (cols < p.cand_per_block * (p.tokens_first ? kSearchRows : Tp)) cols *= 2;
        p.tmem_cols = cols;
        if ((e = search_tensor_map(&xmap, p.X, false, uint64_t(Tp), uint64_t(K), uint32_t(Tp), true)) != cudaSuccess) return e;   // all rows of the piece
        const unsigned groups = unsigned((P + p.cand_per_block - 1) / p.cand_per_block);
        search_error_kernel<<<dim3(row_tiles, groups, unsigned(scales)), kSearchBlock, search_smem_bytes(Tp), st>>>(p, xmap, wmap, imap);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_search_sums(const float *err_rows, int N, int candidates, double *err, cudaStream_t st)
{
    search_sum_kernel<<<unsigned(candidates), 256, 0, st>>>(err_rows, N, err);
    return cudaGetLastError();
}

cudaError_t launch_search_argmin(const double *err, int count, int P, int *best, cudaStream_t st)
{
    search_argmin_kernel<<<1, 32, 0, st>>>(err, count, P, best);
    return cudaGetLastError();
}

cudaError_t search_status_take(int *status)
{
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_search_status, sizeof(int));
    if (e != cudaSuccess) return e;
    if (v != 0) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_search_status, &zero, sizeof(int));
    }
    *status = v;
    return e;
}

}  // namespace bcq
