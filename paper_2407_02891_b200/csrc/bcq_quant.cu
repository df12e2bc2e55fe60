// On-device quantiser front end: fp16 weights -> packed binary-coded operand in one call.
//
//   step 1 (Eq. gptqt, with the scale of section "Re-explore Scaling Factor"), per (row, group):
//       qbias = Wmin,  S = fp16( s_factor (Wmax - Wmin) / (2^n - 1) ),
//       W_int = clamp( round((W - qbias) / S), 0, 2^n - 1 )        (nearest, ties to even)
//   step 2 (Eq. round): W_int -> code of the nearest integer the merged planes reach
//   fusion (Eq. fuse_step3): alpha_j = S m_j,  z = S (2^n - 1)/2 + qbias
//   packing: code bit i -> plane i, written straight into the layout of the descriptor.
//
// The quantiser is the inverse of the dequantisation S W_int + qbias and uses the fp16 S that is
// stored.  The integer is defined in fp64: W - qbias is exact there, the quotient is rounded once,
// so the decision does not depend on evaluation order.
//
// One kernel.  A warp takes one 128-weight segment of eight rows at a time, 32 weights per lane (see bcq_planes.cuh).
// Groups of 128, 64 and 32 are 4, 2 and 1 of those lanes: range by shuffles, one pass over W.  Other group lengths (and
// one scale per row) take the range first, eight rows per block, and read the rows a second time from L2.
//
// Bound: instruction issue (slots 68 % busy, 20.6 instructions per weight), then HBM (2 bytes per weight).  7168 x 7168, q = 3, groups of 128: 201 us with a chunk of 8 weights per
// thread, byte stores and a 16-lane range reduction; 52.9 us with 32 weights per lane; 49.5 us with integers of up to 4 bits looked up
// two at a time; 47.1 us (2.7 TB/s) without the comparison with the top integer where no weight lies beyond it.
#include "bcq_planes.cuh"

namespace bcq {

struct QuantTable {
    uint8_t code_of_int[256];
    double plane_weight[4];
    double centre;      // (2^n - 1) / 2
    double top;         // 2^n - 1
    double s_factor;
};

__device__ __forceinline__ void range_to_scale(float lo, float hi, double s_factor, double top, __half &s_h, __half &b_h)
{
    if (lo == 0.f) lo = 0.f;   // a zero minimum is stored as +0
    const double range = double(hi) - double(lo);   // exact
    s_h = __double2half(__ddiv_rn(__dmul_rn(s_factor, range), top));
    b_h = __float2half_rn(lo);                      // exact: lo is an fp16 value
}

// alpha_j = S m_j (j < q), z = S centre + qbias (j = q) of one (row, group): exact in fp64, rounded once.
__device__ __forceinline__ uint16_t fused_scale(__half s_h, __half b_h, const QuantTable &tab, int q, int j)
{
    const double s = double(__half2float(s_h));
    return __half_as_ushort(__double2half(j < q ? s * tab.plane_weight[j & 3] : s * tab.centre + double(__half2float(b_h))));
}

// the integer by its definition
__device__ __noinline__ uint32_t exact_int(uint32_t w16, __half b_h, __half s_h, double top)
{
    const double w = double(__half2float(__ushort_as_half(uint16_t(w16)))), b = double(__half2float(b_h)), s = double(__half2float(s_h));
    if (!(s > 0.0)) return 0u;                         // a constant group (or a NaN scale)
    const double r = rint(__ddiv_rn(w - b, s));        // the subtraction is exact in fp64
    return uint32_t(fmin(fmax(r, 0.0), top));
}

// Per-group constants of the integer decision.  t = (W - qbias)/S is evaluated as ONE fp32 fused multiply-add onto a
// constant that carries 2^23 / 2^FR, one half and a margin of e ulps: the result's mantissa then holds t + 1/2 + margin
// in fixed point with FR fraction bits, its integer part being the rounded quotient, unless the fraction is below
// 2 e -- then the quotient lies within the error bound of a rounding boundary (exact ties do) and the fp64 definition
// decides.  Error in units of 2^-FR: 1/2 for the rounding of the result, (|qbias/S| + 257) 2^(FR - 24) for the constant,
// t 2^(FR - 24) <= 1 for the reciprocal where t is inside the range (beyond it every value clamps to the top).
template <int FR>
struct IntDecision {
    float inv, c;
    int ceiling;         // bit pattern of "top": everything beyond is the top integer
    uint32_t doubt;      // fractions below this go to fp64; > 65535: all do
    __device__ IntDecision(__half s_h, __half b_h, float lo, float hi, double top)
    {
        const float sf = __half2float(s_h), bf = __half2float(b_h);
        constexpr float kOne = float(1 << FR), kBase = 8388608.f / kOne;   // [kBase, 2 kBase): ulp 2^-FR
        inv = sf > 0.f ? __frcp_rn(sf) : 0.f;   // S = 0: every integer is 0
        const float far = fabsf(bf) * inv;
        // (S overflowed, or the range or a weight is not a finite number: leave it to the definition)
        const bool plain = sf < 65536.f && fabsf(lo) < 65536.f && fabsf(hi) < 65536.f && far < 1048576.f;
        const int e = plain ? 4 + int(far * (1.f / 256.f)) : 0;
        doubt = plain ? uint32_t(2 * e) : 0x10000u;
        c = plain ? fmaf(-bf, inv, kBase + 0.5f + float(e) / kOne) : kBase;
        if (!plain) inv = 0.f;
        ceiling = __float_as_int(kBase + float(top) + 0.5f);
    }
    // Whether the integer part for this weight is above the top: half a unit above the ceiling, which is the middle of the top
    // integer's cell (fractions up to there are one half and more, and never in doubt).  NaN counts as above.
    __device__ bool beyond_top(float w) const { return __float_as_int(fmaf(w, inv, c)) >= ceiling + (1 << (FR - 1)); }
};

// Integers of the 8 weights of one 16-byte piece, one per byte.  CLAMP: some weight may lie beyond the top integer.
template <int FR, bool CLAMP = true>
__device__ __forceinline__ uint2 piece_ints(const uint4 raw, const IntDecision<FR> &dec, __half s_h, __half b_h, double top)
{
    const uint32_t word[4] = {raw.x, raw.y, raw.z, raw.w};
    uint32_t bits[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&word[j]));
        const int t0 = __float_as_int(fmaf(f.x, dec.inv, dec.c)), t1 = __float_as_int(fmaf(f.y, dec.inv, dec.c));
        bits[2 * j] = uint32_t(CLAMP ? min(t0, dec.ceiling) : t0);
        bits[2 * j + 1] = uint32_t(CLAMP ? min(t1, dec.ceiling) : t1);
    }
    uint32_t least = 0xffffffffu;   // smallest fraction, two halves
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t pair = __byte_perm(bits[2 * j], bits[2 * j + 1], 0x5410u);
        if (FR == 15) pair &= 0x7fff7fffu;
        least = __vminu2(least, pair);
    }
    if (FR == 15) {
#pragma unroll
        for (int j = 0; j < 8; ++j) bits[j] <<= 1;   // the integer into byte 2
    }
    if (min(least & 0xffffu, least >> 16) < dec.doubt) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t frac = FR == 15 ? (bits[j] & 0xffffu) >> 1 : bits[j] & 0xffffu;
            if (frac < dec.doubt) bits[j] = exact_int(word[j >> 1] >> (16 * (j & 1)), b_h, s_h, top) << 16;
        }
    }
    return make_uint2(__byte_perm(__byte_perm(bits[0], bits[1], 0x0062u), __byte_perm(bits[2], bits[3], 0x0062u), 0x5410u),
                      __byte_perm(__byte_perm(bits[4], bits[5], 0x0062u), __byte_perm(bits[6], bits[7], 0x0062u), 0x5410u));
}

// entry t of the table = the code of step-1 integer t with code bit i moved to bit 8 i: the 8 entries of a chunk,
// shifted by their position and added up, are the chunk's byte of plane i in byte i
__device__ __forceinline__ uint32_t chunk_planes(const uint2 ints, const uint32_t *lut)
{
    uint32_t spread = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        spread += lut[(ints.x >> (8 * j)) & 0xffu] << j;
        spread += lut[(ints.y >> (8 * j)) & 0xffu] << (4 + j);
    }
    return spread;
}

// The same for integers of at most 4 bits, two at a time: entry a + 16 b of the table = the entry of a, and the entry of b moved up
// by one.
__device__ __forceinline__ uint32_t chunk_planes_pairs(const uint2 ints, const uint32_t *lut)
{
    const uint32_t x = ints.x | (ints.x >> 4), y = ints.y | (ints.y >> 4);   // a pair in bytes 0 and 2 of each
    return lut[x & 0xffu] + (lut[(x >> 16) & 0xffu] << 2) + (lut[y & 0xffu] << 4) + (lut[(y >> 16) & 0xffu] << 6);
}

// Ranges of M groups of any length by one warp, all M on their way together (NaN weights are ignored).  Lane 8 m + i (M = 1:
// lane i) returns the range of group m; the other lanes' values are not used.
template <int M>
__device__ __forceinline__ void warp_ranges(const __half *const (&w)[M], int L, float &lo, float &hi)
{
    const int lane = threadIdx.x & 31;
    __half2 lo2[M], hi2[M];
#pragma unroll
    for (int m = 0; m < M; ++m) lo2[m] = hi2[m] = __half2half2(w[m][0]);
    constexpr int kAtOnce = M == 1 ? 8 : 1;   // 16-byte pieces of a group on their way together (L is a multiple of 32)
    for (int k = 8 * lane; k < L; k += 256 * kAtOnce) {
        uint4 raw[M][kAtOnce];
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int c = 0; c < kAtOnce; ++c) raw[m][c] = *reinterpret_cast<const uint4 *>(w[m] + min(k + 256 * c, L - 8));   // (the last one again)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const __half2 *h = reinterpret_cast<const __half2 *>(raw[m]);
#pragma unroll
            for (int i = 0; i < 4 * kAtOnce; ++i) lo2[m] = __hmin2(lo2[m], h[i]), hi2[m] = __hmax2(hi2[m], h[i]);
        }
    }
    uint32_t both[M];   // (minimum, maximum) of a group, combined over the lanes
#pragma unroll
    for (int m = 0; m < M; ++m) {
        __half a = __hmin(__low2half(lo2[m]), __high2half(lo2[m])), b = __hmax(__low2half(hi2[m]), __high2half(hi2[m]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const __half2 mine = __halves2half2(a, b);
            const uint32_t got = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<const uint32_t *>(&mine), o);
            const __half2 other = *reinterpret_cast<const __half2 *>(&got);
            a = __hmin(a, __low2half(other)), b = __hmax(b, __high2half(other));
        }
        const __half2 r = __halves2half2(a, b);
        both[m] = *reinterpret_cast<const uint32_t *>(&r);
    }
    uint32_t own = both[0];
#pragma unroll
    for (int m = 1; m < M; ++m) own = (lane >> 3) == m ? both[m] : own;
    const __half2 r = *reinterpret_cast<const __half2 *>(&own);
    lo = __low2float(r), hi = __high2float(r);
}
// The groups g0 .. g1 of a block's row unit u, a warp per group or, where groups are short, per four of them: their ranges
// go to use(row, group, i, lo, hi), in the lanes i = 0 .. 7 of each.  (A warp per group of 96 has 12 lanes with weights and
// waits for one load after the other: 4096 x 4032, 162 us, 72 so.)
template <class Use>
__device__ __forceinline__ void unit_ranges(const __half *W, int N, int K, int L, int u, int g0, int g1, const Use &use)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = min(kUnitRows, N - u * kUnitRows), groups = g1 - g0 + 1, count = rows * groups;
    auto row = [&](int i) { return u * kUnitRows + i / groups; };
    auto group = [&](int i) { return g0 + i % groups; };
    auto at = [&](int i) { return W + size_t(row(i)) * K + size_t(group(i)) * L; };
    float lo, hi;
    if (L > 512) {
        for (int i = warp; i < count; i += 8) {
            const __half *w[1] = {at(i)};
            warp_ranges<1>(w, L, lo, hi);
            if (lane < 8) use(row(i), group(i), lane, lo, hi);
        }
    } else {
        for (int i = 4 * warp; i < count; i += 32) {
            const __half *w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = at(min(i + m, count - 1));
            warp_ranges<4>(w, L, lo, hi);
            const int mine = i + (lane >> 3);
            if (mine < count) use(row(mine), group(mine), lane & 7, lo, hi);
        }
    }
}
// the largest of a lane's 8 NR weights, NaN if there is one
template <int NR>
__device__ __forceinline__ __half lane_max(const uint4 (&raw)[NR])
{
    const __half2 *h = reinterpret_cast<const __half2 *>(raw);
    __half2 hi2 = h[0];
#pragma unroll
    for (int i = 1; i < 4 * NR; ++i) hi2 = __hmax2_nan(hi2, h[i]);
    return __hmax_nan(__low2half(hi2), __high2half(hi2));
}
// Range of a group that LANES neighbouring lanes hold, 8 NR weights each, in fp16 (exact).  A NaN weight is ignored by
// (lo, hi_scale), but shows in hi: it makes the group go by the definition.
template <int LANES, int NR>
__device__ __forceinline__ void lanes_range(const uint4 (&raw)[NR], float &lo, float &hi, float &hi_scale)
{
    const __half2 *h = reinterpret_cast<const __half2 *>(raw);
    __half2 lo2 = h[0];
#pragma unroll
    for (int i = 1; i < 4 * NR; ++i) lo2 = __hmin2(lo2, h[i]);
    __half lo_h = __hmin(__low2half(lo2), __high2half(lo2)), hi_h = lane_max(raw);
    for (int o = 1; o < LANES; o *= 2) {
        const __half2 both = __halves2half2(lo_h, hi_h);
        const uint32_t got = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<const uint32_t *>(&both), o);
        const __half2 other = *reinterpret_cast<const __half2 *>(&got);
        lo_h = __hmin(lo_h, __low2half(other)), hi_h = __hmax_nan(hi_h, __high2half(other));
    }
    lo = __half2float(lo_h), hi = hi_scale = __half2float(hi_h);
    if (__any_sync(0xffffffffu, hi != hi)) {
        __half2 hi2 = h[0];
#pragma unroll
        for (int i = 1; i < 4 * NR; ++i) hi2 = __hmax2(hi2, h[i]);
        hi_h = __hmax(__low2half(hi2), __high2half(hi2));
        for (int o = 1; o < LANES; o *= 2) {
            const uint32_t mine = __half_as_ushort(hi_h);
            hi_h = __hmax(hi_h, __ushort_as_half(uint16_t(__shfl_xor_sync(0xffffffffu, mine, o))));
        }
        hi_scale = __half2float(hi_h);
    }
}

// LANES: lanes per group, 4, 2 or 1 for groups of 128, 64 and 32 (one pass; jobs = (row unit, segment), segments
// fastest); 0 for any other group length L: a block takes the row unit blockIdx.x, ranges first, and of its segments the
// part blockIdx.y (groups that two parts share are done by both, with the same results).
// PAIRS: integers of at most 4 bits, looked up two at a time.  VOTE: a warp asks whether any of its weights lies beyond the top
// integer, and leaves the comparison out where none does; otherwise it compares them all.
template <int FR, int LANES, bool PAIRS, bool VOTE>
__global__ void __launch_bounds__(256, 3) rtn_kernel(const __half *__restrict__ W, const __grid_constant__ QuantTable tab, int L,
                                                  __half *S, __half *qbias, uint8_t *__restrict__ w_int, const View dst)
{
    __shared__ uint32_t lut[256];
    const int lane = threadIdx.x & 31, j = lane >> 2, l = lane & 3, warp = threadIdx.x >> 5;
    const auto spread = [&](uint32_t v) {
        const uint32_t code = tab.code_of_int[v];
        return (code & 1u) | ((code & 2u) << 7) | ((code & 4u) << 14) | ((code & 8u) << 21);
    };
    lut[threadIdx.x] = PAIRS ? spread(threadIdx.x & 15u) + (spread(threadIdx.x >> 4) << 1) : spread(threadIdx.x);
    const int N = dst.N, K = dst.K, G = K / L, q = dst.q;
    const int segs = (K + kSegment - 1) / kSegment;

    const int seg0 = LANES ? 0 : int((long long)segs * blockIdx.y / gridDim.y), seg1 = LANES ? segs : int((long long)segs * (blockIdx.y + 1) / gridDim.y);
    if constexpr (LANES == 0)
        unit_ranges(W, N, K, L, blockIdx.x, seg0 * kSegment / L, (min(seg1 * kSegment, K) - 1) / L,
                    [&](int n, int g, int i, float lo, float hi) {
                        __half s_h, b_h;
                        range_to_scale(lo, hi, tab.s_factor, tab.top, s_h, b_h);
                        if (i == 6) S[size_t(n) * G + g] = s_h;
                        if (i == 7) qbias[size_t(n) * G + g] = b_h;
                        if (i <= q) *(i < q ? dst.alpha_elem(i, n, g) : dst.z_elem(n, g)) = fused_scale(s_h, b_h, tab, q, i);
                    });
    __syncthreads();

    const PlaneWriter out(dst);
    const size_t stride = dst.plane_stride();
    const int units = LANES ? (N + kUnitRows - 1) / kUnitRows : int(blockIdx.x) + 1;   // the walk ends there
    SegmentWalk at_job(LANES ? (long long)blockIdx.x * 8 + warp : (long long)blockIdx.x * segs + seg0 + warp, LANES ? (long long)gridDim.x * 8 : 8, segs);
    uint4 raw[4];
    auto more = [&](const SegmentWalk &w) { return w.u < units && (LANES || w.seg < seg1); };
    auto fetch = [&](const SegmentWalk &w) {
        const int n = w.u * kUnitRows + j, k = w.seg * kSegment + 32 * l;
        const bool in = more(w) && n < N && k < K;
        const uint4 *src = reinterpret_cast<const uint4 *>(W + size_t(n) * K + k);
#pragma unroll
        for (int c = 0; c < 4; ++c) raw[c] = in ? src[c] : make_uint4(0u, 0u, 0u, 0u);
    };
    fetch(at_job);
    while (more(at_job)) {
        const int u = at_job.u, seg = at_job.seg;
        const int n = u * kUnitRows + j, k = seg * kSegment + 32 * l;
        const bool in = n < N && k < K;
        __half s_h, b_h;
        float lo, hi;
        if constexpr (LANES > 0) {
            float hi_scale;
            lanes_range<LANES>(raw, lo, hi, hi_scale);
            range_to_scale(lo, hi_scale, tab.s_factor, tab.top, s_h, b_h);
            const int li = l & (LANES - 1);          // this lane inside its group
            const int g = seg * (4 / LANES) + l / LANES;
            if (in && li == 0) {
                S[size_t(n) * G + g] = s_h;
                qbias[size_t(n) * G + g] = b_h;
            }
            if (in) {   // the group's lanes share out its q + 1 fused scales
                constexpr int sub = 4 / LANES;
                const int per = q + 1;
                uint16_t *tile_scales = reinterpret_cast<uint16_t *>(dst.packed + dst.tile_base(seg >> 2, u) + size_t(q) * 512) +
                                        (size_t(8 * (seg & 3) + j) * sub + tile_phase(sub, j, l / LANES)) * per;
                for (int i = li; i <= q; i += LANES) {
                    uint16_t *to = out.tiled ? tile_scales + i : (i < q ? dst.alpha + (size_t(i) * N + n) * G + g : dst.z + size_t(n) * G + g);
                    *to = fused_scale(s_h, b_h, tab, q, i);
                }
            }
        } else {
            const size_t unit = in ? size_t(n) * G + k / L : 0;
            s_h = S[unit], b_h = qbias[unit];
            lo = __half2float(b_h);
            hi = __half2float(lane_max(raw));   // (a NaN weight in a group that has other numbers shows up here, not in the range)
        }
        const IntDecision<FR> dec(s_h, b_h, lo, hi, tab.top);
        uint2 ints[4];
        // The quotient grows with the weight: where the largest weight's rounds to the top integer or less, every weight's does
        // (with scale factors of 1 and more that is every group but those whose scale is among the smallest numbers).
        if (!VOTE || __any_sync(0xffffffffu, dec.beyond_top(hi))) {
#pragma unroll
            for (int c = 0; c < 4; ++c) ints[c] = piece_ints<FR, true>(raw[c], dec, s_h, b_h, tab.top);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) ints[c] = piece_ints<FR, false>(raw[c], dec, s_h, b_h, tab.top);
        }
        at_job.next();
        fetch(at_job);   // the next job's weights are on their way while this one's planes are put together
        if (w_int && in) {
            uint2 *to = reinterpret_cast<uint2 *>(w_int + size_t(n) * K + k);
#pragma unroll
            for (int c = 0; c < 4; ++c) to[c] = ints[c];
        }
        uint32_t p[4];   // byte i of p[c]: plane i's byte of chunk c
#pragma unroll
        for (int c = 0; c < 4; ++c) p[c] = PAIRS ? chunk_planes_pairs(ints[c], lut) : chunk_planes(ints[c], lut);
        unsigned char *at = out.at(dst, u, seg);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < q) {
                const uint32_t ab = __byte_perm(p[0], p[1], 0x0040u + 0x11u * i), cd = __byte_perm(p[2], p[3], 0x0040u + 0x11u * i);
                const uint32_t w = out.word(__byte_perm(ab, cd, 0x5410u));
                if (in) *reinterpret_cast<uint32_t *>(at + i * stride) = w;
            }
        }
    }
    __threadfence();   // operands visible device-wide before the block counts as finished (products fetch them early)
}

// Parts of a row unit's segments in the forms that take the ranges first: where there are fewer row units than the blocks the
// GPU holds, as many parts as fill it (8 x 131072, one scale per row: 185 us with one block, 34 so; 128 x 28672: 50 and 25).
// At most 16: with one scale per row every part ranges the whole rows.  At least a segment per warp.
static cudaError_t unit_grid(int N, int K, int per_sm, dim3 &grid)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int units = (N + kUnitRows - 1) / kUnitRows, segs = (K + kSegment - 1) / kSegment;
    int parts = sms * per_sm / units;
    parts = parts > 16 ? 16 : parts;
    parts = parts > segs / 8 ? segs / 8 : parts;
    grid = dim3(unsigned(units), unsigned(parts < 1 ? 1 : parts));
    return cudaSuccess;
}

// grid of the one-pass forms: as many blocks as the GPU holds, each walking many jobs (the set-up of a block and its
// closing fence cost about as much as a job)
static cudaError_t walk_grid(int N, int K, int per_sm, dim3 &grid)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long blocks = (segment_jobs(N, K) + 7) / 8, most = static_cast<long long>(sms) * per_sm;
    grid = dim3(unsigned(blocks < most ? blocks : most));
    return cudaSuccess;
}

// Whether warps vote (VOTE above).  With factors above top / (top + 1/2) the largest weight of a group rounds to the top integer, but
// for scales among the smallest numbers, and the comparison is left out nearly everywhere; with smaller factors every group has
// weights beyond the top, and the vote is for nothing.  7168 x 7168, q = 3, tiled, with / without the vote, us:
//   factor 1    groups of 128: 4 bits 44.5 / 47.2, 8 bits 52.3 / 54.2; of 64: 5 bits 49.8 / 51.5; of 32: 5 bits 48.1 / 49.7,
//               8 bits 53.0 / 53.3 (canonical 56.0 / 55.8, of 1024 x 4096 9.53 / 9.43)
//   factor 0.9  groups of 64: 5 bits 52.5 / 51.4, 8 bits 57.6 / 56.5; of 32: 5 bits 51.6 / 50.4, 8 bits 55.6 / 53.9; of 128: 8 bits
//               55.1 / 54.5, but 5 bits 50.2 / 50.7; one scale per row: 8 bits 69.1 / 68.8, but 4 bits 59.8 / 60.7, 5 bits 60.7 / 61.4
static bool rtn_votes(int n_bits, int lanes, double s_factor, double top)
{
    const bool inside = s_factor * (top + 0.5) > top;
    if (n_bits == 8) return inside && lanes != 1;
    return inside || lanes == 4 || lanes == 0;
}

template <int FR, bool PAIRS>
static auto rtn_kernel_of(int lanes, bool votes)
{
    if (lanes == 4) {
        if constexpr (FR == 15)
            if (!votes) return rtn_kernel<FR, 4, PAIRS, false>;
        return rtn_kernel<FR, 4, PAIRS, true>;
    }
    if (lanes == 2) return votes ? rtn_kernel<FR, 2, PAIRS, true> : rtn_kernel<FR, 2, PAIRS, false>;
    if (lanes == 1) {
        if constexpr (FR != 15)
            if (votes) return rtn_kernel<FR, 1, PAIRS, true>;
        return rtn_kernel<FR, 1, PAIRS, false>;
    }
    if constexpr (FR == 15)
        if (!votes) return rtn_kernel<FR, 0, PAIRS, false>;
    return rtn_kernel<FR, 0, PAIRS, true>;
}

template <int FR, bool PAIRS>
static cudaError_t launch_rtn(const __half *w, const QuantTable &tab, int n_bits, __half *s, __half *b, uint8_t *w_int, const View &dst, cudaStream_t st)
{
    const int L = dst.group == 0 ? dst.K : dst.group;
    const int lanes = (L == 128 || L == 64 || L == 32) ? L / 32 : 0;
    dim3 grid;
    const cudaError_t e = lanes ? walk_grid(dst.N, dst.K, 3, grid) : unit_grid(dst.N, dst.K, 3, grid);
    if (e != cudaSuccess) return e;
    const auto kernel = rtn_kernel_of<FR, PAIRS>(lanes, rtn_votes(n_bits, lanes, tab.s_factor, tab.top));
    kernel<<<grid, 256, 0, st>>>(w, tab, L, s, b, w_int, dst);
    return cudaGetLastError();
}

cudaError_t launch_quantize_rtn(const uint16_t *W, int n_bits, double s_factor, const uint8_t *code_of_int /*[256]*/,
                                const double *plane_weight /*[q]*/, uint16_t *S, uint16_t *qbias, uint8_t *w_int,
                                const View &dst, cudaStream_t st)
{
    QuantTable tab;
    for (int t = 0; t < 256; ++t) tab.code_of_int[t] = code_of_int[t];
    for (int j = 0; j < 4; ++j) tab.plane_weight[j] = j < dst.q ? plane_weight[j] : 0.0;
    tab.top = double((1u << n_bits) - 1u);
    tab.centre = tab.top / 2.0;
    tab.s_factor = s_factor;
    const __half *w = reinterpret_cast<const __half *>(W);
    __half *s = reinterpret_cast<__half *>(S), *b = reinterpret_cast<__half *>(qbias);
    // 16 fraction bits leave 7 integer bits in the mantissa
    if (n_bits <= 4) return launch_rtn<16, true>(w, tab, n_bits, s, b, w_int, dst, st);
    return n_bits <= 7 ? launch_rtn<16, false>(w, tab, n_bits, s, b, w_int, dst, st) : launch_rtn<15, false>(w, tab, n_bits, s, b, w_int, dst, st);
}

// ---- step 1 for the search: several scale factors in one pass over W -----------------------------------------------

struct StepOneTable {
    double top;
    double s_factor[kStepOneScales];
    int scales;
};

// Per scale factor f: S (fp16, [N][G], scale_stride elements apart), four times W_int ([N][K] bytes: the search uses it as
// an offset into a table of words) and the residual of step 1, r = S W_int + qbias - W (fp32, rounded to fp16 once, [N][K]).
// A warp takes eight rows of a 128-weight segment, four lanes per row; lane l holds chunks l, l + 4, l + 8, l + 12 of the
// row's 16, so that every load and store covers whole 32-byte sectors (half sectors: 214 us against the 120 of eight
// passes with 32 consecutive weights per lane, 4096 x 4096, eight factors).  UNIT: weights per scaling unit, 128 or 64;
// 0: other multiples of 64, ranges first, a block per row unit (qbias keeps the minima).
template <int UNIT>
__global__ void __launch_bounds__(256, 2) step_one_kernel(const __half *__restrict__ W, const __grid_constant__ StepOneTable tab, int N, int K, int L,
                                                          __half *S, size_t scale_stride, __half *qbias, uint8_t *__restrict__ offsets,
                                                          __half *__restrict__ resid)
{
    const int lane = threadIdx.x & 31, j = lane >> 2, l = lane & 3, warp = threadIdx.x >> 5;
    const int G = K / L, segs = (K + kSegment - 1) / kSegment;
    constexpr bool kOnePass = UNIT != 0;
    constexpr int kParts = UNIT == 128 ? 1 : 2, kChunks = 4 / kParts;   // a segment's parts with scales of their own
    if constexpr (!kOnePass) {
        unit_ranges(W, N, K, L, blockIdx.x, 0, G - 1, [&](int n, int g, int i, float lo, float hi) {
            if (i < tab.scales) {
                __half s_h, b_h;
                range_to_scale(lo, hi, tab.s_factor[i], tab.top, s_h, b_h);
                S[i * scale_stride + size_t(n) * G + g] = s_h;
                if (i == 0) qbias[size_t(n) * G + g] = b_h;
            }
        });
        __syncthreads();
    }
    const int units = kOnePass ? (N + kUnitRows - 1) / kUnitRows : int(blockIdx.x) + 1;
    SegmentWalk at_job(kOnePass ? (long long)blockIdx.x * 8 + warp : (long long)blockIdx.x * segs + warp,
                       kOnePass ? (long long)gridDim.x * 8 : 8, segs);
    const size_t plane = size_t(N) * K;
    for (; at_job.u < units; at_job.next()) {
        const int n = at_job.u * kUnitRows + j;
#pragma unroll
        for (int part = 0; part < kParts; ++part) {
            const int k = at_job.seg * kSegment + 64 * part;   // (K is a multiple of 64)
            const bool in = n < N && k < K;
            const size_t at = in ? size_t(n) * K + k + 8 * l : 0, unit = in ? size_t(n) * G + k / L : 0;
            uint4 raw[kChunks];
#pragma unroll
            for (int c = 0; c < kChunks; ++c) raw[c] = in ? *reinterpret_cast<const uint4 *>(W + at + 32 * c) : make_uint4(0u, 0u, 0u, 0u);
            float lo, hi, hi_scale = 0.f;
            __half b_h = __float2half_rn(0.f);
            if constexpr (kOnePass) {
                lanes_range<4>(raw, lo, hi, hi_scale);
            } else {
                b_h = qbias[unit];
                lo = __half2float(b_h), hi = __half2float(lane_max(raw));
            }
#pragma unroll 1
            for (int f = 0; f < tab.scales; ++f) {
                __half s_h;
                if constexpr (kOnePass) {
                    range_to_scale(lo, hi_scale, tab.s_factor[f], tab.top, s_h, b_h);
                    if (in && l == 0) S[f * scale_stride + unit] = s_h;
                } else {
                    s_h = S[f * scale_stride + unit];
                }
                const IntDecision<16> dec(s_h, b_h, lo, hi, tab.top);
                const float sf = __half2float(s_h), bf = __half2float(b_h);
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    const uint2 ints = piece_ints<16>(raw[c], dec, s_h, b_h, tab.top);
                    const uint32_t word[4] = {raw[c].x, raw[c].y, raw[c].z, raw[c].w};
                    uint32_t out[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 w2 = __half22float2(*reinterpret_cast<const __half2 *>(&word[i]));
                        const uint32_t v4 = i < 2 ? ints.x : ints.y;   // an integer v as the fp32 number 2^23 + v, minus 2^23
                        const float v0 = __uint_as_float(__byte_perm(v4, 0x4B000000u, 0x7650u + ((2 * i) & 3))) - 8388608.f;
                        const float v1 = __uint_as_float(__byte_perm(v4, 0x4B000000u, 0x7650u + ((2 * i + 1) & 3))) - 8388608.f;
                        const __half2 r = __floats2half2_rn(fmaf(sf, v0, bf - w2.x), fmaf(sf, v1, bf - w2.y));
                        out[i] = *reinterpret_cast<const uint32_t *>(&r);
                    }
                    if (in) {
                        *reinterpret_cast<uint2 *>(offsets + f * plane + at + 32 * c) = make_uint2(ints.x << 2, ints.y << 2);
                        *reinterpret_cast<uint4 *>(resid + f * plane + at + 32 * c) = make_uint4(out[0], out[1], out[2], out[3]);
                    }
                }
            }
        }
    }
}

cudaError_t launch_step_one(const uint16_t *W, int N, int K, int group, int n_bits, const double *s_factors, int scales, uint16_t *S,
                            size_t scale_stride, uint16_t *qbias, uint8_t *offsets, uint16_t *resid, cudaStream_t st)
{
    StepOneTable tab;
    tab.top = double((1u << n_bits) - 1u);
    tab.scales = scales;
    for (int f = 0; f < kStepOneScales; ++f) tab.s_factor[f] = f < scales ? s_factors[f] : 1.0;
    const int L = group == 0 ? K : group;
    dim3 grid(unsigned((N + kUnitRows - 1) / kUnitRows));
    if (L == 128 || L == 64) {
        const cudaError_t e = walk_grid(N, K, 2, grid);
        if (e != cudaSuccess) return e;
    }
    const auto kernel = L == 128 ? step_one_kernel<128> : L == 64 ? step_one_kernel<64> : step_one_kernel<0>;
    kernel<<<grid, 256, 0, st>>>(reinterpret_cast<const __half *>(W), tab, N, K, L, reinterpret_cast<__half *>(S), scale_stride,
                                 reinterpret_cast<__half *>(qbias), offsets, reinterpret_cast<__half *>(resid));
    return cudaGetLastError();
}

}  // namespace bcq
