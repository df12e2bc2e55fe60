// The BCQ product on the canonical layout, any shape the layout has (K and the scaling unit multiples of 32, any number of
// rows), 1..16 columns, without a workspace.
//
//   Y[b] = sum_g ( sum_i alpha_i (B_i X[b])_g + z (sum X[b])_g )          (Eq. bcw + Eq. fuse_step3)
//
// The sums go through the tensor cores as in the small-batch kernel: weight bits as sparsity metadata (bcq_mma_core.cuh), 16
// rows x 128 weights x 8 columns per 8 MMAs and plane, also for one column -- direct sign arithmetic takes two instructions
// per weight, plane and column (4096 x 11008, q = 3, one column: 111 us).  A block of eight warps owns 16 rows; its warps
// take the 128-weight segments of K in turn, plane words straight from global memory two segments ahead (rows of the layout
// are only 4-byte aligned), and are added up in a fixed order.  x is staged in operand order, as many windows of 512 as fit
// at a time.  Where 16-row blocks alone do not give every SM one, K is split over the blocks of a cluster, whose sums meet in
// the first one's shared memory, in rank order.
//
// Scaling units: one per row or multiples of 128 are applied to the sum of a segment in fp32; any other multiple of 32 goes
// into the MMAs as the non-zeros, a value per word of 32 weights.  Either way the MMAs add up one segment, the segments are
// added in fp32: the tensor cores cut their running sum off at every step instead of rounding it (2048 x 11008, groups of 32,
// 16 columns: 0.8 % of the outputs were not the correctly rounded ones with sums that ran along K, 0.1 % so).
//
// Bound: the MMAs (26 % of the tensor pipe, seven of eight columns unused at one column) and the latency of plane words and
// scales, with two blocks on some SMs and one on the others.  4096 x 11008, q = 3, groups of 128: 18.4 us at one column (16.2
// with the operand in L2), 21.5 at four.  Scales staged in shared memory, folded into the non-zeros, prefetched into L2, K
// split over more blocks, three blocks per SM: none faster.
#include <cooperative_groups.h>

#include "bcq_mma_core.cuh"

namespace cg = cooperative_groups;

namespace bcq {

constexpr int kCanonWarps = 8;
constexpr int kCanonThreads = kCanonWarps * 32;
constexpr int kCanonSmemBytes = 100 * 1024;   // two blocks per SM
constexpr int kCanonMaxCluster = 8;
constexpr int kCanonSegment = 128;
enum { kScaleRow = 0, kScaleSegment = 1, kScaleWord = 2 };

struct CanonParams {
    const uint8_t *packed;   // [i][n][k / 8]
    const uint16_t *alpha;   // [i][n][g]
    const uint16_t *z;       // [n][g]
    const __half *X;         // [B][K]
    __half *Y;               // [B][N]
    int N, K, B, G, L;       // L weights per scaling unit
    int windows, phase_windows;
    uint32_t ones;           // (1, 1) in fp16
};

template <int Q, int MODE, bool WIDE>
__global__ void __launch_bounds__(kCanonThreads, 2) canon_kernel(const __grid_constant__ CanonParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int BR = WIDE ? 16 : 8, NA = WIDE ? 8 : 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = lane >> 2, t = lane & 3;
    const cg::cluster_group cluster = cg::this_cluster();
    const int ranks = int(cluster.num_blocks()), rank = int(cluster.block_rank());
    const int row0 = int(blockIdx.x) / ranks * 16;
    const int w0 = rank * p.windows / ranks, w1 = (rank + 1) * p.windows / ranks;   // this block's windows of K

    float *part = reinterpret_cast<float *>(smem);                        // [warp][lane][NA]; later the block's sums
    float *xsum = part + kCanonWarps * 32 * NA;                           // [window][word][column]: sums of 32 activations
    unsigned char *xs = reinterpret_cast<unsigned char *>(xsum + size_t(p.phase_windows) * 16 * BR);   // [window][column]

    // this lane's rows (rows beyond N: the last row; not stored) and their planes and scales
    const int n0 = min(row0 + m, p.N - 1), n1 = min(row0 + m + 8, p.N - 1);
    const size_t pitch = size_t(p.K) / 8, plane = size_t(p.N) * pitch, splane = size_t(p.N) * p.G;
    const uint8_t *base0 = p.packed + size_t(n0) * pitch + 4 * t, *base1 = p.packed + size_t(n1) * pitch + 4 * t;
    const uint16_t *al0 = p.alpha + size_t(n0) * p.G, *al1 = p.alpha + size_t(n1) * p.G;
    const uint16_t *z0 = p.z + size_t(n0) * p.G, *z1 = p.z + size_t(n1) * p.G;
    auto h2f = [](uint16_t v) { return __half2float(__ushort_as_half(v)); };

    struct Words {
        uint32_t a[Q], b[Q];   // word t of a segment of rows m and m + 8
    };
    auto fetch = [&](int seg, int end) {
        Words w;
        const bool in = seg < end && seg * kCanonSegment + 32 * t < p.K;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            w.a[i] = in ? __ldg(reinterpret_cast<const uint32_t *>(base0 + i * plane + size_t(seg) * 16)) : 0u;
            w.b[i] = in ? __ldg(reinterpret_cast<const uint32_t *>(base1 + i * plane + size_t(seg) * 16)) : 0u;
        }
        return w;
    };

    struct NonZeros {   // per plane and pair of words: rows m, m + 8 of the first word, then of the second
        uint32_t v[MODE == kScaleWord ? Q : 1][MODE == kScaleWord ? 2 : 1][4];
        __device__ const uint32_t (&operator()(int i, int f) const)[4] { return MODE == kScaleWord ? v[i % (MODE == kScaleWord ? Q : 1)][f % (MODE == kScaleWord ? 2 : 1)] : v[0][0]; }
    } nz;
    if constexpr (MODE != kScaleWord)
#pragma unroll
        for (int e = 0; e < 4; ++e) nz.v[0][0][e] = p.ones;

    const unsigned char *xa0 = xs + (m < p.B ? m : 0) * kXColBytes + t * 16;        // columns beyond B: a staged one; not stored
    const unsigned char *xb0 = xs + (m + 8 < p.B ? m + 8 : 0) * kXColBytes + t * 16;
    float acc[NA], c[Q][4], ch[WIDE ? Q : 1][4];
#pragma unroll
    for (int e = 0; e < NA; ++e) acc[e] = 0.f;
    [[maybe_unused]] uint16_t sc[2][Q + 1];   // the scales of rows m and m + 8 in unit g
    auto fetch_scales = [&](int g) {
#pragma unroll
        for (int i = 0; i < Q; ++i) sc[0][i] = __ldg(al0 + i * splane + g), sc[1][i] = __ldg(al1 + i * splane + g);
        sc[0][Q] = __ldg(z0 + g), sc[1][Q] = __ldg(z1 + g);
    };
    if constexpr (MODE == kScaleRow) fetch_scales(0);
    // acc += a * (lo4, hi4) for the rows of half h
    auto scaled = [&](int h, float a, const float (&lo4)[4], const float (&hi4)[4]) {
        acc[2 * h] = fmaf(a, lo4[2 * h], acc[2 * h]);
        acc[2 * h + 1] = fmaf(a, lo4[2 * h + 1], acc[2 * h + 1]);
        if constexpr (WIDE) {
            acc[4 + 2 * h] = fmaf(a, hi4[2 * h], acc[4 + 2 * h]);
            acc[5 + 2 * h] = fmaf(a, hi4[2 * h + 1], acc[5 + 2 * h]);
        }
    };

    for (int lo = w0; lo < w1; lo += p.phase_windows) {
        // segments 4 lo .. end - 1; the last window's segments beyond K have neither bits nor scales
        const int nw = min(p.phase_windows, w1 - lo), end = min(4 * (lo + nw), (p.K + kCanonSegment - 1) / kCanonSegment);
        int seg = 4 * lo + warp;
        Words cur = fetch(seg, end), next = fetch(seg + kCanonWarps, end);   // on their way while x is staged
        if (lo > w0) __syncthreads();
#pragma unroll 2
        for (int base = warp * 32; base < nw * p.B * 16; base += kCanonThreads) {
            const int task = min(base + lane, nw * p.B * 16 - 1);
            const int st = task & 3, sg = (task >> 2) & 3, wb = task >> 4, w = wb / p.B, b = wb - w * p.B;
            const int k = (lo + w) * kWindow + 128 * sg + 32 * st;
            uint4 raw[4];
            const uint4 *src = reinterpret_cast<const uint4 *>(p.X + size_t(b) * p.K + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) raw[j] = k < p.K ? __ldg(src + j) : make_uint4(0u, 0u, 0u, 0u);   // K is a multiple of 32
            xsum[(w * 16 + sg * 4 + st) * BR + b] = stage_word(raw, xs + size_t(w * p.B + b) * kXColBytes + sg * kXSegBytes, st);
        }
        __syncthreads();
#pragma unroll 1
        for (; seg < end; seg += kCanonWarps) {
            const Words after = fetch(seg + 2 * kCanonWarps, end);
            const int wl = (seg >> 2) - lo, sg = seg & 3;
            const unsigned char *xa = xa0 + size_t(wl * p.B) * kXColBytes + sg * kXSegBytes;
            const unsigned char *xb = xb0 + size_t(wl * p.B) * kXColBytes + sg * kXSegBytes;
            const float *xw = xsum + (wl * 16 + sg * 4) * BR + 2 * t;
            uint32_t bits[Q][2];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                bits[i][0] = __byte_perm(cur.a[i], cur.b[i], 0x5410u);
                bits[i][1] = __byte_perm(cur.a[i], cur.b[i], 0x7632u);
            }
            if constexpr (MODE == kScaleSegment) fetch_scales(seg * kCanonSegment / p.L);   // asked for now, used after the MMAs
            if constexpr (MODE == kScaleWord) {
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const int k = seg * kCanonSegment + 32 * w, g = k / p.L;
                    const bool in = k < p.K;   // words of the last segment beyond K: scales 0
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        nz.v[i][w >> 1][2 * (w & 1)] = in ? __ldg(al0 + i * splane + g) * 0x10001u : 0u;
                        nz.v[i][w >> 1][2 * (w & 1) + 1] = in ? __ldg(al1 + i * splane + g) * 0x10001u : 0u;
                    }
                    const float zz[2] = {in ? h2f(__ldg(z0 + g)) : 0.f, in ? h2f(__ldg(z1 + g)) : 0.f};
                    const float2 xl = *reinterpret_cast<const float2 *>(xw + w * BR);
                    float2 xh = make_float2(0.f, 0.f);
                    if constexpr (WIDE) xh = *reinterpret_cast<const float2 *>(xw + w * BR + 8);
                    const float l4[4] = {xl.x, xl.y, xl.x, xl.y}, h4[4] = {xh.x, xh.y, xh.x, xh.y};
                    scaled(0, zz[0], l4, h4), scaled(1, zz[1], l4, h4);
                }
                segment_sums<Q, WIDE, true>(bits, xa, xb, nz, c, ch);
#pragma unroll
                for (int i = 0; i < Q; ++i) scaled(0, 1.f, c[i], ch[WIDE ? i : 0]), scaled(1, 1.f, c[i], ch[WIDE ? i : 0]);
            } else {
                segment_sums<Q, WIDE, true>(bits, xa, xb, nz, c, ch);
                float4 xt = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float2 xl = *reinterpret_cast<const float2 *>(xw + w * BR);
                    xt.x += xl.x, xt.y += xl.y;
                    if constexpr (WIDE) {
                        const float2 xh = *reinterpret_cast<const float2 *>(xw + w * BR + 8);
                        xt.z += xh.x, xt.w += xh.y;
                    }
                }
                const float l4[4] = {xt.x, xt.y, xt.x, xt.y}, h4[4] = {xt.z, xt.w, xt.z, xt.w};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    scaled(h, h2f(sc[h][Q]), l4, h4);
#pragma unroll
                    for (int i = 0; i < Q; ++i) scaled(h, h2f(sc[h][i]), c[i], ch[WIDE ? i : 0]);
                }
            }
            cur = next, next = after;
        }
    }

    // ---- the warps' sums in order, then the cluster's ------------------------------------------------------------
#pragma unroll
    for (int e = 0; e < NA; ++e) part[(warp * 32 + lane) * NA + e] = acc[e];
    __syncthreads();
    constexpr int kOut = 32 * NA;   // one thread per output
    static_assert(kOut <= kCanonThreads, "outputs");
    float v = 0.f;
    if (tid < kOut) {
        v = part[tid];
#pragma unroll
        for (int w = 1; w < kCanonWarps; ++w) v += part[w * kOut + tid];
    }
    if (ranks > 1) {
        if (tid < kOut) part[tid] = v;
        cluster.sync();
        if (rank == 0 && tid < kOut)
            for (int r = 1; r < ranks; ++r) v += cluster.map_shared_rank(part, r)[tid];
        cluster.sync();   // the other blocks' shared memory stays until it has been read
        if (rank != 0) return;
    }
    if (tid < kOut) {
        const int l = tid / NA, e = tid % NA;
        const int n = row0 + 8 * ((e >> 1) & 1) + (l >> 2), b = 8 * (e >> 2) + 2 * (l & 3) + (e & 1);
        if (n < p.N && b < p.B) p.Y[size_t(b) * p.N + n] = __float2half_rn(v);
    }
}

template <int Q, int MODE, bool WIDE>
static cudaError_t launch_canon_q(CanonParams prm, cudaStream_t st)
{
    constexpr int BR = WIDE ? 16 : 8, NA = WIDE ? 8 : 4;
    static bool configured[64] = {};   // the shared-memory opt-in is per function and per device
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(canon_kernel<Q, MODE, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCanonSmemBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    const int blocks = (prm.N + 15) / 16;
    // K over as many blocks as leave one per SM (measured: 94 blocks 3.3 us unsplit, 4.1 and 6.6 as 2 and 3 ranks; 64 blocks
    // 5.1 us unsplit, 4.8 as 2; 19 blocks of 22 windows 9.4 us unsplit, 4.7 as 6, 5.5 as 8)
    int ranks = sms / blocks;
    ranks = ranks < 1 ? 1 : (ranks > kCanonMaxCluster ? kCanonMaxCluster : ranks);
    if (ranks > prm.windows) ranks = prm.windows;
    const int each = (prm.windows + ranks - 1) / ranks;
    const int fixed = kCanonWarps * 32 * NA * int(sizeof(float)), per_window = prm.B * kXColBytes + 16 * BR * int(sizeof(float));
    prm.phase_windows = (kCanonSmemBytes - fixed) / per_window;
    if (prm.phase_windows > each) prm.phase_windows = each;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(blocks) * unsigned(ranks));
    cfg.blockDim = dim3(kCanonThreads);
    cfg.dynamicSmemBytes = size_t(fixed) + size_t(prm.phase_windows) * per_window;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(ranks), attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, canon_kernel<Q, MODE, WIDE>, prm);
}

template <int Q>
static cudaError_t launch_canon_sel(const CanonParams &prm, int mode, cudaStream_t st)
{
    const bool wide = prm.B > 8;
    if (mode == kScaleRow) return wide ? launch_canon_q<Q, kScaleRow, true>(prm, st) : launch_canon_q<Q, kScaleRow, false>(prm, st);
    if (mode == kScaleSegment) return wide ? launch_canon_q<Q, kScaleSegment, true>(prm, st) : launch_canon_q<Q, kScaleSegment, false>(prm, st);
    return wide ? launch_canon_q<Q, kScaleWord, true>(prm, st) : launch_canon_q<Q, kScaleWord, false>(prm, st);
}

cudaError_t launch_canon(const bcq_desc &d, const void *packed, const uint16_t *alpha, const uint16_t *z, const uint16_t *X, uint16_t *Y, int B,
                         cudaStream_t st)
{
    CanonParams prm = {};
    prm.packed = static_cast<const uint8_t *>(packed);
    prm.alpha = alpha, prm.z = z;
    prm.X = reinterpret_cast<const __half *>(X);
    prm.Y = reinterpret_cast<__half *>(Y);
    prm.N = d.N, prm.K = d.K, prm.B = B, prm.G = n_groups(d), prm.L = d.K / prm.G;
    prm.windows = (d.K + kWindow - 1) / kWindow;
    prm.ones = 0x3C003C00u;
    const int mode = prm.G == 1 ? kScaleRow : (prm.L % kCanonSegment == 0 ? kScaleSegment : kScaleWord);
    switch (d.q) {
        case 1: return launch_canon_sel<1>(prm, mode, st);
        case 2: return launch_canon_sel<2>(prm, mode, st);
        case 3: return launch_canon_sel<3>(prm, mode, st);
        case 4: return launch_canon_sel<4>(prm, mode, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace bcq
