// Operand preparation kernels: linear-int -> merged binary code (Eq. round, Eq. fuse_step3),
// code -> bit-plane packing, and the canonical <-> tiled permutations.  All run once per
// layer, offline.
#include "bcq_planes.cuh"

namespace bcq {

// ---- merge ---------------------------------------------------------------------------------

struct MergeTable {
    uint8_t code_of_int[256];  // code of the reachable integer nearest to each step-1 integer
    double plane_weight[4];    // m_j = sum of 2^(i-2) over the step-1 bits i of plane j
    double centre;             // (2^n - 1) / 2
};

// codes[t] = code of w_int[t], 16 per thread and step (one 16-byte load and store; the 256-byte table sits in shared
// memory, conflict-free up to 7 step-1 bits), and, by the blocks from code_blocks on, the fused scales:
// alpha_j = S * m_j and z = S * centre + qbias, each evaluated exactly in fp64 (the products and the sum of two
// fp16-derived values fit 53 bits) and rounded once to fp16.  Bound by the look-ups (load and store pipe 69 % busy at
// 7168 x 7168, 19.6 us) beside HBM (38 %): one byte in, one byte out per weight.
__global__ void __launch_bounds__(256) merge_kernel(const uint4 *__restrict__ w_int, uint4 *__restrict__ codes, size_t pieces, int code_blocks,
                                                    const __half *__restrict__ S, const __half *__restrict__ qbias, size_t units, int q,
                                                    __half *__restrict__ alpha, __half *__restrict__ z, const __grid_constant__ MergeTable tab)
{
    if (int(blockIdx.x) >= code_blocks) {
        const size_t t = size_t(blockIdx.x - code_blocks) * blockDim.x + threadIdx.x;
        if (t >= units) return;
        const double s = double(__half2float(S[t]));
        const double b = double(__half2float(qbias[t]));
        for (int j = 0; j < q; ++j) alpha[size_t(j) * units + t] = __double2half(s * tab.plane_weight[j]);
        z[t] = __double2half(s * tab.centre + b);
        return;
    }
    __shared__ uint8_t lut[256];
    lut[threadIdx.x] = tab.code_of_int[threadIdx.x];
    __syncthreads();
    auto look4 = [&](uint32_t w) {
        const uint32_t a = lut[w & 0xffu], b = lut[(w >> 8) & 0xffu], c = lut[(w >> 16) & 0xffu], d = lut[w >> 24];
        return __byte_perm(__byte_perm(a, b, 0x0040u), __byte_perm(c, d, 0x0040u), 0x5410u);
    };
    const size_t stride = size_t(code_blocks) * 256;
    for (size_t t = size_t(blockIdx.x) * 256 + threadIdx.x; t < pieces; t += 2 * stride) {
        const bool two = t + stride < pieces;
        const uint4 v = w_int[t];
        uint4 v2 = make_uint4(0u, 0u, 0u, 0u);
        if (two) v2 = w_int[t + stride];
        codes[t] = make_uint4(look4(v.x), look4(v.y), look4(v.z), look4(v.w));
        if (two) codes[t + stride] = make_uint4(look4(v2.x), look4(v2.y), look4(v2.z), look4(v2.w));
    }
}

cudaError_t launch_merge(const bcq_desc &d, const uint8_t *w_int, const uint16_t *S, const uint16_t *qbias, int n_bits,
                         const uint8_t *code_of_int, const double *plane_weight, uint8_t *codes, uint16_t *alpha,
                         uint16_t *z, cudaStream_t st)
{
    MergeTable tab;
    for (int t = 0; t < 256; ++t) tab.code_of_int[t] = code_of_int[t];
    for (int j = 0; j < 4; ++j) tab.plane_weight[j] = j < d.q ? plane_weight[j] : 0.0;
    tab.centre = (double((1u << n_bits) - 1u)) / 2.0;
    const size_t pieces = size_t(d.N) * d.K / 16;   // K is a multiple of 32
    const size_t units = size_t(d.N) * n_groups(d);
    const size_t wanted = (pieces + 511) / 512;      // two pieces per thread
    const int code_blocks = int(wanted < 65536 ? wanted : 65536);
    const unsigned scale_blocks = unsigned((units + 255) / 256);
    merge_kernel<<<unsigned(code_blocks) + scale_blocks, 256, 0, st>>>(
        reinterpret_cast<const uint4 *>(w_int), reinterpret_cast<uint4 *>(codes), pieces, code_blocks, reinterpret_cast<const __half *>(S),
        reinterpret_cast<const __half *>(qbias), units, d.q, reinterpret_cast<__half *>(alpha), reinterpret_cast<__half *>(z), tab);
    return cudaGetLastError();
}

// ---- pack ------------------------------------------------------------------------------------
//
// A warp packs one (row unit, segment) at a time: 32 codes per lane (two 16-byte loads).  Codes are at most 4 bits, so
// eight of them fit one word (two nibbles per byte); plane i of the eight is one shift, one AND and one multiplication
// that gathers the eight bits into the top byte (the products of the other bits fall below it or out of the word, and
// no two of them meet).  A block walks many jobs, the next job's codes on their way while one is packed: a block's
// closing fence costs more than a job.  Bound by instruction issue (slots 63 % busy, 264 instructions per job) and the
// latency of the codes (a third of a warp's time), HBM 31 % busy (codes not in L2).  Merge and pack of 7168 x 7168, q = 3,
// groups of 128: 212 us as one byte per thread and store, in four launches; 44 us so.

__device__ __forceinline__ uint32_t plane_word(const uint32_t (&z)[4], int i)
{
    uint32_t p[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) p[c] = ((z[c] >> i) & 0x11111111u) * 0x01020408u;   // chunk c's byte on top
    return __byte_perm(__byte_perm(p[0], p[1], 0x0073u), __byte_perm(p[2], p[3], 0x0073u), 0x5410u);
}

// Q planes; SUB: scaling units per segment when the canonical scales (alpha, z) go into the tiles, else 0.
template <int Q, int SUB>
__global__ void __launch_bounds__(256, 4) pack_kernel(const uint8_t *__restrict__ codes, const uint16_t *__restrict__ alpha,
                                                   const uint16_t *__restrict__ z, const View dst)
{
    const int lane = threadIdx.x & 31, j = lane >> 2, l = lane & 3;
    const PlaneWriter out(dst);
    const int segs = (dst.K + kSegment - 1) / kSegment;
    const size_t stride = dst.plane_stride();
    const int units = (dst.N + kUnitRows - 1) / kUnitRows;
    // scales: the quad's lanes share out the (Q + 1) values of each of the row's scaling units in the segment
    constexpr int kValues = SUB * (Q + 1), kPer = (kValues + 3) / 4;
    [[maybe_unused]] const uint16_t *from[kPer > 0 ? kPer : 1];   // row j's value of row unit 0, segment 0
    [[maybe_unused]] int to[kPer > 0 ? kPer : 1];                 // its place in the tile's scales
    if constexpr (SUB > 0) {
#pragma unroll
        for (int v = 0; v < kPer; ++v) {
            const int e = min(l + 4 * v, kValues - 1), sg = e / (Q + 1), i = e % (Q + 1);
            from[v] = (i < Q ? alpha + size_t(i) * dst.N * dst.G() : z) + size_t(j) * dst.G() + sg;
            to[v] = (j * SUB + tile_phase(SUB, j, sg)) * (Q + 1) + i;
        }
    }
    SegmentWalk at_job((long long)blockIdx.x * 8 + (threadIdx.x >> 5), (long long)gridDim.x * 8, segs);
    uint4 a, b;
    auto fetch = [&](const SegmentWalk &w) {
        const int n = w.u * kUnitRows + j, k = w.seg * kSegment + 32 * l;
        a = make_uint4(0u, 0u, 0u, 0u), b = a;
        if (n < dst.N && k < dst.K) {
            const uint4 *src = reinterpret_cast<const uint4 *>(codes + size_t(n) * dst.K + k);
            a = src[0], b = src[1];
        }
    };
    fetch(at_job);
    while (at_job.u < units) {
        const int u = at_job.u, seg = at_job.seg;
        const bool in = u * kUnitRows + j < dst.N && seg * kSegment + 32 * l < dst.K;
        const uint32_t lo = 0x0f0f0f0fu;
        const uint32_t z8[4] = {(a.x & lo) | ((a.y & lo) << 4), (a.z & lo) | ((a.w & lo) << 4), (b.x & lo) | ((b.y & lo) << 4),
                                (b.z & lo) | ((b.w & lo) << 4)};
        at_job.next();
        fetch(at_job);
        unsigned char *at = out.at(dst, u, seg);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const uint32_t w = out.word(plane_word(z8, i));
            if (in) *reinterpret_cast<uint32_t *>(at + i * stride) = w;
        }
        if constexpr (SUB > 0) {
            uint16_t *sp = reinterpret_cast<uint16_t *>(dst.packed + dst.tile_base(seg >> 2, u) + size_t(Q) * 512) + 8 * (seg & 3) * kValues;
            const size_t at_unit = size_t(u) * kUnitRows * dst.G() + size_t(seg) * SUB;
#pragma unroll
            for (int v = 0; v < kPer; ++v)
                if (l + 4 * v < kValues) sp[to[v]] = from[v][at_unit];
        }
    }
    // The products start fetching packed operands before they wait for the kernel in front of them: every
    // kernel that writes operands makes its writes visible device-wide before its blocks count as finished.
    __threadfence();
}

template <int Q>
static void launch_pack_q(int sub, unsigned grid, const uint8_t *codes, const uint16_t *alpha, const uint16_t *z, const View &dst, cudaStream_t st)
{
    switch (sub) {
        case 1: pack_kernel<Q, 1><<<grid, 256, 0, st>>>(codes, alpha, z, dst); break;
        case 2: pack_kernel<Q, 2><<<grid, 256, 0, st>>>(codes, alpha, z, dst); break;
        case 4: pack_kernel<Q, 4><<<grid, 256, 0, st>>>(codes, alpha, z, dst); break;
        default: pack_kernel<Q, 0><<<grid, 256, 0, st>>>(codes, alpha, z, dst); break;
    }
}

// alpha_in, z_in: canonical scales that travel inside the tiles, or null
cudaError_t launch_pack(const uint8_t *codes, const uint16_t *alpha_in, const uint16_t *z_in, const View &dst, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // as many blocks as the GPU holds, each walking many jobs: a block's closing fence costs more than a job
    const long long blocks = (segment_jobs(dst.N, dst.K) + 7) / 8;
    const unsigned grid = unsigned(blocks < sms * 4LL ? blocks : sms * 4LL);
    const int sub = alpha_in ? dst.subs() : 0;
    switch (dst.q) {
        case 1: launch_pack_q<1>(sub, grid, codes, alpha_in, z_in, dst, st); break;
        case 2: launch_pack_q<2>(sub, grid, codes, alpha_in, z_in, dst, st); break;
        case 3: launch_pack_q<3>(sub, grid, codes, alpha_in, z_in, dst, st); break;
        default: launch_pack_q<4>(sub, grid, codes, alpha_in, z_in, dst, st); break;
    }
    return cudaGetLastError();
}

// ---- permutations between layouts -----------------------------------------------------------

__global__ void permute_planes_kernel(const View src, const View dst)
{
    const int kbytes = src.K / 8;
    size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= size_t(src.q) * src.N * kbytes) return;
    const int kb = int(t % kbytes);
    const int n = int((t / kbytes) % src.N);
    const int i = int(t / (size_t(kbytes) * src.N));
    *dst.plane_byte(i, n, kb) = *src.plane_byte(i, n, kb);
    __threadfence();   // see pack_kernel
}

__global__ void permute_scales_kernel(const View src, const View dst)
{
    const int G = src.G();
    size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= size_t(src.N) * G) return;
    const int n = int(t / G), g = int(t % G);
    for (int i = 0; i < src.q; ++i) *dst.alpha_elem(i, n, g) = *src.alpha_elem(i, n, g);
    *dst.z_elem(n, g) = *src.z_elem(n, g);
    __threadfence();   // see pack_kernel
}

cudaError_t launch_permute_planes(const View &src, const View &dst, cudaStream_t st)
{
    size_t count = size_t(src.q) * src.N * (src.K / 8);
    permute_planes_kernel<<<unsigned((count + 255) / 256), 256, 0, st>>>(src, dst);
    return cudaGetLastError();
}

cudaError_t launch_permute_scales(const View &src, const View &dst, cudaStream_t st)
{
    size_t count = size_t(src.N) * src.G();
    permute_scales_kernel<<<unsigned((count + 255) / 256), 256, 0, st>>>(src, dst);
    return cudaGetLastError();
}

}  // namespace bcq
