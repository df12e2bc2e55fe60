// The tensor-core form of the BCQ product, shared by the tiled and the canonical kernel.
//
// The weight bits ARE the operand: mma.sp m16n8k32 multiplies a matrix with two non-zeros in every four columns, whose
// positions are given by two metadata bits each.  With the rows of B laid out as (-x_0, x_0, -x_1, x_1), ... and all
// non-zeros 1, the first non-zero of a four sits at position 0 or 1 and the second at 2 or 3 according to one weight bit
// each: metadata = weight bits spread to the even bit positions, with the odd positions of the second non-zeros set.
// A 16-bit piece of a plane (rows m in the lower, m + 8 in the upper half of a word) makes two metadata words -- its even
// and its odd bits -- with three logic operations, and each serves two MMAs (the instruction takes its metadata from lanes
// t = 0, 1 or 2, 3 of every four).  Products are exact (+-1 times fp16 x), sums fp32; the scale is applied in fp32 to the
// sum of 128 weights.
//
// Why this form: expanding bits to fp16 numbers +-alpha costs a shift and a logic operation per register of two weights,
// half-rate instructions both (16 dispatch cycles per MMA of 8); one logic operation per register (a bit as sign, exponent
// or mantissa bit, bases subtracted) came to 13.2 cycles per MMA.  Metadata: 1 operation per MMA; mma.sp itself issues
// every 9 cycles per SM sub-partition.
#pragma once
#include "bcq_async.cuh"
#include "bcq_internal.cuh"

namespace bcq {

constexpr int kXSegBytes = 256;          // operand-ordered x of one (column, 128-weight segment): 4 step pairs x 4 lanes x 16 bytes
constexpr int kXColBytes = 4 * kXSegBytes + 64;   // of one (column, window), padded: conflict-free 16-byte loads

// The B operand of one step: (-x, x) for each of four activations, by a packed multiplication each.  (Staged in that form
// the loads of x keep the shared-memory pipe 60 % busy and half as many windows' x fit: no faster, 16 columns slower.)
__device__ __forceinline__ uint4 signed_pairs(uint32_t x01, uint32_t x23)
{
    const __half2 sign = __halves2half2(__ushort_as_half((unsigned short)0xBC00u), __ushort_as_half((unsigned short)0x3C00u));   // (-1, 1)
    const __half2 a = *reinterpret_cast<const __half2 *>(&x01), b = *reinterpret_cast<const __half2 *>(&x23);
    const __half2 r[4] = {__hmul2(__low2half2(a), sign), __hmul2(__high2half2(a), sign), __hmul2(__low2half2(b), sign), __hmul2(__high2half2(b), sign)};
    return make_uint4(*reinterpret_cast<const uint32_t *>(&r[0]), *reinterpret_cast<const uint32_t *>(&r[1]), *reinterpret_cast<const uint32_t *>(&r[2]),
                      *reinterpret_cast<const uint32_t *>(&r[3]));
}

template <int F>   // F: metadata from lanes t = 0, 1 (0) or t = 2, 3 (1) of every four
__device__ __forceinline__ void mma_sp(float (&d)[4], const uint32_t (&a)[4], const uint4 &b, uint32_t meta, float c0, float c1, float c2, float c3)
{
    asm("mma.sp::ordered_metadata.sync.aligned.m16n8k32.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9,%10,%11}, "
        "{%12,%13,%14,%15}, %16, %17;"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w), "f"(c0), "f"(c1), "f"(c2), "f"(c3), "r"(meta),
          "n"(F));
}

// Sums of one 128-weight segment: c[i][.] += the non-zeros a (1, or the weights' scale) times plane i's signs times x, for
// rows m and m + 8 and columns 2t, 2t + 1 (ch: columns 8 + those).  Lane (m = lane / 4, t = lane % 4) gives
// z[i][h], the bits of chunks 4 t + 2 h and the next one (16 weights from 32 t + 16 h on) of rows m (lower half) and m + 8
// (upper half); xa / xb: its 16-byte pieces of the staged x of columns m and m + 8.  a: per plane; [f] = the non-zeros
// of the weights of lanes 2 f (a[0], a[1]: rows m, m + 8) and 2 f + 1 (a[2], a[3]).  FIRST: the sums start at 0.
template <int Q, bool WIDE, bool FIRST, class A>
__device__ __forceinline__ void segment_sums(const uint32_t (&z)[Q][2], const unsigned char *xa, const unsigned char *xb, const A &a,
                                             float (&c)[Q][4], float (&ch)[WIDE ? Q : 1][4])
{
    static_for<0, 2>([&](auto H) {
        constexpr int h = decltype(H)::value;
        static_for<0, 2>([&](auto O) {
            constexpr int o = decltype(O)::value;   // even or odd bits
            uint32_t meta[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) meta[i] = ((o ? z[i][h] >> 1 : z[i][h]) & 0x55555555u) | 0x88888888u;
            const uint4 xr = *reinterpret_cast<const uint4 *>(xa + (h * 2 + o) * 64);
            uint4 yr = make_uint4(0u, 0u, 0u, 0u);
            if constexpr (WIDE) yr = *reinterpret_cast<const uint4 *>(xb + (h * 2 + o) * 64);
            static_for<0, 2>([&](auto FF) {
                constexpr int f = decltype(FF)::value;
                constexpr bool start = FIRST && h == 0 && o == 0 && f == 0;
                const uint4 x = f == 0 ? signed_pairs(xr.x, xr.y) : signed_pairs(xr.z, xr.w);
                uint4 y = make_uint4(0u, 0u, 0u, 0u);
                if constexpr (WIDE) y = f == 0 ? signed_pairs(yr.x, yr.y) : signed_pairs(yr.z, yr.w);
                static_for<0, Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    if constexpr (start)
                        mma_sp<f>(c[i], a(i, f), x, meta[i], 0.f, 0.f, 0.f, 0.f);
                    else
                        mma_sp<f>(c[i], a(i, f), x, meta[i], c[i][0], c[i][1], c[i][2], c[i][3]);
                    if constexpr (WIDE) {
                        if constexpr (start)
                            mma_sp<f>(ch[i], a(i, f), y, meta[i], 0.f, 0.f, 0.f, 0.f);
                        else
                            mma_sp<f>(ch[i], a(i, f), y, meta[i], ch[i][0], ch[i][1], ch[i][2], ch[i][3]);
                    }
                });
            });
        });
    });
}

// Stage 32 activations (weights 32 w .. 32 w + 31 of a segment, one column) in operand order; returns their sum.
// Activation 16 h + 2 i + o of them is number 4 (w / 2) + 2 (w % 2) + i / 4 of lane t = i % 4 at step pair (h, o).
__device__ __forceinline__ float stage_word(const uint4 (&src)[4], unsigned char *dst, int w)
{
    const uint32_t x2[16] = {src[0].x, src[0].y, src[0].z, src[0].w, src[1].x, src[1].y, src[1].z, src[1].w,
                             src[2].x, src[2].y, src[2].z, src[2].w, src[3].x, src[3].y, src[3].z, src[3].w};
    float sum = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int o = 0; o < 2; ++o)
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint32_t out = __byte_perm(x2[8 * h + t], x2[8 * h + t + 4], o ? 0x7632u : 0x5410u);   // i = t and t + 4
                *reinterpret_cast<uint32_t *>(dst + (h * 2 + o) * 64 + t * 16 + w * 4) = out;
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&out));
                sum += f.x + f.y;
            }
    return sum;
}

}  // namespace bcq
