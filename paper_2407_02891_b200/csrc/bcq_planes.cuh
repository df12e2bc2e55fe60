// How the preparation kernels write bit planes.  A warp owns eight rows (one row unit of the tiled layout) of one
// 128-weight segment of K: lane 4 j + l holds weights 32 l .. 32 l + 31 of the segment of row j, i.e. one 32-bit word
// per plane (four chunks of eight weights).  In the tiled layout the four words of a row are the 16 bytes of its tile
// lane, permuted in halves of a word (tile_chunk pairs chunks 2 p, 2 p + 1), and the warp's 32 words of a plane are 128
// consecutive bytes: two shuffles and a byte-permute turn the words into the tile's own words, so that a plane leaves
// the warp as one full 128-byte store instead of 128 single bytes.  In the canonical layout the words are stored as they
// are (16 consecutive bytes per row).
#pragma once
#include "bcq_internal.cuh"

namespace bcq {

constexpr int kSegment = 128;   // weights along K per warp and step

__host__ __device__ inline long long segment_jobs(int N, int K)   // (row unit, segment) pairs
{
    return (long long)((N + kUnitRows - 1) / kUnitRows) * ((K + kSegment - 1) / kSegment);
}

// A warp's walk over the (row unit, segment) pairs, segments fastest, `stride` pairs at a time; divisions once, at the
// start (a 64-bit division per step would cost as much as a third of a step's work).
struct SegmentWalk {
    int u, seg, segs, du, dseg;
    __device__ SegmentWalk(long long first, long long stride, int segs_)
        : u(int(first / segs_)), seg(int(first % segs_)), segs(segs_), du(int(stride / segs_)), dseg(int(stride % segs_))
    {
    }
    __device__ void next()
    {
        u += du, seg += dseg;
        if (seg >= segs) seg -= segs, ++u;
    }
};

struct PlaneWriter {
    int src0, src1;      // lanes that hold the two halves of this lane's stored word
    uint32_t sel;        // which half of each
    bool tiled;

    __device__ explicit PlaneWriter(const View &v)
    {
        const int lane = threadIdx.x & 31, j = lane >> 2, l = lane & 3, sub = v.subs();
        tiled = v.layout == BCQ_LAYOUT_TILED;
        const int p0 = tile_chunk(sub, j, 4 * l) >> 1, p1 = tile_chunk(sub, j, 4 * l + 2) >> 1;
        src0 = 4 * j + (p0 >> 1), src1 = 4 * j + (p1 >> 1);
        sel = ((p0 & 1) ? 0x32u : 0x10u) | ((p1 & 1) ? 0x7600u : 0x5400u);
        if (!tiled) src0 = src1 = lane, sel = 0x3210u;
    }
    // where plane 0's word of this lane goes (row unit u, segment seg)
    __device__ unsigned char *at(const View &v, int u, int seg) const
    {
        const int lane = threadIdx.x & 31, j = lane >> 2, l = lane & 3;
        if (tiled) return v.packed + v.tile_base(seg >> 2, u) + size_t(8 * (seg & 3) + j) * 16 + 4 * l;
        return v.packed + size_t(u * kUnitRows + j) * size_t(v.K / 8) + size_t(seg) * (kSegment / 8) + 4 * l;
    }
    // the word this lane stores (all lanes of the warp take part)
    __device__ uint32_t word(uint32_t mine) const
    {
        if (!tiled) return mine;
        const uint32_t a = __shfl_sync(0xffffffffu, mine, src0), b = __shfl_sync(0xffffffffu, mine, src1);
        return __byte_perm(a, b, sel);
    }
};

}  // namespace bcq
