// The coverage count of one tile (warp-level).
#pragma once
#include "raster_common.cuh"
#include "row_span.h"

namespace hexfc {

constexpr int kConsumerWarps = kTilePix / 32;   // warps of the count pass
constexpr int kCountBlocks = 4;                 // its blocks an SM (64 registers a thread; 5: 2-6% slower)
constexpr int kCountSlices = 8;                 // blocks a tile at most

// Per tile: coverage of every chunk of 32 triangles as per-pixel bit masks;
// the masks are kept for the drawing pass and their bit counts are the
// per-pixel list lengths. A warp takes every so-many-th chunk of the tile's list
// on its own: its 32 lanes stage the chunk's triangles, then take the
// triangles' row pairs (clipped to the tile) one per lane: a triangle covers
// one run of samples in a row, found from where its three edges cross the row,
// and the lane writes the runs as bits of the triangle's tile bitmap (256 bits,
// pixel ly * kTileW + lx). Eight 32 x 32 bit transposes turn the 32 bitmaps into
// the 256 pixels' masks. No block barrier until the per-pixel totals are summed.
//
// Bound by instruction issue. What it spends a row on was cut: values that fit 32
// bits (all but triangles that reach 64 pixels beyond the tile's corner), one
// estimate and one exact remainder an edge instead of an error bound and its
// slow path, two rows a lane's turn, a store a row pair instead of an atomic per
// covered sample. 64^3 at 1920x1080 (127,000 chunks): 0.248 -> 0.156 ms; 128^3 at
// 3840x2160: 1.80 -> 1.07 ms.
struct CountWarp {
    int4 edge[3][kChunk];   // stage_edges
    // the chunk's row pairs as one sequence: triangle j's start at seq[j].x; its box seq[j].y. r2j maps
    // the rank of a non-empty triangle to its index.
    uint2 seq[kChunk];
    uint8_t r2j[kChunk];
    uint32_t rows[kTilePix / 32][kChunk];   // [w][j]: pixels 32 w .. of triangle j's bitmap; at the end the
                                            // warp's counts of the 256 pixels
};

// 32 x 32 bit transpose over a warp: bit i of lane l becomes bit l of lane i
// (Warren, Hacker's Delight, section 7-3, with a lane per row).
__device__ __forceinline__ uint32_t warp_transpose(uint32_t v, int lane)
{
    uint32_t o = __shfl_xor_sync(0xffffffffu, v, 16);
    v = __byte_perm(v, o, (lane & 16) ? 0x3276 : 0x5410);
    o = __shfl_xor_sync(0xffffffffu, v, 8);
    v = __byte_perm(v, o, (lane & 8) ? 0x3715 : 0x6240);
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) {
        const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
        o = __shfl_xor_sync(0xffffffffu, v, s);
        v = (lane & s) ? (v & ~m) | ((o >> s) & m) : (v & m) | ((o << s) & ~m);
    }
    return v;
}

__device__ __forceinline__ void count_chunks(CountWarp& me, int lane, const uint32_t* __restrict__ bins,
                                             const FaceFrame* __restrict__ fframe, uint64_t beg, uint32_t n_chunks,
                                             uint32_t first, uint32_t step, int px0, int py0, int W, int H,
                                             uint32_t* __restrict__ masks)
{
    constexpr int kWords = kTilePix / 32;
    using Row = typename std::conditional<kTileW == 8, uint8_t,
                                          typename std::conditional<kTileW == 16, uint16_t, uint32_t>::type>::type;
    constexpr int kRowsPerWord = 32 / kTileW;
    static_assert(kTileW <= 32 && kTileH <= 32, "stage_edges, row_span");
    const int rows = H - py0;   // rows of the image from the tile's first
    uint32_t count[kWords];   // pixels lane + 32 k
#pragma unroll
    for (int k = 0; k < kWords; ++k) count[k] = 0;
    uint32_t f2t = first < n_chunks ? bins[beg + (uint64_t)first * kChunk + lane] : kPadBin;
    for (uint32_t c = first; c < n_chunks; c += step) {
        int4 a = make_int4(0, 0, 0, 0), b = a;
        if (f2t != kPadBin) {
            const Pair16 v = load32(&fframe[f2t >> 1].X);
            a = as_int4(v.a);
            b = as_int4(v.b);
        }
        const uint32_t f2t_next =
            c + step < n_chunks ? bins[beg + (uint64_t)(c + step) * kChunk + lane] : kPadBin;
#pragma unroll
        for (int k = 0; k < kWords; ++k) me.rows[k][lane] = 0u;
        uint32_t box = 0u;
        if (f2t != kPadBin) {
            const bool second = f2t & 1u;
            const int ox = 256 * px0, oy = 256 * py0;
            const int32_t x[3] = {a.x - ox, (second ? a.z : a.y) - ox, (second ? a.w : a.z) - ox};
            const int32_t y[3] = {b.x - oy, (second ? b.z : b.y) - oy, (second ? b.w : b.z) - oy};
            box = stage_edges(x, y, min(kTileW, W - px0), min(kTileH, rows), &me.edge[0][lane], kChunk);
        }
        f2t = f2t_next;
        // the row pairs of the chunk's 32 triangles as one sequence, so that
        // every round gives each lane a pair whatever the boxes' sizes
        const uint32_t rows_l = (uint32_t)box_pairs(box);
        uint32_t incl = rows_l;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t start_l = incl - rows_l, total = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned nonempty = __ballot_sync(0xffffffffu, rows_l != 0);
        me.seq[lane] = make_uint2(start_l, box);
        if (rows_l) me.r2j[__popc(nonempty & ((1u << lane) - 1u))] = (uint8_t)lane;
        __syncwarp();
        for (uint32_t g = 0; g < total; g += 32) {
            // triangles starting in [g, g + 32) (bit = offset) and those before g
            const bool starts = rows_l != 0 && start_l >= g && start_l < g + 32;
            const uint32_t smask = __reduce_or_sync(0xffffffffu, starts ? 1u << (start_l - g) : 0u);
            const int before = __popc(__ballot_sync(0xffffffffu, rows_l != 0 && start_l < g));
            const uint32_t idx = g + (uint32_t)lane;
            if (idx < total) {
                const int n = before + __popc(smask & (0xffffffffu >> (31 - lane)));   // starts in [0, idx]
                const int j = me.r2j[n - 1];
                const uint2 sq = me.seq[j];
                const int ry = 2 * (int)(idx - sq.x), ly = box_ly0(sq.y) + ry;
                int lo0 = box_lx0(sq.y), hi0 = box_lx1(sq.y), lo1 = lo0, hi1 = hi0;
                if (sq.y & kBoxBig) {
                    const int2 s0 = row_span_big(&me.edge[0][j], kChunk, kTileW, ry, lo0, hi0);
                    const int2 s1 = row_span_big(&me.edge[0][j], kChunk, kTileW, ry + 1, lo1, hi1);
                    lo0 = s0.x; hi0 = s0.y;
                    lo1 = s1.x; hi1 = s1.y;
                } else {
                    const int4 e[3] = {me.edge[0][j], me.edge[1][j], me.edge[2][j]};
                    row_span(e, ry, lo0, hi0);
                    row_span(e, ry + 1, lo1, hi1);
                }
                const uint32_t r0 = lo0 <= hi0 ? ((2u << (hi0 - lo0)) - 1u) << lo0 : 0u;
                const uint32_t r1 = lo1 <= hi1 && ly + 1 < rows ? ((2u << (hi1 - lo1)) - 1u) << lo1 : 0u;
                if constexpr (kTileW == 16) {
                    me.rows[ly / 2][j] = r0 | (r1 << 16);
                } else {
                    reinterpret_cast<Row*>(&me.rows[ly / kRowsPerWord][j])[ly % kRowsPerWord] = (Row)r0;
                    reinterpret_cast<Row*>(&me.rows[(ly + 1) / kRowsPerWord][j])[(ly + 1) % kRowsPerWord] = (Row)r1;
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const uint32_t m = warp_transpose(me.rows[k][lane], lane);
            masks[(beg / kChunk + c) * kTilePix + 32 * k + lane] = m;
            count[k] += __popc(m);
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < kWords; ++k) me.rows[k][lane] = count[k];
}

}  // namespace hexfc
