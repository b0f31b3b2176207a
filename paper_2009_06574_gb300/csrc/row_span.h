// The samples of a raster tile that a triangle covers, a row at a time: edge
// values set up once for the tile, then the covered columns of any row, exact.
// Compiles for the device and, for tests, for the host.
#pragma once
#include <stdint.h>

#include <cstring>

#if defined(__CUDACC__)
#define HEXFC_ROW __device__ __forceinline__
#define HEXFC_ROW_COLD static __device__ __noinline__
#else
#include <algorithm>
#define HEXFC_ROW inline
#define HEXFC_ROW_COLD inline
#endif

namespace hexfc {

#if !defined(__CUDACC__)
// the device's names
using std::max;
using std::min;
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
inline int2 make_int2(int x, int y) { return int2{x, y}; }
inline float __int_as_float(int v) { float f; std::memcpy(&f, &v, 4); return f; }
inline int __float_as_int(float f) { int v; std::memcpy(&v, &f, 4); return v; }
inline float __fdividef(float a, float b) { return a / b; }
inline float __saturatef(float v) { return std::min(std::max(v, 0.f), 1.f); }
#endif

// A triangle's box in the tile: first column, first row (even), last column, row
// pairs (0: no samples); whether its values need 64 bits.
constexpr uint32_t kBoxBig = 1u << 31;
HEXFC_ROW int box_lx0(uint32_t b) { return (int)(b & 255u); }
HEXFC_ROW int box_ly0(uint32_t b) { return (int)((b >> 8) & 255u); }
HEXFC_ROW int box_lx1(uint32_t b) { return (int)((b >> 16) & 255u); }
HEXFC_ROW int box_pairs(uint32_t b) { return (int)((b >> 24) & 127u); }

// Corners on the tile's samples or at most this far from its corner (16.8): every
// edge value at a sample of the tile is below 2 * 2^15 * (2^14 + 2^13) < 2^31.
constexpr int32_t kSmallTri = 16384;

// Triangle with corners (x, y), 16.8 and relative to the tile's corner (below 2^24
// in magnitude), in a tile of cols x rows samples (at most 32 x 32): its box, and
// per edge k its row data: value at column 0 of the box' first row, 256 dx, 256 dy
// (edge vector), 1 / (64 * 256 dy) as float bits; for a large triangle low word, dx,
// dy, high word. The value is exact, and less by one where the top-left rule does
// not give the edge's own samples to the triangle, so that a sample is inside iff
// no value is negative. Edge k goes to edge[k * stride].
HEXFC_ROW uint32_t stage_edges(const int32_t xin[3], const int32_t yin[3], int cols, int rows, int4* edge,
                               int stride)
{
    int32_t x[3] = {xin[0], xin[1], xin[2]}, y[3] = {yin[0], yin[1], yin[2]};
    const int64_t area = (int64_t)(x[1] - x[0]) * (y[2] - y[0]) - (int64_t)(y[1] - y[0]) * (x[2] - x[0]);
    if (area < 0) {   // wound to positive area
        const int32_t tx = x[1], ty = y[1];
        x[1] = x[2]; y[1] = y[2];
        x[2] = tx; y[2] = ty;
    }
    const int32_t xmin = min(x[0], min(x[1], x[2])), xmax = max(x[0], max(x[1], x[2]));
    const int32_t ymin = min(y[0], min(y[1], y[2])), ymax = max(y[0], max(y[1], y[2]));
    // sample p has its centre at 256 p + 128
    const int x0 = max((xmin + 127) >> 8, 0), x1 = min((xmax - 128) >> 8, cols - 1);
    const int y0 = max((ymin + 127) >> 8, 0), y1 = min((ymax - 128) >> 8, rows - 1);
    if (area == 0 || x0 > x1 || y0 > y1) return 0u;
    const bool big = xmin < -kSmallTri || ymin < -kSmallTri || xmax > kSmallTri || ymax > kSmallTri;
    const int yf = y0 & ~1;   // row pairs start at even rows
    const int32_t sx = 128, sy = 256 * yf + 128;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int ia = (k + 1) % 3, ib = (k + 2) % 3;
        const int32_t dx = x[ib] - x[ia], dy = y[ib] - y[ia];
        const int own = (dy < 0) || (dy == 0 && dx > 0) ? 0 : 1;   // the edge's own samples: top-left rule
        int4 e;
        if (!big) {
            e.x = dx * (sy - y[ia]) - dy * (sx - x[ia]) - own;
            e.y = dx * 256;
            e.z = dy * 256;
            e.w = __float_as_int(__fdividef(1.f, 16384.f * (float)dy));
            if (dy == 0) {   // the sign is all that matters: odd values, far from 0 in units of 1/64
                e.x = 2 * (dx > 0 ? sy - y[ia] : y[ia] - sy) + 1 - 2 * own;
                e.y = dx > 0 ? 512 : -512;
                e.w = __float_as_int(1.f);
            }
        } else {
            const int64_t v = (int64_t)dx * (sy - y[ia]) - (int64_t)dy * (sx - x[ia]) - own;
            e.x = (int32_t)(uint32_t)v;
            e.y = dx;
            e.z = dy;
            e.w = (int32_t)(v >> 32);
        }
        edge[k * stride] = e;
    }
    return (uint32_t)x0 | ((uint32_t)yf << 8) | ((uint32_t)x1 << 16) | ((uint32_t)((y1 - yf) / 2 + 1) << 24) |
           (big ? kBoxBig : 0u);
}

// The covered columns [lo, hi] of the tile's row ry below the triangle's first
// (empty if lo > hi), within [lo, hi] as they come in. An edge's value at column c
// is A - D c, so it crosses zero at A / D: the nearest whole number q in [-32, 32]
// to a float estimate of it (within 2^-15 of it in that range) and the exact value
// there, A - D q, give the last or first column inside.
HEXFC_ROW void row_span(const int4 e[3], int ry, int& lo, int& hi)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int32_t A = e[k].x + e[k].y * ry;
        const float t = __saturatef((float)A * __int_as_float(e[k].w) + 0.5f);             // (A / D + 32) / 64
        const int32_t q = __float_as_int(t * 64.f + (12582912.f - 32.f)) - 0x4B400000;     // nearest integer
        const int out = (int)((uint32_t)(A - e[k].z * q) >> 31);
        if (e[k].z >= 0) hi = min(hi, q - out);
        else lo = max(lo, q + out);
    }
}

// The same for a large triangle: a binary search on each edge over the tile's columns.
HEXFC_ROW_COLD int2 row_span_big(const int4* edge, int stride, int cols, int ry, int lo, int hi)
{
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const int4 e = edge[k * stride];
        const int64_t A = (int64_t)(((uint64_t)(uint32_t)e.w << 32) | (uint32_t)e.x) + (int64_t)e.y * (ry * 256);
        const int64_t dy = e.z;
        if (dy == 0) {
            if (A < 0) hi = -1;
            continue;
        }
        int a = -1, z = cols;   // dy > 0: inside up to a, outside from z; else the other way round
        while (z - a > 1) {
            const int m = (a + z) >> 1;
            if ((A - dy * (m * 256) >= 0) == (dy > 0)) a = m;
            else z = m;
        }
        if (dy > 0) hi = min(hi, a);
        else lo = max(lo, z);
    }
    return make_int2(lo, hi);
}

}  // namespace hexfc
