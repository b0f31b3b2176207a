// Geometry and fragment stages of the renderer.
//
//   k_vertex_setup  per vertex: camera transform (in double by definition, no
//                   FMA; from pairs of floats where those decide the result),
//                   window position snapped to 16.8 fixed point, 24-bit window
//                   depth.
//   k_face_setup    per unique face: gather the 4 projected corners, edge
//                   visibility masks of Eq. 1, triangle validity, and the
//                   number of raster tiles each triangle's box touches.
//   k_tile_scan     the tiles' offsets, and the tiles by decreasing work.
//   k_bin_fill      per triangle: into the list of every touched tile.
//   k_bin_sort      per tile: counting sort of the tile's triangles by depth.
//   k_count         per tile: exact coverage as per-chunk masks and per-pixel
//                   counts.
//
// The drawing pass is in k_draw.cu.
//
// Each face is drawn as two triangles (Section "Method Overview"; Section "GPU
// Implementation"), and all covered samples take part (the paper keeps them in
// per-pixel fragment lists, Section "GPU Implementation"; here they are bits of
// the coverage masks, in the tile's depth order).
#include <algorithm>

#include <cooperative_groups.h>

#include "count_tiles.cuh"
#include "lens_test.h"
#include "shade.cuh"

namespace hexfc {
namespace {

inline unsigned grid_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Small meshes: log2 of the threads a face or triangle gets, as many as one block
// an SM has room for. A warp goes through the tiles of its large triangles one
// triangle at a time, so with fewer of them a warp is done sooner, on SMs that
// have nothing else to do (a 4^3 grid at 256x256: face setup 19 -> 5 us, binning
// 19 -> 3.5 us).
inline int spread_for(int64_t n)
{
    int spread = 0;
    while (spread < 5 && n << (spread + 1) <= 152 * 256) ++spread;
    return spread;
}

// ------------------------------------------------------------------ vertex stage

// Thread per vertex: window position on 1/256 pixel, 24-bit depth, eye depth, and
// the importance that the frame is drawn with.
// It also clears the frame's counters (tile_cnt, tile_big, tile_skip, tile_cur, and the
// device scalars but the error word), which every frame starts from zero.
__global__ void __launch_bounds__(256) k_vertex_setup(const float* __restrict__ verts,
                                                      const int32_t* __restrict__ vkey, int64_t n,
                                                      const __grid_constant__ CamParams cam,
                                                      const __grid_constant__ CamPairs pairs,
                                                      int4* __restrict__ vproj, float* __restrict__ ved,
                                                      uint32_t* __restrict__ tile_cnt,
                                                      uint32_t* __restrict__ tile_big,
                                                      uint32_t* __restrict__ tile_skip,
                                                      uint32_t* __restrict__ tile_cur, int64_t n_tiles,
                                                      uint64_t* __restrict__ scal)
{
    chain_begin();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = v; i < n_tiles; i += (int64_t)gridDim.x * blockDim.x) {
        tile_cnt[i] = 0;
        tile_big[i] = 0;
        if (tile_skip) tile_skip[i] = 0;
        tile_cur[i] = 0;
    }
    if (v < kScalAll && v != 5) scal[v] = 0;
    if (v >= n) return;
    const float x = verts[3 * v], y = verts[3 * v + 1], z = verts[3 * v + 2];
    ProjVertex o;
    if (!pairs.usable || !vertex_pairs(x, y, z, pairs, cam, o)) vertex_double(x, y, z, cam, o);
    vproj[v] = make_int4(o.x, o.y, o.z | (o.valid ? kVertexValid : 0), vkey[v]);
    ved[v] = o.depth;
}

// ------------------------------------------------------------------ face stage

__device__ __forceinline__ void tile_range(const TriGeom& t, int& tx0, int& ty0, int& tx1, int& ty1)
{
    tx0 = t.bx0 / kTileW; tx1 = t.bx1 / kTileW;
    ty0 = t.by0 / kTileH; ty1 = t.by1 / kTileH;
}

// A triangle's depths in one word: the sum of its three window depths (below
// 3 * 2^24) and, in the top six bits, a class e for how far its least depth lies
// below the mean: floor(sum / 3) - least <= depth_spread(e).
__host__ __device__ __forceinline__ uint32_t depth_spread(uint32_t e) { return ((2u + (e & 1u)) << (e >> 1)) >> 1; }
constexpr uint32_t kZSum = (1u << 26) - 1u;

__device__ __forceinline__ uint32_t pack_depths(uint32_t a, uint32_t b, uint32_t c)
{
    const uint32_t sum = a + b + c, spread = sum / 3u - min(a, min(b, c));
    uint32_t e = 0;
    if (spread > 1) {   // the least class: spread lies in (2^(k-1), 2^k]
        const uint32_t k = 32u - (uint32_t)__clz((int)(spread - 1u));
        e = 2u * k;
        if (depth_spread(e - 1u) >= spread) --e;
    }
    return sum | (e << 26);
}

// A lower bound of the triangle's window depths.
__device__ __forceinline__ uint32_t packed_least(uint32_t v)
{
    const uint32_t mean = (v & kZSum) / 3u, s = depth_spread(v >> 26);
    return mean > s ? mean - s : 0u;
}

// A triangle's tiles in one word: the first one's column and row, whether it
// touches a second column and row (kRangeSmall) and that it covers no sample
// (kRangeSkip), or that there are more than 2x2 (kRangeBig: found again in the
// second pass).
constexpr uint32_t kRangeMore = 3u << 22, kRangeSmall = 1u << 24, kRangeBig = 1u << 25, kRangeSkip = 1u << 26;
__device__ __forceinline__ uint32_t pack_range(int tx0, int ty0, int tx1, int ty1)
{
    return (uint32_t)tx0 | ((uint32_t)ty0 << 11) | ((uint32_t)(tx1 - tx0) << 22) | ((uint32_t)(ty1 - ty0) << 23) |
           kRangeSmall;
}
static_assert(16384 / 8 <= 2048, "eleven bits of tile column and row");

// Each lane's place in the counters of up to four tiles (tile < 0: none): one
// atomic per distinct tile of the warp, lanes of one tile in lane order. All
// lanes of the warp call it. The four tiles' atomics are in flight together. With
// `skip` set the lane's tiles are counted apart, in ctr_skip.
__device__ __forceinline__ uint4 count_places(uint32_t* ctr, uint32_t* ctr_skip, bool skip, const int (&tile)[4])
{
    const int lane = threadIdx.x & 31;
    const int apart = skip ? 1 << 30 : 0;   // (no tile, -1, stays -1)
    uint32_t* const c = skip ? ctr_skip : ctr;
    unsigned peers[4];
    uint32_t base[4], place[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        base[k] = 0;
        peers[k] = 0xffffffffu;
        if (!__any_sync(0xffffffffu, tile[k] >= 0)) continue;
        peers[k] = __match_any_sync(0xffffffffu, tile[k] | apart);
        if (tile[k] >= 0 && lane == __ffs(peers[k]) - 1) base[k] = atomicAdd(c + tile[k], (uint32_t)__popc(peers[k]));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        place[k] = __shfl_sync(0xffffffffu, base[k], __ffs(peers[k]) - 1) +
                   (uint32_t)__popc(peers[k] & ((1u << lane) - 1u));
    return make_uint4(place[0], place[1], place[2], place[3]);
}

// f(tile) for every tile of the box of each lane that has `big` set, the warp
// on one lane's box at a time: a triangle over the whole frame is no serial loop.
template <class F>
__device__ __forceinline__ void for_big_tiles(bool big, int tx0, int ty0, int tx1, int ty1, int tiles_x, F&& f)
{
    const int lane = threadIdx.x & 31;
    for (unsigned todo = __ballot_sync(0xffffffffu, big); todo != 0; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int x0 = __shfl_sync(0xffffffffu, tx0, src), y0 = __shfl_sync(0xffffffffu, ty0, src);
        const int w = __shfl_sync(0xffffffffu, tx1, src) - x0 + 1, h = __shfl_sync(0xffffffffu, ty1, src) - y0 + 1;
        for (int i = lane; i < w * h; i += 32) f((y0 + i / w) * tiles_x + x0 + i % w, src);
    }
}

// Is the triangle's sample at pixel (px, py) covered (top-left rule)?
__device__ __forceinline__ bool covers(const TriGeom& t, int px, int py)
{
    bool in = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a = (k + 1) % 3, b = (k + 2) % 3;
        const int64_t e = edge_fn(t.X[a], t.Y[a], t.X[b], t.Y[b], 256 * px + 128, 256 * py + 128);
        in = in && (e > 0 || (e == 0 && top_left(t.X[a], t.Y[a], t.X[b], t.Y[b])));
    }
    return in;
}

// Thread per face: its record of the frame, its triangles' depths, and the
// counts of the tiles they touch. Bound by the latency of its gathers (41% of the
// issue slots; five blocks an SM for that, the atomics issued before the rest did
// not help). A triangle of at most 2x2 tiles keeps the places its counts gave it,
// the first beside its range, so that the binning needs no second round of atomics:
// that pass 64 -> 36 us at 64^3 and 1920x1080, of which the scattered 4-byte writes
// into 8160 lists remain. A face of which nothing is drawn gets no record, records
// are written a sector at a time, and the lens test reads the vertices, which the
// caches hold, instead of the faces' 64-byte static records (96^3 at 320x180: 153
// -> 131 us; 128^3 at 3840x2160: 400 -> 372 us; 64^3 at 1920x1080: 71 -> 70 us).
// Triangles of more tiles are counted by their whole warp (a 4^3 grid at 256x256,
// one block: 25 + 31 us for both passes with a loop per thread, 12 + 8 us with).
__global__ void __launch_bounds__(256, 5) k_face_setup(const int4* __restrict__ fverts, const int4* __restrict__ fedges,
                                                    const uint8_t* __restrict__ fbound,
                                                    const float* __restrict__ verts,
                                                    const uint8_t* __restrict__ elevel,
                                                    const float* __restrict__ eattr, const int4* __restrict__ vproj,
                                                    const float* __restrict__ ved, int64_t n_faces,
                                                    const __grid_constant__ ShadeParams sp, int W, int H, int tiles_x,
                                                    int reverse, FaceFrame* __restrict__ fframe,
                                                    uint32_t* __restrict__ tzsum, uint2* __restrict__ trange,
                                                    uint4* __restrict__ slots, FaceExtra* __restrict__ fextra,
                                                    uint32_t* __restrict__ tile_cnt, uint32_t* __restrict__ tile_big,
                                                    uint32_t* __restrict__ tile_skip, int spread)
{
    chain_begin();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = g >> spread;
    const bool in = i < n_faces && i << spread == g;
    const int64_t f = !in ? 0 : reverse ? n_faces - 1 - i : i;
    const int4 c = fverts[f], e = fedges[f];
    const int id[4] = {c.x, c.y, c.z, c.w}, eid[4] = {e.x, e.y, e.z, e.w};
    int32_t X[4], Y[4];
    uint32_t Z[4];
    float E[4];
    bool ok[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int4 p = vproj[id[k]];
        X[k] = p.x; Y[k] = p.y; Z[k] = (uint32_t)p.z & kZ24; ok[k] = in && (p.z & kVertexValid) != 0;
        E[k] = ved[id[k]];
    }
    uint32_t edges = 0, flags = fbound[f] ? kFaceBoundary : 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool vis_c = (int)elevel[eid[k]] >= sp.lod;
        const bool vis_f = vis_c || eattr[eid[k]] >= sp.delta;
        edges |= (vis_f ? 1u : 0u) << k;
        edges |= (vis_c ? 1u : 0u) << (4 + k);
    }
    uint32_t range[2] = {0u, 0u}, area[2] = {0u, 0u};
    uint4 place[2];
#pragma unroll
    for (int tri = 0; tri < 2; ++tri) {
        const bool vok = ok[0] && ok[1 + tri] && ok[2 + tri];
        TriGeom t;
        tri_setup(X, Y, tri, W, H, t);
        const bool drawn = vok && t.valid;
        int tx0 = 0, ty0 = 0, tx1 = 0, ty1 = 0;
        if (drawn) {
            if (t.vi[1] != 1 + tri) flags |= kFaceSwapped << tri;
            area[tri] = t.area < (1ll << 26) ? (uint32_t)t.area : 0u;
            tile_range(t, tx0, ty0, tx1, ty1);
        }
        const bool small = drawn && slots && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
        // A box of one or two samples, none of them covered: set aside, neither
        // ordered nor drawn (it still counts for the tile's depth range and the
        // frame's pairs). A third of the pairs where triangles are about a pixel
        // (96^3 at 320x180: 4.2 -> 2.8 million, 2.01 -> 1.35 ms a frame), none at
        // 64^3 and 1920x1080; boxes of up to four samples would be 1% more.
        const bool skip = small && t.bx1 - t.bx0 + t.by1 - t.by0 <= 1 && !covers(t, t.bx0, t.by0) && !covers(t, t.bx1, t.by1);
        if (drawn && !skip) flags |= kFaceDrawn << tri;
        if (small) range[tri] = pack_range(tx0, ty0, tx1, ty1) | (skip ? kRangeSkip : 0u);
        else if (drawn) range[tri] = kRangeBig;
        const int t0 = ty0 * tiles_x + tx0;
        const bool c2 = small && tx1 > tx0, r2 = small && ty1 > ty0;
        const int tile[4] = {small ? t0 : -1, c2 ? t0 + 1 : -1, r2 ? t0 + tiles_x : -1, c2 && r2 ? t0 + tiles_x + 1 : -1};
        place[tri] = count_places(tile_cnt, tile_skip, skip, tile);
        for_big_tiles(drawn && !small, tx0, ty0, tx1, ty1, tiles_x, [&](int at, int) { atomicAdd(tile_big + at, 1u); });
    }
    if (!in) return;
    if (sp.lens_mode == HEXFC_LENS_SPHERE && sp.bounded && (flags & (3u * kFaceDrawn))) {
        float o[4][3];   // (from the vertices, which neighbours share in the caches)
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int d = 0; d < 3; ++d) o[k][d] = __ldg(verts + 3 * (int64_t)id[k] + d) - sp.lens_c[d];
#pragma unroll
        for (int tri = 0; tri < 2; ++tri) {
            const float v[3][3] = {{o[0][0], o[0][1], o[0][2]},
                                   {o[1 + tri][0], o[1 + tri][1], o[1 + tri][2]},
                                   {o[2 + tri][0], o[2 + tri][1], o[2 + tri][2]}};
            const float d[3] = {E[0], E[1 + tri], E[2 + tri]};
            if (outside_lens(v, d, sp.ortho != 0, sp.lens_inv_r)) flags |= kFaceOut << tri;
        }
    }
    reinterpret_cast<uint2*>(tzsum)[f] = make_uint2(pack_depths(Z[0], Z[1], Z[2]), pack_depths(Z[0], Z[2], Z[3]));
    if (slots) {
        reinterpret_cast<uint4*>(trange)[f] = make_uint4(range[0], place[0].x, range[1], place[1].x);
        if (range[0] & kRangeMore) slots[2 * f] = place[0];
        if (range[1] & kRangeMore) slots[2 * f + 1] = place[1];
        if (!(flags & (3u * kFaceDrawn))) return;   // in no list that is drawn
    }
    const int4 fx = make_int4(X[0], X[1], X[2], X[3]), fy = make_int4(Y[0], Y[1], Y[2], Y[3]);
    FaceFrame& r = fframe[f];
    store32(&r.X, make_uint4(fx.x, fx.y, fx.z, fx.w), make_uint4(fy.x, fy.y, fy.z, fy.w));
    store32(&r.Z, make_uint4(Z[0] | (edges << 24), Z[1] | (flags << 24), Z[2], Z[3]),
            as_uint4(sp.ortho ? make_float4(1.f, 1.f, 1.f, 1.f)
                              : make_float4(__frcp_rn(E[0]), __frcp_rn(E[1]), __frcp_rn(E[2]), __frcp_rn(E[3]))));
    if (slots)
        store32(&fextra[f], as_uint4(edge_scales(fx, fy)),
                make_uint4(area[0], area[1], __float_as_uint(__frcp_rn((float)area[0])),
                           __float_as_uint(__frcp_rn((float)area[1]))));
}

// Thread per triangle (2 face + triangle): into the lists of its tiles.
__global__ void __launch_bounds__(256) k_bin_fill(const FaceFrame* __restrict__ fframe,
                                                  const uint2* __restrict__ trange, const uint4* __restrict__ slots,
                                                  int64_t n_tris, int W, int H, int tiles_x,
                                                  const uint64_t* __restrict__ tile_off,
                                                  const uint32_t* __restrict__ tile_cnt, uint32_t* __restrict__ tile_cur,
                                                  uint32_t* __restrict__ bins, int spread,
                                                  const uint64_t* __restrict__ n_bins, uint64_t bin_limit)
{
    chain_begin();
    if (*n_bins > bin_limit) return;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, t = g >> spread;
    uint32_t range = 0, place = 0;
    if (t < n_tris && t << spread == g) {
        if (trange) {
            const uint2 v = trange[t];
            range = v.x;
            place = v.y;
        } else if ((face_tris(fframe[t >> 1].Z) >> (t & 1)) & 1u) {
            range = kRangeBig;
        }
    }
    if (range & kRangeSmall) {
        const int tile = (int)((range >> 11) & 2047u) * tiles_x + (int)(range & 2047u);
        const bool c2 = (range >> 22) & 1u, r2 = (range >> 23) & 1u;
        // set aside: from the end of the tile's list down
        const uint64_t* off = range & kRangeSkip ? tile_off + 1 : tile_off;
        const uint32_t down = range & kRangeSkip ? ~0u : 0u;   // (~place is -1 - place)
        auto put = [&](int at, uint32_t k) { bins[(int64_t)off[at] + (int32_t)(k ^ down)] = (uint32_t)t; };
        put(tile, place);
        if (c2 || r2) {
            const uint4 p = slots[t];
            if (c2) put(tile + 1, p.y);
            if (r2) put(tile + tiles_x, p.z);
            if (c2 && r2) put(tile + tiles_x + 1, p.w);
        }
    }
    int tx0 = 0, ty0 = 0, tx1 = 0, ty1 = 0;
    if (range & kRangeBig) {
        const int4 a = fframe[t >> 1].X, b = fframe[t >> 1].Y;
        const int32_t X[4] = {a.x, a.y, a.z, a.w}, Y[4] = {b.x, b.y, b.z, b.w};
        TriGeom g;
        tri_setup(X, Y, (int)(t & 1), W, H, g);
        tile_range(g, tx0, ty0, tx1, ty1);
    }
    const int64_t first = g - (threadIdx.x & 31);
    for_big_tiles(range & kRangeBig, tx0, ty0, tx1, ty1, tiles_x, [&](int tile, int src) {
        bins[tile_off[tile] + tile_cnt[tile] + atomicAdd(tile_cur + tile, 1u)] = (uint32_t)((first + src) >> spread);
    });
}

// ------------------------------------------------------------------ tile offsets and order

constexpr int kScanTiles = 16384;   // most tiles of the one-block scan (16 a thread)

// One block: the tiles' offsets in the bins (each list padded to whole chunks)
// and the tiles in decreasing order of their chunks (a counting sort into 1024
// classes; order inside a class is arbitrary, no result depends on it), so that
// the per-tile passes start the longest tiles first and the shortest ones fill
// the tail of the launch. One launch for what four took (64^3 at 1920x1080, 8160
// tiles: 14 us, before 13 for the scan and 19 for the order).
__global__ void __launch_bounds__(1024) k_tile_scan(const uint32_t* __restrict__ tile_cnt,
                                                    const uint32_t* __restrict__ tile_big,
                                                    const uint32_t* __restrict__ tile_skip, int n,
                                                    uint64_t* __restrict__ tile_off, uint32_t* __restrict__ order,
                                                    uint64_t* __restrict__ total, uint64_t* __restrict__ h_total)
{
    chain_begin();
    constexpr int kPer = kScanTiles / 1024;
    __shared__ uint32_t s_hist[1024], s_warp[32], s_max[32], s_empty;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (n + 1023) / 1024, t0 = threadIdx.x * per;
    uint32_t nc[kPer], sum = 0, mx = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int t = t0 + k;
        nc[k] = k < per && t < n ? (tile_cnt[t] + tile_big[t] + (tile_skip ? tile_skip[t] : 0u) + kChunk - 1) / kChunk : 0u;
        sum += nc[k];
        mx = max(mx, nc[k]);
    }
    s_hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_empty = 0;
    uint32_t all = 0;   // the scan's total
    auto block_scan = [&](uint32_t v) -> uint32_t {   // exclusive, over the block's threads
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t w = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const uint32_t before = __shfl_sync(0xffffffffu, w, warp - 1);
        all = __shfl_sync(0xffffffffu, w, 31);
        return incl - v + (warp > 0 ? before : 0u);
    };
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) s_max[warp] = mx;
    uint64_t at = block_scan(sum);   // (fewer than 2^32 chunks: its barriers publish s_max, s_hist, s_empty too)
    if (threadIdx.x == 1023) {
        tile_off[n] = (uint64_t)all * kChunk;
        *total = (uint64_t)all * kChunk;
        if (h_total) *h_total = (uint64_t)all * kChunk;
    }
    // Three drawing blocks an SM hold all tiles of a small frame at once: any order
    // does (but not for long lists, whose form has one, launch_draw).
    if (n <= 3 * 152 && all < 3u * (uint32_t)n) {
        if ((int)threadIdx.x < n) {   // (a tile a thread)
            tile_off[threadIdx.x] = at * kChunk;
            order[threadIdx.x] = threadIdx.x;
        }
        return;
    }
    mx = __reduce_max_sync(0xffffffffu, s_max[lane]);
    int shift = 0;
    while ((mx >> shift) >= 1024u) ++shift;
    uint32_t rank[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int t = t0 + k;
        const bool here = k < per && t < n;
        if (here) tile_off[t] = at * kChunk;
        at += nc[k];
        // empty tiles (often most of them) are counted by the warp, the others one by one
        rank[k] = 0;
        if (k < per) {
            const unsigned none = __ballot_sync(0xffffffffu, here && nc[k] == 0);
            uint32_t base = 0;
            if (none && lane == 0) base = atomicAdd(&s_empty, (uint32_t)__popc(none));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (here) {
                if (nc[k] == 0) rank[k] = base + (uint32_t)__popc(none & ((1u << lane) - 1u));
                else rank[k] = atomicAdd(&s_hist[1023u - (nc[k] >> shift)], 1u);
            }
        }
    }
    __syncthreads();
    const uint32_t h = s_hist[threadIdx.x];
    const uint32_t first = block_scan(h);
    s_hist[threadIdx.x] = first;
    __syncthreads();
    const uint32_t filled = (uint32_t)n - s_empty;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int t = t0 + k;
        if (k < per && t < n)
            order[(nc[k] == 0 ? filled : s_hist[1023u - (nc[k] >> shift)]) + rank[k]] = (uint32_t)t;
    }
}

// ------------------------------------------------------------------ bin order

constexpr int kDepthBucketsMax = 4096;
__host__ __device__ constexpr size_t sort_smem(int threads, int items, int nb)
{
    const size_t cap = (size_t)threads * items;
    return sizeof(uint32_t) * (cap + (size_t)(nb < threads ? threads : nb) + cap / kChunk + 64);
}

// Orders each tile's list front to back by a counting sort of the triangles
// into nb buckets (a power of two, 256..kDepthBucketsMax) of their depth (sum of
// the three window depths) over the tile's depth range, and pads it to whole
// chunks. Any order gives the same image; this one makes every pixel meet its
// fragments sorted or nearly sorted (order within a bucket is arbitrary). zsuf
// receives, per chunk, a lower bound of the depths of the triangles from that
// chunk on: a pixel that is opaque in front of it is finished. nb 0: no order.
//
// A block of kT threads holds up to kT * kItems entries in registers (read
// once); longer lists go through global scratch. The block also leaves the tile's
// features of the capacity network (cf).
// Bound by the latency of its steps and barriers (40% of the issue slots): short
// lists take fewer buckets, those of a chunk one warp without any (29^3 at 1280x720,
// 160 entries a tile: binning 48 -> 41 us, 4^3 at 256x256, 26 a tile: 12.5 -> 10.6).
template <int kT, int kItems>
__global__ void __launch_bounds__(kT, kT == 1024 ? 1 : kItems == 8 ? 6 : 5) k_bin_sort(const uint64_t* __restrict__ tile_off,
                                                            const uint32_t* __restrict__ tile_cnt,
                                                 const uint32_t* __restrict__ tile_big,
                                                 const uint32_t* __restrict__ tile_skip,
                                                 uint32_t* __restrict__ tile_chunks, uint32_t* __restrict__ bins,
                                                 const uint32_t* __restrict__ tzsum, int nb,
                                                 uint32_t* __restrict__ tmp, uint32_t* __restrict__ zsuf,
                                                 const uint64_t* __restrict__ n_bins, uint64_t bin_limit,
                                                 const CapFeatures cf)
{
    chain_begin();
    if (*n_bins > bin_limit) return;
    constexpr uint32_t kMax = kT * kItems, kLow = kMax / kChunk;
    constexpr bool kShort = kItems == 8;   // the form for short lists: they are common in it
    extern __shared__ uint32_t sort_sm[];
    uint32_t* s_out = sort_sm;                 // [kMax]
    uint32_t* s_low = s_out + kMax;            // [kLow] least depth of each chunk
    uint32_t* s_red = s_low + kLow;            // [2][32]
    uint32_t* s_hist = s_red + 64;             // [max(nb, kT)]
    const int tile = blockIdx.x;
    const uint64_t beg = tile_off[tile];
    const uint32_t n = tile_cnt[tile] + tile_big[tile], n_skip = tile_skip ? tile_skip[tile] : 0u;
    const uint32_t n_chunks = (n + kChunk - 1) / kChunk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto pad = [&]() {   // the last chunk, over what was read of the rest
        for (uint32_t i = n + threadIdx.x; i < n_chunks * kChunk; i += kT) bins[beg + i] = kPadBin;
    };
    if (threadIdx.x == 0) tile_chunks[tile] = n_chunks;
    uint32_t zmin = 0xFFFFFFFFu, zmax = 0;
    if (n + n_skip < 2 || nb == 0) {   // nothing to order
        pad();
        for (uint32_t i = threadIdx.x; i < n_chunks; i += kT) zsuf[beg / kChunk + i] = 0u;
        zmin = 0;
    } else if (kShort && n <= 32) {   // one warp, each entry's rank counted
        if (warp != 0) return;
        const uint32_t* aside = bins + tile_off[tile + 1] - n_skip;
        for (uint32_t i = lane; i < n_skip; i += 32) {
            const uint32_t z = tzsum[aside[i]] & kZSum;
            zmin = min(zmin, z);
            zmax = max(zmax, z);
        }
        const bool in = (uint32_t)lane < n;
        const uint32_t f = in ? bins[beg + lane] : kPadBin;
        const uint32_t zs = in ? tzsum[f] : 0u, z = zs & kZSum;
        uint32_t rank = 0;
        for (uint32_t j = 0; j < n; ++j) {
            const uint32_t o = __shfl_sync(0xffffffffu, z, j);
            rank += o < z || (o == z && j < (uint32_t)lane) ? 1u : 0u;
        }
        __syncwarp();   // (the list and what was set aside have been read)
        if (n > 0) bins[beg + (in ? rank : (uint32_t)lane)] = f;
        const uint32_t low = __reduce_min_sync(0xffffffffu, in ? packed_least(zs) : 0xFFFFFFFFu);
        if (n > 0 && lane == 0) zsuf[beg / kChunk] = low;
        zmin = __reduce_min_sync(0xffffffffu, in ? min(zmin, z) : zmin);
        zmax = __reduce_max_sync(0xffffffffu, in ? max(zmax, z) : zmax);
    } else {
        if (kShort)
            while (nb > 256 && (uint32_t)nb >= 8 * n) nb >>= 1;   // as many buckets an entry as long lists have
        // triangles that cover no sample count for the tile's depth range only
        if (n_skip) {
            const uint32_t* aside = bins + tile_off[tile + 1] - n_skip;
#pragma unroll 1
            for (uint32_t i = threadIdx.x; i < n_skip; i += kT) {
                const uint32_t z = tzsum[aside[i]] & kZSum;
                zmin = min(zmin, z);
                zmax = max(zmax, z);
            }
        }
        const bool big = n > kMax;   // entries re-read, scatter through tmp
        uint32_t f2t[kItems], zs[kItems];
        if (!big) {
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                const uint32_t i = threadIdx.x + (uint32_t)(kT * k);
                if (kT * k >= (int)n) break;   // (the same for the block)
                f2t[k] = i < n ? bins[beg + i] : 0u;
            }
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (kT * k >= (int)n) break;
                const bool in = threadIdx.x + (uint32_t)(kT * k) < n;
                zs[k] = in ? tzsum[f2t[k]] : 0u;
                zmin = min(zmin, in ? zs[k] & kZSum : 0xFFFFFFFFu);
                zmax = max(zmax, zs[k] & kZSum);
            }
        } else {
            for (uint32_t i = threadIdx.x; i < n; i += kT) {
                const uint32_t z = tzsum[bins[beg + i]] & kZSum;
                zmin = min(zmin, z);
                zmax = max(zmax, z);
            }
        }
        for (int i = threadIdx.x; i < nb; i += kT) s_hist[i] = 0;
        for (uint32_t i = threadIdx.x; i < kLow; i += kT) s_low[i] = 0xFFFFFFFFu;
        zmin = __reduce_min_sync(0xffffffffu, zmin);
        zmax = __reduce_max_sync(0xffffffffu, zmax);
        if (lane == 0) {
            s_red[warp] = zmin;
            s_red[32 + warp] = zmax;
        }
        __syncthreads();
        pad();
        zmin = __reduce_min_sync(0xffffffffu, s_red[lane % (kT / 32)]);
        zmax = __reduce_max_sync(0xffffffffu, s_red[32 + lane % (kT / 32)]);
        const float scale = (float)nb / (float)(zmax - zmin + 1);
        auto bucket = [&](uint32_t z) -> int { return min((int)((float)((z & kZSum) - zmin) * scale), nb - 1); };
        // histogram
        if (!big) {
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (kT * k >= (int)n) break;
                if (threadIdx.x + (uint32_t)(kT * k) < n) atomicAdd(&s_hist[bucket(zs[k])], 1u);
            }
        } else {
            for (uint32_t i = threadIdx.x; i < n; i += kT) atomicAdd(&s_hist[bucket(tzsum[bins[beg + i]])], 1u);
        }
        __syncthreads();
        // exclusive scan of the histogram: nb / kT buckets a thread (at least one)
        {
            const int per = nb >= kT ? nb / kT : 1;
            const bool mine = (int)threadIdx.x * per < nb;
            uint32_t* h = s_hist + threadIdx.x * per;
            uint32_t sum = 0;
            for (int k = 0; k < per && mine; ++k) sum += h[k];
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            __syncthreads();   // s_red has been read
            if (lane == 31) s_red[warp] = incl;
            __syncthreads();
            const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? s_red[lane] : 0u);
            uint32_t base = before + incl - sum;
            for (int k = 0; k < per && mine; ++k) {
                const uint32_t v = h[k];
                h[k] = base;
                base += v;
            }
        }
        __syncthreads();
        // scatter (arbitrary order inside a bucket), then write back
        if (!big) {
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (kT * k >= (int)n) break;
                if (threadIdx.x + (uint32_t)(kT * k) < n) {
                    const uint32_t at = atomicAdd(&s_hist[bucket(zs[k])], 1u);
                    s_out[at] = f2t[k];
                    atomicMin(&s_low[at / kChunk], packed_least(zs[k]));
                }
            }
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < n; i += kT) bins[beg + i] = s_out[i];
        } else {
            for (uint32_t i = threadIdx.x; i < n; i += kT) {
                const uint32_t f = bins[beg + i];
                tmp[beg + atomicAdd(&s_hist[bucket(tzsum[f])], 1u)] = f;
            }
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < n_chunks * kChunk; i += kT) {   // (a warp: one chunk)
                uint32_t low = 0xFFFFFFFFu;
                if (i < n) {
                    const uint32_t f = tmp[beg + i];
                    bins[beg + i] = f;
                    low = packed_least(tzsum[f]);
                }
                low = __reduce_min_sync(0xffffffffu, low);
                if (lane == 0) zsuf[(beg + i) / kChunk] = low;
            }
        }
        __syncthreads();
        if (warp == 0) {   // the least from each chunk on, 32 chunks at a time from the end
            uint32_t after = 0xFFFFFFFFu;
            for (int c0 = (int)((n_chunks - 1) & ~31u); c0 >= 0; c0 -= 32) {
                const bool in = (uint32_t)(c0 + lane) < n_chunks;
                uint32_t* z = zsuf + beg / kChunk + c0 + lane;
                uint32_t low = !in ? 0xFFFFFFFFu : big ? *z : s_low[c0 + lane];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_down_sync(0xffffffffu, low, o);
                    if (lane + o < 32) low = min(low, y);
                }
                low = min(low, after);
                if (in) *z = low;
                after = __shfl_sync(0xffffffffu, low, 0);
            }
        }
    }
    if (cf.X && threadIdx.x == 0) {
        // log of the previous frame's count, the tile's depth range (of 3 * 2^24), its
        // distance to the lens on screen, the camera's motion
        const float cx = (float)((tile % cf.tiles_x) * kTileW) + 0.5f * kTileW;
        const float cy = (float)((tile / cf.tiles_x) * kTileH) + 0.5f * kTileH;
        const float dx = cx - cf.lens_x, dy = cy - cf.lens_y;
        float4 x;
        x.x = log1pf(cf.prev ? (float)cf.prev[tile] : 0.f) * (1.f / 12.f);
        x.y = (float)(zmax - zmin) * (1.f / 50331648.f);
        x.z = fminf(sqrtf(dx * dx + dy * dy) * cf.inv_diag, 2.f);
        x.w = cf.motion;
        reinterpret_cast<float4*>(cf.X)[tile] = x;
    }
}

// ------------------------------------------------------------------ tile order

constexpr int kOrderBuckets = 4096;   // chunk counts above kOrderBuckets - 1 share the first class

// Rank of lane's value among the lanes of the warp holding the same value, and
// how many hold it, so that one lane per value does the shared-memory atomic.
__device__ __forceinline__ uint32_t warp_add_same(uint32_t* s, uint32_t b, bool active)
{
    const unsigned act = __ballot_sync(0xffffffffu, active);
    if (!active) return 0;
    const unsigned peers = __match_any_sync(act, b);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&s[b], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
}

// The tiles in decreasing order of their number of chunks, as k_tile_scan
// leaves them, for frames of more tiles than that takes. One block.
__global__ void __launch_bounds__(1024) k_tile_order(const uint64_t* __restrict__ tile_off, int n_tiles,
                                                     uint32_t* __restrict__ order)
{
    __shared__ uint32_t s_hist[kOrderBuckets];
    __shared__ uint32_t s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto cls = [&](int t) -> uint32_t {
        const uint64_t nc = (tile_off[t + 1] - tile_off[t]) / kChunk;
        return (uint32_t)(kOrderBuckets - 1) - (uint32_t)min(nc, (uint64_t)(kOrderBuckets - 1));
    };
    // the classes of tiles threadIdx.x + 1024 k, k < kReg, are read once, all
    // loads in flight together, and kept in registers for both passes
    constexpr int kReg = 16;
    uint32_t cl[kReg];
#pragma unroll
    for (int k = 0; k < kReg; ++k) {
        const int t = k * 1024 + threadIdx.x;
        cl[k] = t < n_tiles ? cls(t) : 0u;
    }
    for (int i = threadIdx.x; i < kOrderBuckets; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kReg; ++k)
        if (k * 1024 < n_tiles) warp_add_same(s_hist, cl[k], k * 1024 + (int)threadIdx.x < n_tiles);
    for (int t0 = kReg * 1024; t0 < n_tiles; t0 += blockDim.x) {
        const int t = t0 + threadIdx.x;
        warp_add_same(s_hist, t < n_tiles ? cls(t) : 0u, t < n_tiles);
    }
    __syncthreads();
    // exclusive scan of the histogram: kOrderBuckets / 1024 classes per thread
    constexpr int kPer = kOrderBuckets / 1024;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = s_hist[threadIdx.x * kPer + k];
        sum += v[k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t base = incl - sum;
    for (int w = 0; w < warp; ++w) base += s_warp[w];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        s_hist[threadIdx.x * kPer + k] = base;
        base += v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kReg; ++k) {
        const int t = k * 1024 + threadIdx.x;
        if (k * 1024 < n_tiles) {
            const uint32_t slot = warp_add_same(s_hist, cl[k], t < n_tiles);
            if (t < n_tiles) order[slot] = (uint32_t)t;
        }
    }
    for (int t0 = kReg * 1024; t0 < n_tiles; t0 += blockDim.x) {
        const int t = t0 + threadIdx.x;
        const uint32_t slot = warp_add_same(s_hist, t < n_tiles ? cls(t) : 0u, t < n_tiles);
        if (t < n_tiles) order[slot] = (uint32_t)t;
    }
}

// Per tile: coverage of every chunk as per-pixel bit masks (kept for the
// drawing pass) and the per-pixel list lengths; the tile's total goes to
// tile_frag, and into copy tile % kStatCopies of the frame's statistics (after
// the device scalars scal): [0] += fragments, [1] = longest list, [2] += lists
// longer than kLongList. The last of the frame's tiles sums the copies into
// scal[0..2] and writes them to the host itself, as the tile scan does with the
// bin total: a copy on the stream would hold up the kernel after it (5-7 us).
// The count of one tile (the body of k_count and k_count_batch), by the blocks
// of a cluster: block `slice` of `slices` takes every slices-th run of
// kConsumerWarps chunks, the first sums the pixels' counts.
__device__ __forceinline__ void count_tile(int tile, const CountItem& a, uint32_t slice, uint32_t slices)
{
    if (a.scal[8] > a.bin_limit) return;   // (all blocks alike)
    extern __shared__ __align__(16) unsigned char count_smem[];
    CountWarp* s_w = reinterpret_cast<CountWarp*>(count_smem);   // [kConsumerWarps]
    const int px0 = (tile % a.tiles_x) * kTileW, py0 = (tile / a.tiles_x) * kTileH;
    const uint64_t beg = a.tile_off[tile];   // a multiple of kChunk
    const uint32_t n_chunks = a.tile_chunks[tile];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    count_chunks(s_w[warp], lane, a.bins, a.fframe, beg, n_chunks, slice * kConsumerWarps + warp,
                 slices * kConsumerWarps, px0, py0, a.W, a.H, a.masks);
    __syncthreads();
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < kConsumerWarps; ++w) n += (&s_w[w].rows[0][0])[threadIdx.x];
    if (slices > 1) {
        const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
        __shared__ uint32_t s_cnt[kTilePix];
        s_cnt[threadIdx.x] = n;
        cluster.sync();
        if (slice == 0)
            for (uint32_t k = 1; k < slices; ++k) n += cluster.map_shared_rank(s_cnt, k)[threadIdx.x];
        cluster.sync();   // (a block's shared memory lives until it was read)
        if (slice != 0) return;
    }
    a.cnt[(int64_t)tile * kTilePix + threadIdx.x] = n;
    __shared__ uint32_t s_red[3][kConsumerWarps];
    const uint32_t sum = __reduce_add_sync(0xffffffffu, n), mx = __reduce_max_sync(0xffffffffu, n);
    const uint32_t lg = __reduce_add_sync(0xffffffffu, n > (uint32_t)kLongList ? 1u : 0u);
    if (lane == 0) {
        s_red[0][warp] = sum;
        s_red[1][warp] = mx;
        s_red[2][warp] = lg;
    }
    __syncthreads();
    if (warp != 0) return;
    uint32_t last = 0;
    if (lane == 0) {
        uint32_t total = 0, m = 0, l = 0;
#pragma unroll
        for (int w = 0; w < kConsumerWarps; ++w) {
            total += s_red[0][w];
            m = max(m, s_red[1][w]);
            l += s_red[2][w];
        }
        a.tile_frag[tile] = total;
        unsigned long long* st = a.scal + kScal + (tile % kStatCopies) * 4;
        if (total) atomicAdd(&st[0], (unsigned long long)total);
        if (m) atomicMax(&st[1], (unsigned long long)m);
        if (l) atomicAdd(&st[2], (unsigned long long)l);
        __threadfence();
        last = atomicAdd(&a.scal[15], 1ull) + 1ull == (unsigned long long)a.n_tiles;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    static_assert(kStatCopies == 32, "one copy a lane");
    const unsigned long long* st = a.scal + kScal + lane * 4;
    unsigned long long v0 = __ldcg(&st[0]), v2 = __ldcg(&st[2]);
    const uint32_t v1 = __reduce_max_sync(0xffffffffu, (uint32_t)__ldcg(&st[1]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    }
    if (lane == 0) {
        a.scal[0] = v0;
        a.scal[1] = v1;
        a.scal[2] = v2;
        if (a.h_scal) {
            a.h_scal[0] = v0;
            a.h_scal[1] = v1;
            a.h_scal[2] = v2;
            a.h_scal[5] = __ldcg(&a.scal[5]);
        }
    }
}

__global__ void __launch_bounds__(kTilePix, kCountBlocks) k_count(const __grid_constant__ CountItem a)
{
    chain_wait();
    const uint32_t slices = cooperative_groups::this_cluster().num_blocks();
    if (blockIdx.x / slices >= (uint32_t)a.n_tiles) return;   // (not reached while grid and clusters belong together)
    count_tile((int)a.order[blockIdx.x / slices], a, blockIdx.x % slices, slices);
}

// The count of several frames in one grid (a batch).
__global__ void __launch_bounds__(kTilePix, kCountBlocks) k_count_batch(const __grid_constant__ CountBatch b)
{
    const int i = batch_item(b.tile_begin, b.n, blockIdx.x);
    count_tile((int)b.it[i].order[blockIdx.x - b.tile_begin[i]], b.it[i], 0, 1);
}

}  // namespace

cudaError_t prepare_raster_kernels()
{
    cudaError_t e = cudaFuncSetAttribute(k_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kConsumerWarps * sizeof(CountWarp)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_bin_sort<1024, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sort_smem(1024, 16, kDepthBucketsMax));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_count_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kConsumerWarps * sizeof(CountWarp)));
    return e;
}

cudaError_t launch_vertex_setup(const DevMesh& m, const CamParams& cam, FrameBufs& fb, int64_t n_tiles, cudaStream_t s)
{
    const unsigned tiles = std::min(grid_for(n_tiles, 256), 1216u);   // (two blocks' worth of clears an SM at most)
    return launch_chained(k_vertex_setup, std::max(grid_for(m.n_verts, 256), tiles), 256, 0, s, false, m.verts, m.vkey,
                          m.n_verts, cam, cam_pairs(cam), fb.vproj, fb.ved, fb.tile_cnt, fb.tile_big, fb.tile_skip, fb.tile_cur,
                          n_tiles, fb.scal);
}

cudaError_t launch_face_setup(const DevMesh& m, const CamParams& cam, const ShadeParams& sp, FrameBufs& fb,
                              int tiles_x, int tiles_y, int reverse, cudaStream_t s)
{
    (void)tiles_y;
    const int spread = spread_for(m.n_faces);
    return launch_chained(k_face_setup, grid_for(m.n_faces << spread, 256), 256, 0, s, fb.chained, m.fverts, m.fedges,
                          m.fbound, m.verts, m.elevel, m.eattr, fb.vproj, fb.ved, m.n_faces, sp, cam.W, cam.H,
                          tiles_x, reverse, fb.fframe, fb.tzsum, fb.trange, fb.slots, fb.fextra, fb.tile_cnt, fb.tile_big,
                          fb.tile_skip, spread);
}

cudaError_t launch_tile_scan(FrameBufs& fb, int64_t n_tiles, bool* ordered, cudaStream_t s)
{
    *ordered = n_tiles <= kScanTiles;
    if (!*ordered)
        return scan_u32_to_u64(fb.tile_cnt, fb.tile_off, n_tiles, fb.part, fb.part_max, fb.scal + 8, 0xFFFFFFFFu, s,
                               (uint32_t)kChunk, fb.tile_big, fb.slots ? fb.tile_skip : nullptr);
    return launch_chained(k_tile_scan, 1, 1024, 0, s, fb.chained, fb.tile_cnt, fb.tile_big,
                          fb.slots ? fb.tile_skip : nullptr, (int)n_tiles, fb.tile_off, fb.tile_order, fb.scal + 8,
                          fb.h_scal ? fb.h_scal + 8 : nullptr);
}

cudaError_t launch_bin_fill(const DevMesh& m, FrameBufs& fb, int tiles_x, int W, int H, cudaStream_t s)
{
    const int spread = spread_for(2 * m.n_faces);
    return launch_chained(k_bin_fill, grid_for((2 * m.n_faces) << spread, 256), 256, 0, s, fb.chained, fb.fframe, fb.trange,
                          fb.slots, 2 * m.n_faces, W, H, tiles_x, fb.tile_off, fb.tile_cnt, fb.tile_cur, fb.bins, spread,
                          fb.scal + 8, fb.bin_limit);
}

cudaError_t launch_bin_sort(FrameBufs& fb, int64_t n_tiles, int64_t n_bins, int buckets, const CapFeatures& cf,
                            cudaStream_t s)
{
    auto go = [&](auto kernel, int threads, int items) {
        return launch_chained(kernel, (unsigned)n_tiles, threads, sort_smem(threads, items, buckets), s, fb.chained,
                              fb.tile_off, fb.tile_cnt, fb.tile_big, fb.slots ? fb.tile_skip : nullptr, fb.tile_cur,
                              fb.bins, fb.tzsum, buckets, fb.bins_tmp, fb.zsuf, fb.scal + 8, fb.bin_limit, cf);
    };
    // Many tiles: several blocks an SM, to go on with others while one waits at its
    // barriers; 16 entries a thread where lists of more than 8 x 256 are common
    // (128^3 at 3840x2160, 1050 a tile: 0.45 ms, with 8 entries 0.85; 64^3 at
    // 1920x1080, 500 a tile: 8 entries 0.061 ms, 16 entries 0.076). Few tiles with
    // long lists (a large mesh drawn small): most of an SM for each (96^3 at
    // 320x180: 0.51 ms with 256 threads, 0.07 with 1024).
    if (n_bins <= 768 * n_tiles) return go(k_bin_sort<256, 8>, 256, 8);
    if (n_tiles > 1024) return go(k_bin_sort<256, 16>, 256, 16);
    return go(k_bin_sort<1024, 16>, 1024, 16);
}

cudaError_t launch_tile_order(FrameBufs& fb, int n_tiles, cudaStream_t s)
{
    k_tile_order<<<1, 1024, 0, s>>>(fb.tile_off, n_tiles, fb.tile_order);
    return cudaGetLastError();
}

CountItem count_item(const FrameBufs& fb, int tiles_x, int tiles_y, int W, int H)
{
    return CountItem{fb.tile_off, fb.tile_cur, fb.bins, fb.fframe, fb.tile_order, fb.cnt, fb.masks, fb.tile_frag,
                     reinterpret_cast<unsigned long long*>(fb.scal), fb.h_scal, fb.bin_limit, tiles_x, W, H, tiles_x * tiles_y};
}

unsigned count_slices(int64_t n_tiles, int64_t n_bins)
{
    // Few tiles with long lists: several blocks a tile, up to four times what the
    // chip holds at once, so that the longest list does not decide alone, and a
    // run of chunks for every warp (96^3 at 320x180, 240 tiles of up to 1500
    // chunks: one block 0.48 ms, as many as fit at once 0.26, twice 0.15, four
    // times 0.11). The blocks of a tile are a cluster.
    unsigned slices = 1;
    while (slices < kCountSlices && 2 * slices * n_tiles <= 4 * 152 * kCountBlocks &&
           slices * n_tiles * 2 * kConsumerWarps * kChunk < n_bins)
        slices *= 2;
    return slices;
}

cudaError_t launch_count(FrameBufs& fb, int tiles_x, int tiles_y, int W, int H, int64_t n_bins, cudaStream_t s,
                         bool to_host)
{
    const int64_t n_tiles = (int64_t)tiles_x * tiles_y;
    const unsigned slices = count_slices(n_tiles, n_bins);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)n_tiles * slices);
    cfg.blockDim = dim3(kTilePix);
    cfg.dynamicSmemBytes = kConsumerWarps * sizeof(CountWarp);
    cfg.stream = s;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = slices;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = fb.chained ? 2 : 1;
    CountItem it = count_item(fb, tiles_x, tiles_y, W, H);
    if (!to_host) it.h_scal = nullptr;
    return cudaLaunchKernelEx(&cfg, k_count, it);
}

cudaError_t launch_count_batch(const CountBatch& b, cudaStream_t s)
{
    const size_t smem = kConsumerWarps * sizeof(CountWarp);
    if (b.n == 0 || b.tile_begin[b.n] == 0) return cudaSuccess;
    k_count_batch<<<b.tile_begin[b.n], kTilePix, smem, s>>>(b);
    return cudaGetLastError();
}

}  // namespace hexfc
