// Geometry and fragment stages of the renderer.
//
//   k_vertex_setup  per vertex: camera transform in double (no FMA), window
//                   position snapped to 16.8 fixed point, 24-bit window depth.
//   k_face_setup    per unique face: gather the 4 projected corners, edge
//                   visibility masks of Eq. 1, triangle validity, and the
//                   number of raster tiles each triangle's box touches.
//   k_bin_fill      per face: append 2*face+tri to the list of every touched tile.
//   k_bin_sort      per tile: counting sort of the tile's triangles by depth.
//   k_tile_order    the tiles by decreasing work (for count and draw).
//   k_count         per tile: exact coverage as per-chunk masks and per-pixel
//                   counts.
//
// The drawing pass is in k_draw.cu.
//
// Each face is drawn as two triangles (Section "Method Overview"; Section "GPU
// Implementation"), all covered samples are kept (per-pixel fragment lists,
// Section "GPU Implementation"), and the fragment shader computes focus from
// the lens, the edge distance to the four face edges ignoring invisible ones,
// and Eqs. 1-4 (Section "Focus+Context").
#include "count_tiles.cuh"

namespace hexfc {
namespace {

inline unsigned grid_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// ------------------------------------------------------------------ vertex stage

// Thread per vertex: window position on 1/256 pixel, 24-bit depth, eye depth.
__global__ void __launch_bounds__(256) k_vertex_setup(const float* __restrict__ verts, int64_t n,
                                                      const __grid_constant__ CamParams cam,
                                                      const __grid_constant__ CamPairs pairs,
                                                      int4* __restrict__ vproj, float* __restrict__ ved)
{
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const float x = verts[3 * v], y = verts[3 * v + 1], z = verts[3 * v + 2];
    ProjVertex o;
    if (!pairs.usable || !vertex_pairs(x, y, z, pairs, cam, o)) vertex_double(x, y, z, cam, o);
    vproj[v] = make_int4(o.x, o.y, o.z, o.valid);
    ved[v] = o.depth;
}

// ------------------------------------------------------------------ face stage

// atomicAdd(ctr + idx, 1) for every calling lane, one atomic per distinct idx
// among the lanes that call together; returns the value this lane's own
// increment would have returned (lanes of one index in lane order).
__device__ __forceinline__ uint32_t agg_inc(uint32_t* ctr, int idx)
{
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, idx);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(ctr + idx, (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
}

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

// Whether the triangle of corners with offsets o[k] from the sphere lens' centre
// and eye depths e[k] lies wholly outside the lens. The offsets, projected on
// the direction of their sum, are all above the radius, so every point of the
// triangle is. The margin covers the rounding of a sample's distance (affine
// sums of offset / w and 1 / w in float: below 12 * 2^-24 of the largest
// offset, times the ratio of the eye depths), so that the computed distance is
// at least 1 too, and the sample's focus exactly 0.
__device__ __forceinline__ bool outside_lens(const float (&o)[3][3], const float (&e)[3], bool ortho, float inv_r)
{
    const float mx = o[0][0] + o[1][0] + o[2][0], my = o[0][1] + o[1][1] + o[2][1],
                mz = o[0][2] + o[1][2] + o[2][2];
    const float im = rsqrtf(mx * mx + my * my + mz * mz);
    float lo = INFINITY, far = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo = fminf(lo, (o[k][0] * mx + o[k][1] * my + o[k][2] * mz) * im);
        far = fmaxf(far, fabsf(o[k][0]) + fabsf(o[k][1]) + fabsf(o[k][2]));
    }
    const float e_lo = fminf(e[0], fminf(e[1], e[2])), e_hi = fmaxf(e[0], fmaxf(e[1], e[2]));
    const float ratio = ortho ? 1.f : __fdividef(e_hi, e_lo);
    return (ortho || e_lo > 0.f) && lo * inv_r >= 1.0001f + 8e-6f * far * inv_r * ratio;
}

__global__ void k_face_setup(const int4* __restrict__ fverts, const int4* __restrict__ fedges,
                             const uint8_t* __restrict__ fbound, const FaceStatic* __restrict__ fstat,
                             const uint8_t* __restrict__ elevel, const float* __restrict__ eattr,
                             const int4* __restrict__ vproj, const float* __restrict__ ved, int64_t n_faces,
                             const __grid_constant__ ShadeParams sp, int W, int H, int tiles_x,
                             FaceFrame* __restrict__ fframe, uint32_t* __restrict__ tzsum,
                             uint32_t* __restrict__ tile_cnt)
{
    int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= n_faces) return;
    int4 c = fverts[f];
    int id[4] = {c.x, c.y, c.z, c.w};
    int32_t X[4], Y[4];
    uint32_t Z[4];
    float E[4];
    bool ok[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int4 p = vproj[id[k]];
        X[k] = p.x; Y[k] = p.y; Z[k] = (uint32_t)p.z & kZ24; ok[k] = p.w != 0;
        E[k] = ved[id[k]];
    }
    int4 e = fedges[f];
    int eid[4] = {e.x, e.y, e.z, e.w};
    uint32_t edges = 0, flags = fbound[f] ? kFaceBoundary : 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        bool vis_c = (int)elevel[eid[k]] >= sp.lod;
        bool vis_f = vis_c || eattr[eid[k]] >= sp.delta;
        edges |= (vis_f ? 1u : 0u) << k;
        edges |= (vis_c ? 1u : 0u) << (4 + k);
    }
    uint32_t area[2] = {0u, 0u};
    float ia[2] = {0.f, 0.f};
#pragma unroll
    for (int tri = 0; tri < 2; ++tri) {
        bool vok = ok[0] && (tri == 0 ? (ok[1] && ok[2]) : (ok[2] && ok[3]));
        if (!vok) continue;
        TriGeom t;
        tri_setup(X, Y, tri, W, H, t);
        if (!t.valid) continue;
        flags |= kFaceDrawn << tri;
        if (t.vi[1] != 1 + tri) flags |= kFaceSwapped << tri;
        area[tri] = t.area < (1ll << 26) ? (uint32_t)t.area : 0u;
        ia[tri] = 1.f / u64_to_f32((uint64_t)t.area);
        int tx0, ty0, tx1, ty1;
        tile_range(t, tx0, ty0, tx1, ty1);
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) agg_inc(tile_cnt, ty * tiles_x + tx);
    }
    if (sp.lens_mode == HEXFC_LENS_SPHERE && sp.bounded && (flags & (3u * kFaceDrawn))) {
        const float4 px = fstat[f].px, py = fstat[f].py, pz = fstat[f].pz;
        const float o[4][3] = {{px.x - sp.lens_c[0], py.x - sp.lens_c[1], pz.x - sp.lens_c[2]},
                               {px.y - sp.lens_c[0], py.y - sp.lens_c[1], pz.y - sp.lens_c[2]},
                               {px.z - sp.lens_c[0], py.z - sp.lens_c[1], pz.z - sp.lens_c[2]},
                               {px.w - sp.lens_c[0], py.w - sp.lens_c[1], pz.w - sp.lens_c[2]}};
#pragma unroll
        for (int tri = 0; tri < 2; ++tri) {
            const float v[3][3] = {{o[0][0], o[0][1], o[0][2]},
                                   {o[1 + tri][0], o[1 + tri][1], o[1 + tri][2]},
                                   {o[2 + tri][0], o[2 + tri][1], o[2 + tri][2]}};
            const float d[3] = {E[0], E[1 + tri], E[2 + tri]};
            if (outside_lens(v, d, sp.ortho != 0, sp.lens_inv_r)) flags |= kFaceOut << tri;
        }
    }
    float nl[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int k1 = (k + 1) & 3;
        const int32_t ex = X[k1] - X[k], ey = Y[k1] - Y[k];
        const float l2 = u64_to_f32((uint64_t)((int64_t)ex * ex + (int64_t)ey * ey));
        nl[k] = l2 > 0.f ? -(1.f / l2) : 0.f;
    }
    FaceFrame& r = fframe[f];
    r.X = make_int4(X[0], X[1], X[2], X[3]);
    r.Y = make_int4(Y[0], Y[1], Y[2], Y[3]);
    r.Z = make_uint4(Z[0] | (edges << 24), Z[1] | (flags << 24), Z[2], Z[3]);
    r.q = sp.ortho ? make_float4(1.f, 1.f, 1.f, 1.f) : make_float4(1.f / E[0], 1.f / E[1], 1.f / E[2], 1.f / E[3]);
    r.nl = make_float4(nl[0], nl[1], nl[2], nl[3]);
    r.area = make_uint4(area[0], area[1], __float_as_uint(ia[0]), __float_as_uint(ia[1]));
    reinterpret_cast<uint2*>(tzsum)[f] = make_uint2(pack_depths(Z[0], Z[1], Z[2]), pack_depths(Z[0], Z[2], Z[3]));
}

__global__ void k_bin_fill(const FaceFrame* __restrict__ fframe, int64_t n_faces, int W, int H, int tiles_x,
                           int reverse, const uint64_t* __restrict__ tile_off, uint32_t* __restrict__ tile_cur,
                           uint32_t* __restrict__ bins)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_faces) return;
    int64_t f = reverse ? (n_faces - 1 - i) : i;
    const uint32_t tris = face_tris(fframe[f].Z);
    if (tris == 0) return;
    int4 a = fframe[f].X, b = fframe[f].Y;
    int32_t X[4] = {a.x, a.y, a.z, a.w}, Y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int tri = 0; tri < 2; ++tri) {
        if (!(tris & (1u << tri))) continue;
        TriGeom t;
        tri_setup(X, Y, tri, W, H, t);
        int tx0, ty0, tx1, ty1;
        tile_range(t, tx0, ty0, tx1, ty1);
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) {
                int tile = ty * tiles_x + tx;
                const uint32_t slot = agg_inc(tile_cur, tile);
                bins[tile_off[tile] + slot] = (uint32_t)(2 * f + tri);
            }
    }
}

// ------------------------------------------------------------------ bin order

constexpr int kBinSortMax = 4096;   // longer tile lists are sorted through global scratch
constexpr int kDepthBucketsMax = 4096;

// Orders each tile's list front to back by a counting sort of the triangles
// into nb buckets (a power of two, 256..kDepthBucketsMax) of their depth (sum of the three window depths)
// over the tile's depth range; the padding slots stay at the end. Any order
// gives the same image; this one makes every pixel meet its fragments sorted or
// nearly sorted (order within a bucket is arbitrary). zsuf receives, per chunk,
// a lower bound of the depths of the triangles from that chunk on: a pixel that
// is opaque in front of it is finished.
__global__ void __launch_bounds__(256) k_bin_sort(const uint64_t* __restrict__ tile_off,
                                                  const uint32_t* __restrict__ tile_cnt, uint32_t* __restrict__ bins,
                                                  const uint32_t* __restrict__ tzsum, int nb,
                                                  float* __restrict__ tile_zr, uint32_t* __restrict__ tmp,
                                                  uint32_t* __restrict__ zsuf)
{
    constexpr int kItems = kBinSortMax / 256;   // entries per thread of a list held in registers
    __shared__ uint32_t s_hist[kDepthBucketsMax];
    __shared__ uint32_t s_out[kBinSortMax];
    __shared__ uint32_t s_red[2][8];
    __shared__ uint32_t s_low[kBinSortMax / kChunk];   // least depth of each chunk
    const int tile = blockIdx.x;
    const uint64_t beg = tile_off[tile];
    const uint32_t n = tile_cnt[tile];   // real entries; the rest of the padded list is kPadBin
    if (n < 2) {   // nothing to order; depth range 0
        if (threadIdx.x == 0) {
            tile_zr[tile] = 0.f;
            if (n) zsuf[beg / kChunk] = 0u;
        }
        return;
    }
    const uint32_t n_chunks = (n + kChunk - 1) / kChunk;
    const bool big = n > (uint32_t)kBinSortMax;   // entries re-read, scatter through tmp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a list of up to kBinSortMax entries is read once: entry tid + 256 k of
    // the list and its triangle's depth sum (sum of the three window depths)
    // stay in this thread's registers
    uint32_t f2t[kItems], zs[kItems];
    uint32_t zmin = 0xFFFFFFFFu, zmax = 0;
    if (!big) {
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t i = threadIdx.x + 256u * k;
            f2t[k] = i < n ? bins[beg + i] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint32_t i = threadIdx.x + 256u * k;
            zs[k] = i < n ? tzsum[f2t[k]] : 0u;
            if (i < n) {
                zmin = min(zmin, zs[k] & kZSum);
                zmax = max(zmax, zs[k] & kZSum);
            }
        }
    } else {
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t z = tzsum[bins[beg + i]] & kZSum;
            zmin = min(zmin, z);
            zmax = max(zmax, z);
        }
    }
    for (int i = threadIdx.x; i < nb; i += blockDim.x) s_hist[i] = 0;
    if (threadIdx.x < kBinSortMax / kChunk) s_low[threadIdx.x] = 0xFFFFFFFFu;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        zmin = min(zmin, __shfl_xor_sync(0xffffffffu, zmin, o));
        zmax = max(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    }
    if (lane == 0) { s_red[0][warp] = zmin; s_red[1][warp] = zmax; }
    __syncthreads();
    zmin = s_red[0][0];
    zmax = s_red[1][0];
    for (int w = 1; w < 8; ++w) { zmin = min(zmin, s_red[0][w]); zmax = max(zmax, s_red[1][w]); }
    const float scale = (float)nb / (float)(zmax - zmin + 1);
    if (threadIdx.x == 0) tile_zr[tile] = (float)(zmax - zmin) * (1.f / 50331648.f);   // of 3 * 2^24
    auto bucket = [&](uint32_t z) -> int { return min((int)((float)((z & kZSum) - zmin) * scale), nb - 1); };
    // histogram
    if (!big) {
#pragma unroll
        for (int k = 0; k < kItems; ++k)
            if (threadIdx.x + 256u * k < n) atomicAdd(&s_hist[bucket(zs[k])], 1u);
    } else {
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&s_hist[bucket(tzsum[bins[beg + i]])], 1u);
    }
    __syncthreads();
    // exclusive scan of the histogram: nb / 256 buckets per thread
    {
        const int per = nb / 256;
        uint32_t v[kDepthBucketsMax / 256], sum = 0;
#pragma unroll
        for (int k = 0; k < kDepthBucketsMax / 256; ++k) {
            v[k] = k < per ? s_hist[threadIdx.x * per + k] : 0u;
            sum += v[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();   // everyone has read s_hist
        if (lane == 31) s_red[0][warp] = incl;
        __syncthreads();
        uint32_t base = incl - sum;
        for (int w = 0; w < warp; ++w) base += s_red[0][w];
#pragma unroll
        for (int k = 0; k < kDepthBucketsMax / 256; ++k) {
            if (k < per) s_hist[threadIdx.x * per + k] = base;
            base += v[k];
        }
    }
    __syncthreads();
    // scatter (arbitrary order inside a bucket), then write back
    if (!big) {
#pragma unroll
        for (int k = 0; k < kItems; ++k)
            if (threadIdx.x + 256u * k < n) {
                const uint32_t at = atomicAdd(&s_hist[bucket(zs[k])], 1u);
                s_out[at] = f2t[k];
                atomicMin(&s_low[at / kChunk], packed_least(zs[k]));
            }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) bins[beg + i] = s_out[i];
        if (warp == 0) {   // the least from each chunk on: four chunks a lane
            constexpr int kPer = kBinSortMax / kChunk / 32;
            uint32_t v[kPer], low = 0xFFFFFFFFu;
#pragma unroll
            for (int k = kPer - 1; k >= 0; --k) {
                low = min(low, s_low[lane * kPer + k]);
                v[k] = low;
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {   // over the higher lanes
                const uint32_t y = __shfl_down_sync(0xffffffffu, low, o);
                if (lane + o < 32) low = min(low, y);
            }
            uint32_t after = __shfl_down_sync(0xffffffffu, low, 1);
            if (lane == 31) after = 0xFFFFFFFFu;
#pragma unroll
            for (int k = 0; k < kPer; ++k)
                if ((uint32_t)(lane * kPer + k) < n_chunks) zsuf[beg / kChunk + lane * kPer + k] = min(v[k], after);
        }
    } else {
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t f = bins[beg + i];
            tmp[beg + atomicAdd(&s_hist[bucket(tzsum[f])], 1u)] = f;
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n_chunks * kChunk; i += blockDim.x) {   // (a warp: one chunk)
            uint32_t low = 0xFFFFFFFFu;
            if (i < n) {
                const uint32_t f = tmp[beg + i];
                bins[beg + i] = f;
                low = packed_least(tzsum[f]);
            }
            low = __reduce_min_sync(0xffffffffu, low);
            if (lane == 0) zsuf[(beg + i) / kChunk] = low;
        }
        __syncthreads();
        if (warp == 0) {   // the least from each chunk on, 32 chunks at a time from the end
            uint32_t after = 0xFFFFFFFFu;
            for (int c0 = (int)((n_chunks - 1) & ~31u); c0 >= 0; c0 -= 32) {
                uint32_t* z = zsuf + beg / kChunk + c0 + lane;
                const bool in = (uint32_t)(c0 + lane) < n_chunks;
                uint32_t low = in ? *z : 0xFFFFFFFFu;
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

// The tiles in decreasing order of their number of chunks (a counting sort),
// so that the per-tile passes start the longest tiles first and the shortest
// ones fill the tail of the launch. Order inside a class is arbitrary; no
// result depends on it. One block.
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
// scal[0..2].
// The count of one tile (the body of k_count and k_count_batch).
__device__ __forceinline__ void count_tile(int tile, const CountItem& a)
{
    extern __shared__ __align__(16) unsigned char count_smem[];
    CountWarp* s_w = reinterpret_cast<CountWarp*>(count_smem);   // [kConsumerWarps]
    const int px0 = (tile % a.tiles_x) * kTileW, py0 = (tile / a.tiles_x) * kTileH;
    const uint64_t beg = a.tile_off[tile], end = a.tile_off[tile + 1];  // multiples of kChunk
    const uint32_t n_chunks = (uint32_t)((end - beg) / kChunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    count_chunks(s_w, warp, lane, a.bins, a.fframe, beg, n_chunks, px0, py0, a.W, a.H, a.masks);
    __syncthreads();
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < kConsumerWarps; ++w) n += s_w[w].mask[threadIdx.x];
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
    }
}

__global__ void __launch_bounds__(kTilePix, 5) k_count(const __grid_constant__ CountItem a)
{
    count_tile((int)a.order[blockIdx.x], a);
}

// The count of several frames in one grid (a batch).
__global__ void __launch_bounds__(kTilePix, 5) k_count_batch(const __grid_constant__ CountBatch b)
{
    const int i = batch_item(b.tile_begin, b.n, blockIdx.x);
    count_tile((int)b.it[i].order[blockIdx.x - b.tile_begin[i]], b.it[i]);
}

}  // namespace

cudaError_t prepare_raster_kernels()
{
    cudaError_t e = cudaFuncSetAttribute(k_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kConsumerWarps * sizeof(CountWarp)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_count_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kConsumerWarps * sizeof(CountWarp)));
    return e;
}

cudaError_t launch_vertex_setup(const DevMesh& m, const CamParams& cam, FrameBufs& fb, cudaStream_t s)
{
    k_vertex_setup<<<grid_for(m.n_verts, 256), 256, 0, s>>>(m.verts, m.n_verts, cam, cam_pairs(cam), fb.vproj, fb.ved);
    return cudaGetLastError();
}

cudaError_t launch_face_setup(const DevMesh& m, const CamParams& cam, const ShadeParams& sp, FrameBufs& fb,
                              int tiles_x, int tiles_y, cudaStream_t s)
{
    (void)tiles_y;
    k_face_setup<<<grid_for(m.n_faces, 256), 256, 0, s>>>(m.fverts, m.fedges, m.fbound, m.fstat.get(), m.elevel,
                                                           m.eattr, fb.vproj, fb.ved, m.n_faces, sp, cam.W, cam.H,
                                                           tiles_x, fb.fframe, fb.tzsum, fb.tile_cnt);
    return cudaGetLastError();
}

cudaError_t launch_bin_fill(const DevMesh& m, FrameBufs& fb, int tiles_x, int W, int H, int reverse,
                            cudaStream_t s)
{
    k_bin_fill<<<grid_for(m.n_faces, 256), 256, 0, s>>>(fb.fframe, m.n_faces, W, H, tiles_x, reverse,
                                                         fb.tile_off, fb.tile_cur, fb.bins);
    return cudaGetLastError();
}

cudaError_t launch_bin_sort(const DevMesh& m, FrameBufs& fb, int tiles_x, int tiles_y, int64_t n_bins, int buckets,
                            cudaStream_t s)
{
    (void)m;
    if (buckets == 0) {   // no depth order (lists keep the faces' arrival order); depth ranges unknown
        const cudaError_t e = cudaMemsetAsync(fb.tile_zr, 0, sizeof(float) * (size_t)tiles_x * tiles_y, s);
        if (e != cudaSuccess) return e;
        return cudaMemsetAsync(fb.zsuf, 0, sizeof(uint32_t) * (size_t)(n_bins / kChunk), s);
    }
    k_bin_sort<<<(unsigned)(tiles_x * tiles_y), 256, 0, s>>>(fb.tile_off, fb.tile_cnt, fb.bins, fb.tzsum, buckets,
                                                              fb.tile_zr, fb.bins_tmp, fb.zsuf);
    return cudaGetLastError();
}

cudaError_t launch_tile_order(FrameBufs& fb, int n_tiles, cudaStream_t s)
{
    k_tile_order<<<1, 1024, 0, s>>>(fb.tile_off, n_tiles, fb.tile_order);
    return cudaGetLastError();
}

CountItem count_item(const FrameBufs& fb, int tiles_x, int tiles_y, int W, int H)
{
    return CountItem{fb.tile_off, fb.bins, fb.fframe, fb.tile_order, fb.cnt, fb.masks, fb.tile_frag,
                     reinterpret_cast<unsigned long long*>(fb.scal), tiles_x, W, H, tiles_x * tiles_y};
}

cudaError_t launch_count(FrameBufs& fb, int tiles_x, int tiles_y, int W, int H, cudaStream_t s)
{
    k_count<<<(unsigned)(tiles_x * tiles_y), kTilePix, kConsumerWarps * sizeof(CountWarp), s>>>(
        count_item(fb, tiles_x, tiles_y, W, H));
    return cudaGetLastError();
}

cudaError_t launch_count_batch(const CountBatch& b, cudaStream_t s)
{
    const size_t smem = kConsumerWarps * sizeof(CountWarp);
    if (b.n == 0 || b.tile_begin[b.n] == 0) return cudaSuccess;
    k_count_batch<<<b.tile_begin[b.n], kTilePix, smem, s>>>(b);
    return cudaGetLastError();
}

}  // namespace hexfc
