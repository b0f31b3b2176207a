// Drawing pass of the renderer: every covered sample is shaded and blended in
// one kernel, front to back, without its fragment being stored.
//
//   k_draw        per tile: each pixel's covered triangles (from the count
//                 pass's masks, in the tile's depth order) are shaded with
//                 Eqs. 1-4 and blended through a small window of the last ones
//                 met
//   k_draw_wide   the same with more staging, for few tiles
//   k_draw_tail   the pixels whose triangles did not come in depth order: their
//                 list is sorted by key, then shaded and blended
//   k_silhouette  white silhouettes from the boundary surface's depths
//   k_debug_*     sorted lists of requested pixels
//
// Each face is drawn as two triangles (Section "Method Overview"; Section "GPU
// Implementation"), all covered samples take part, sorted by increasing
// distance to the camera and blended in visibility order (Section "Method
// Overview"; Section "GPU Implementation"), and the fragment shader computes
// focus from the lens, the edge distance to the four face edges ignoring
// invisible ones, and Eqs. 1-4 (Section "Focus+Context").
//
// The paper stores the fragments in per-pixel lists and sorts each with a
// priority queue. Here the triangles of a tile are sorted by depth before they
// are rasterised, so a pixel meets its fragments in order or nearly so, and
// blends them as they come. Keys (depth, face, triangle) are unique within a
// pixel, so the order is unique, and every path blends a list one element
// after the other in that order with the same operations: the image does not
// depend on which path resolved a pixel, nor on the window's size, bit for bit.
#include "draw_slot.h"
#include "pipeline.cuh"
#include "shade.cuh"

namespace hexfc {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = kTilePix / 32;          // a warp per group of 32 pixels
constexpr uint32_t kService = 8;               // steps between two looks at the ring (a power of two)
// Chunks staged ahead, and warps that only stage (none: the eight that draw stage too, a slot each).
__host__ __device__ constexpr int ring_of(bool wide) { return wide ? 16 : kWarps; }
__host__ __device__ constexpr int stagers_of(bool wide) { return wide ? 8 : 0; }
static_assert((ring_of(false) & (ring_of(false) - 1)) == 0 && (ring_of(true) & (ring_of(true) - 1)) == 0,
              "slots by the low bits");
constexpr uint32_t kGone = 0xffffffffu;        // progress of a warp that needs no more chunks
constexpr unsigned long long kErrWait = 4ull;  // error bits
constexpr unsigned long long kErrDepth = 1ull;

struct CT { float r, g, b, t; };  // premultiplied colour and transmittance

__device__ __forceinline__ CT ct_over(CT a, const float4& f)  // a in front of fragment f
{
    const float tb = 1.f - f.w;
    return CT{fmaf(a.t, f.x, a.r), fmaf(a.t, f.y, a.g), fmaf(a.t, f.z, a.b), __fmul_rn(a.t, tb)};
}

__device__ __forceinline__ float4 finish(CT c, const ShadeParams& sp)
{
    return make_float4(fmaf(c.t, sp.bg[0], c.r), fmaf(c.t, sp.bg[1], c.g), fmaf(c.t, sp.bg[2], c.b), 1.f - c.t);
}

// The pixel of its tile that thread t of a drawing block owns: a warp's are a group of 8x4.
__device__ __forceinline__ int draw_pixel(int t)
{
    constexpr int kGx = kTileW / 8;
    const int warp = t >> 5, lane = t & 31;
    return ((warp / kGx) * 4 + (lane >> 3)) * kTileW + (warp % kGx) * 8 + (lane & 7);
}

// Output index of drawn pixel (x, y), if it belongs to the output window.
__device__ __forceinline__ bool out_index(const OutWin& w, int x, int y, int64_t& o)
{
    const int u = x - w.x0, v = y - w.y0;
    if (u < 0 || v < 0 || u >= w.w || v >= w.h) return false;
    o = (int64_t)v * w.w + u;
    return true;
}

// Whether the frame may be drawn: no error reported and not yet cleared, its
// longest list within what the sort takes, its lists within the budget
// (scal: see kScal).
__device__ __forceinline__ bool frame_allowed(const DrawItem& a)
{
    const unsigned long long* scal = a.scal;
    return scal[5] == 0 && scal[1] <= (unsigned long long)HEXFC_MAX_LIST && scal[0] <= a.limit && scal[8] <= a.bin_limit;
}

// ------------------------------------------------------------------ staging

// A ring slot: the records of one chunk (draw_slot.h), and its masks in the
// consumers' order (the 32 pixels of a warp's group one after the other).
struct DrawSlot {
    ShadeRec sh[slot_records(kChunk)];
    uint32_t mask[kTilePix];
};

template <int KW, bool kWide>
struct DrawRing {
    static constexpr int kRing = ring_of(kWide);
    DrawSlot ring[kRing];
    float4 window[KW][kTilePix];
    uint64_t full[kRing];               // a slot is staged (the 32 lanes of the warp that staged it arrive)
    uint32_t rel[kWarps];               // chunks that a warp is past (kGone: it needs no more)
};

// ------------------------------------------------------------------ blending window

// The last KW fragments of a pixel: (z + 1, f2t) as the key, so that the places
// start out holding transparent fragments with keys before any real one
// (blending those changes nothing). Each new fragment takes the place of the
// least, which is blended; one before all of them is blended at once, and only
// there can the order of blending break (what stays is never before what was
// blended): the list then has to be sorted. Keys in registers, colours in shared
// memory: moving them between registers cost more than a store and a load.
template <int KW>
struct Window {
    uint64_t k[KW];
    float4* c;   // this pixel's colours, kTilePix apart
    CT acc;
    uint64_t last;
    bool ok;
    __device__ __forceinline__ void init(float4* colours)
    {
        c = colours;
#pragma unroll
        for (int i = 0; i < KW; ++i) {
            k[i] = (uint64_t)(i + 1);
            c[i * kTilePix] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        acc = CT{0.f, 0.f, 0.f, 1.f};
        last = 0;
        ok = true;
    }
    __device__ __forceinline__ int least_place() const
    {
        uint64_t v = k[0];
        int at = 0;
#pragma unroll
        for (int i = 1; i < KW; ++i) {
            at = k[i] < v ? i : at;
            v = k[i] < v ? k[i] : v;
        }
        return at;
    }
    __device__ __forceinline__ void push(uint64_t key, const float4& f)
    {
        const int at = least_place();
        uint64_t v = k[0];
#pragma unroll
        for (int i = 1; i < KW; ++i) v = at == i ? k[i] : v;
        if (key < v) {
            ok = ok && key > last;
            last = key;
            acc = ct_over(acc, f);
        } else {
            last = v;
            acc = ct_over(acc, c[at * kTilePix]);
            c[at * kTilePix] = f;
#pragma unroll
            for (int i = 0; i < KW; ++i) k[i] = at == i ? key : k[i];
        }
    }
    __device__ __forceinline__ void flush()
    {
#pragma unroll
        for (int n = 0; n < KW; ++n) {
            const int at = least_place();
            acc = ct_over(acc, c[at * kTilePix]);
#pragma unroll
            for (int i = 0; i < KW; ++i) k[i] = at == i ? ~0ull : k[i];
        }
    }
};

// ------------------------------------------------------------------ lists of single pixels

struct PixelRef {   // a pixel of the drawn rectangle
    int tile, px0, py0, lx, ly, p;
};
__device__ __forceinline__ PixelRef pixel_ref(int64_t q, int tiles_x)
{
    PixelRef r;
    r.tile = (int)(q / kTilePix);
    r.p = (int)(q % kTilePix);
    r.px0 = (r.tile % tiles_x) * kTileW;
    r.py0 = (r.tile / tiles_x) * kTileH;
    r.lx = r.p % kTileW;
    r.ly = r.p / kTileW;
    return r;
}

// The triangles covering a pixel, in the tile's order: f(i, f2t) for element
// i < limit, found by one whole warp, 32 chunks' masks at a time.
template <class F>
__device__ __forceinline__ void list_walk(const DrawItem& a, const PixelRef& r, int lane, uint32_t limit, F&& f)
{
    const uint64_t cb = a.tile_off[r.tile] / kChunk, ce = cb + a.tile_chunks[r.tile];
    uint32_t k = 0;
    for (uint64_t c0 = cb; c0 < ce; c0 += 32) {
        const uint64_t c = c0 + lane;
        uint32_t m = c < ce ? a.masks[c * kTilePix + r.p] : 0u;
        const uint32_t h = __popc(m);
        uint32_t incl = h;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        for (uint32_t i = k + incl - h; m != 0; ++i) {
            const int j = __ffs(m) - 1;
            m &= m - 1;
            if (i < limit) f(i, a.bins[c * kChunk + j]);
        }
        k += __shfl_sync(kFull, incl, 31);
    }
}

// One fragment on its own: its key (depth << 32 | f2t) and colour, by the same
// operations as the drawing pass.
__device__ __forceinline__ uint64_t fragment_key(const DrawItem& a, const PixelRef& r, uint32_t f2t, bool& bad)
{
    const FaceFrame& ff = a.fframe[f2t >> 1];
    const int4 X = ff.X, Y = ff.Y;
    const uint4 Z = ff.Z;
    const int32_t FX[4] = {X.x, X.y, X.z, X.w}, FY[4] = {Y.x, Y.y, Y.z, Y.w};
    const uint32_t zz[4] = {Z.x & kZ24, Z.y & kZ24, Z.z & kZ24, Z.w & kZ24};
    TriGeom t;
    tri_wind(FX, FY, (int)(f2t & 1u), t);
    uint32_t z[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int cc = t.vi[k];
        z[k] = cc == 0 ? zz[0] : cc == 1 ? zz[1] : cc == 2 ? zz[2] : zz[3];
    }
    const int32_t sx = 256 * (r.px0 + r.lx) + 128, sy = 256 * (r.py0 + r.ly) + 128;
    const int64_t l1 = edge_fn(t.X[2], t.Y[2], t.X[0], t.Y[0], sx, sy);
    const int64_t l2 = edge_fn(t.X[0], t.Y[0], t.X[1], t.Y[1], sx, sy);
    const uint32_t zv = sample_depth(z[0], (int64_t)z[1] - (int64_t)z[0], (int64_t)z[2] - (int64_t)z[0], l1, l2,
                                     t.area, bad);
    return ((uint64_t)zv << 32) | f2t;
}

// kKept: with the importances that the frame has kept itself (dc), not the mesh's.
template <bool kKept>
__device__ __noinline__ float4 fragment_colour(const DrawItem& a, const DrawnCorners& dc, const PixelRef& r, uint32_t f2t,
                                               bool& bad)
{
    ShadeRec R;
    if constexpr (kKept) {
        FaceStatic S = a.fstat[f2t >> 1];
        const int4 v = dc.fverts[f2t >> 1];
        S.imp = make_float4(importance_of(dc.vproj[v.x].w), importance_of(dc.vproj[v.y].w), importance_of(dc.vproj[v.z].w),
                            importance_of(dc.vproj[v.w].w));
        make_record(a.fframe[f2t >> 1], S, nullptr, f2t, r.px0, r.py0, a.sp, R);
    } else {
        make_record(a.fframe[f2t >> 1], a.fstat[f2t >> 1], nullptr, f2t, r.px0, r.py0, a.sp, R);
    }
    const Sample s = sample_of(R, R.zf, R.ha, (uint32_t)r.lx << 8, (uint32_t)r.ly << 8, true, bad);
    const int x = r.px0 + r.lx, y = r.py0 + r.ly;
    const float dist = a.sp.lens_mode == HEXFC_LENS_SCREEN ? screen_lens_dist(x, y, a.sp) : 0.f;
    return shade_fragment(R, R.zf.x >> 24, s.lam1, s.lam2, (float)(256 * x + 128), (float)(256 * y + 128), dist, a.sp);
}

struct PixelList {   // the list of one pixel in a block's shared memory
    uint64_t k[HEXFC_MAX_LIST];
    float4 c[kTilePix];
};

// The n <= HEXFC_MAX_LIST fragments of pixel r, sorted and blended by a block
// of kTilePix threads (thread 0 has the colour); if out_key is given, the
// sorted list is written. A fragment a thread: up to kTilePix of them each
// thread finds the rank of its own key, beyond that a bitonic sort; then they
// are shaded kTilePix at a time, and blended by thread 0.
template <bool kKept>
__device__ __noinline__ CT block_list(const DrawItem& a, const DrawnCorners& dc, const PixelRef& r, uint32_t n, PixelList& L,
                                      uint64_t* out_key, float4* out_rgba, bool& bad)
{
    if (threadIdx.x < 32)
        list_walk(a, r, (int)threadIdx.x, n, [&](uint32_t i, uint32_t f2t) { L.k[i] = f2t; });
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += kTilePix) L.k[i] = fragment_key(a, r, (uint32_t)L.k[i], bad);
    __syncthreads();
    if (n <= (uint32_t)kTilePix) {
        const uint64_t key = threadIdx.x < n ? L.k[threadIdx.x] : kPadKey;
        uint32_t rank = 0;
        for (uint32_t i = 0; i < n; ++i) rank += L.k[i] < key ? 1u : 0u;
        __syncthreads();
        if (threadIdx.x < n) L.k[rank] = key;
        __syncthreads();
    } else {
        uint32_t np2 = 2 * kTilePix;
        while (np2 < n) np2 <<= 1;
        for (uint32_t i = n + threadIdx.x; i < np2; i += kTilePix) L.k[i] = kPadKey;
        __syncthreads();
        for (uint32_t size = 2; size <= np2; size <<= 1)
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                for (uint32_t i = threadIdx.x; i < np2; i += kTilePix) {
                    const uint32_t p = i ^ stride;
                    if (p > i) {
                        const bool up = (i & size) == 0;
                        const uint64_t u = L.k[i], v = L.k[p];
                        if (up ? (u > v) : (u < v)) {
                            L.k[i] = v;
                            L.k[p] = u;
                        }
                    }
                }
                __syncthreads();
            }
    }
    CT c{0.f, 0.f, 0.f, 1.f};
    for (uint32_t b = 0; b < n; b += kTilePix) {
        const uint32_t i = b + threadIdx.x;
        if (i < n) {
            const uint64_t key = L.k[i];
            const float4 f = fragment_colour<kKept>(a, dc, r, (uint32_t)key, bad);
            L.c[threadIdx.x] = f;
            if (out_key) {
                out_key[i] = key;
                out_rgba[i] = f;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const uint32_t e = min(n - b, (uint32_t)kTilePix);
#pragma unroll 4
            for (uint32_t j = 0; j < e; ++j) c = ct_over(c, L.c[j]);
        }
        __syncthreads();
    }
    return c;
}

// The pixels k_draw found out of order, queued by it (the queue's length is
// read on the device, so the grid need not match it), a block each: there are
// few of them, so what counts is how long one takes (a warp each took 43 us for
// the 20 pixels of the 64^3 frame at 1920x1080, a block each 14).
__global__ void __launch_bounds__(kTilePix, 3) k_draw_tail(const __grid_constant__ DrawItem a)
{
    chain_begin();
    extern __shared__ __align__(128) unsigned char smem[];
    if (!__syncthreads_and(frame_allowed(a))) return;
    bool bad = false;
    const uint64_t n_redo = *a.redo_cursor;
    for (uint64_t i = blockIdx.x; i < n_redo; i += gridDim.x) {
        const uint32_t q = a.redo[i];
        const PixelRef r = pixel_ref(q, a.tiles_x);
        const CT c = block_list<false>(a, DrawnCorners{}, r, min(a.cnt[q], (uint32_t)HEXFC_MAX_LIST),
                                       *reinterpret_cast<PixelList*>(smem), nullptr, nullptr, bad);
        int64_t o;
        if (threadIdx.x == 0 && out_index(a.win, r.px0 + r.lx, r.py0 + r.ly, o)) a.out[o] = finish(c, a.sp);
        __syncthreads();   // the list is the next pixel's
    }
    if (bad) atomicOr(a.err, kErrDepth);
}

// ------------------------------------------------------------------ draw

__device__ __forceinline__ void store_release(uint32_t* p, uint32_t v)
{
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_addr(p)), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t load_acquire(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_addr(p)) : "memory");
    return v;
}

// The chunks of a tile's list go through a ring of kRing slots (records ready
// to shade, one lane per triangle). Warp w stages chunks w, w + 8, ..., each as
// soon as every warp is past the chunk its slot held; one warp staging for all
// was what the others waited for (1.00 ms of what is 0.73 now). A warp's 32 lanes
// are a group of 8x4 pixels. Each lane
// goes through its own covered triangles: in each step of the warp every lane
// shades the next triangle of its pixel, whichever chunk of the ring that is
// in, so a pixel with few triangles in one chunk goes on to the next while its
// neighbours are still busy, and the lanes stay occupied without a queue. Slots
// are handed over with one mbarrier each (staged) and one progress counter per
// warp (the chunks all its lanes are past), looked after every few steps.
//
// A fragment behind an opaque one (transmittance exactly 0) is not shaded, only
// its order is checked, and once every triangle of the following chunks lies
// behind the last blended one (zsuf: the least depth from a chunk on) the
// pixel is finished; a warp whose pixels are all finished only stages, and the
// block ends when all have.
//
// Bound by instruction issue: 64^3 at 1920x1080, 77.6 M fragments (mean of an
// orbit) in 0.724 ms (the pass that stored 24-byte fragments and the one that read
// and blended them: 0.91 + 0.39 ms, 4.2 GB of DRAM), at 8.8 warp instructions a
// fragment, of which the edge distances of Eq. 1 are about 3; 128^3 at 3840x2160,
// 604 M fragments, 4.98 ms. Three blocks an SM
// of 80 registers (two or four: 6% and 10% slower); kService steps between looks at
// the ring 8 (4, 16, 32: 1-2% slower).
template <int KW, bool kSil, bool kWide>
__device__ __forceinline__ void draw_tile(DrawRing<KW, kWide>& S, const DrawItem& a, int tile)
{
    constexpr int kRing = ring_of(kWide), kStagers = stagers_of(kWide), kStep = kWide ? kStagers : kWarps;
    const bool allowed = frame_allowed(a);
    const int px0 = (tile % a.tiles_x) * kTileW, py0 = (tile / a.tiles_x) * kTileH;
    const uint64_t beg = a.tile_off[tile];   // a multiple of kChunk
    const uint32_t n_chunks = a.tile_chunks[tile];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < kRing) mbar_init(&S.full[threadIdx.x], 32);
    if (threadIdx.x < kWarps) S.rel[threadIdx.x] = 0;
    constexpr int kWords = sizeof(ShadeRec) / sizeof(uint32_t);   // the slots' blank records
    for (int i = threadIdx.x; i < kRing * kWords; i += blockDim.x)
        reinterpret_cast<uint32_t*>(&S.ring[i / kWords].sh[kSlotBlank])[i % kWords] = 0u;
    mbar_init_fence();
    if (!__syncthreads_and(allowed)) return;   // (one answer for the block: another may set an error bit meanwhile)
    // staging: this warp's next chunk and its triangles
    uint32_t mine = (uint32_t)(kWide ? warp - kWarps : warp);   // (the wide form's consumers: not used)
    uint32_t f2t_m = mine < n_chunks ? a.bins[beg + (uint64_t)mine * kChunk + lane] : kPadBin;
    auto stage = [&]() {
        DrawSlot& D = S.ring[kWide ? mine & (kRing - 1) : warp];
        // the masks: eight pixels of a row a lane
        const uint4* mp = reinterpret_cast<const uint4*>(a.masks + (beg / kChunk + mine) * kTilePix) + 2 * lane;
        const int mx = (8 * lane) % kTileW, my = (8 * lane) / kTileW;
        uint4* md = reinterpret_cast<uint4*>(&D.mask[((my / 4) * (kTileW / 8) + mx / 8) * 32 + (my % 4) * 8]);
        const uint4 ma = mp[0], mb = mp[1];
        if (f2t_m != kPadBin)
            make_record(a.fframe[f2t_m >> 1], a.fstat[f2t_m >> 1], a.fextra ? a.fextra + (f2t_m >> 1) : nullptr, f2t_m, px0,
                        py0, a.sp, D.sh[slot_place(lane)]);
        md[0] = ma;
        md[1] = mb;
        mbar_arrive(&S.full[kWide ? mine & (kRing - 1) : warp]);
        mine += kStep;
        f2t_m = mine < n_chunks ? a.bins[beg + (uint64_t)mine * kChunk + lane] : kPadBin;
    };
    // the least progress of the block's warps (kGone: all are finished). What those
    // warps read before it comes before what any lane of this one writes after it: a
    // lane's acquire is the warp's by the __syncwarp (the reduction orders no memory).
    auto slowest = [&]() {
        const uint32_t r = __reduce_min_sync(kFull, lane < kWarps ? load_acquire(&S.rel[lane]) : kGone);
        __syncwarp();
        return r;
    };
    // what is left to stage, as slots become free. The wait is bounded from the last
    // progress of the slowest warp: a tile may take longer than a wait.
    auto stage_rest = [&]() {
        long long t0 = clock64();
        uint32_t seen = 0;
        while (mine < n_chunks) {
            const uint32_t r = slowest();
            if (r == kGone) break;
            if (r != seen) {
                seen = r;
                t0 = clock64();
            }
            if (mine < r + kRing) {
                stage();
            } else {
                if (__any_sync(kFull, clock64() - t0 > kWaitCycles)) {
                    if (lane == 0) atomicOr(a.err, kErrWait);
                    break;
                }
                __nanosleep(kWide ? 40 : 200);
            }
        }
    };
    if (kWide && warp >= kWarps) {
        stage_rest();
        return;
    }
    if (!kWide && mine < n_chunks) stage();
    // consumers
    const int p = draw_pixel(threadIdx.x), lx = p % kTileW, ly = p / kTileW;
    const int x = px0 + lx, y = py0 + ly;
    const float sx = (float)(256 * x + 128), sy = (float)(256 * y + 128);
    float dist = 0.f;
    bool in_lens = !a.sp.bounded;   // within the screen lens: a constant of the pixel
    if (a.sp.lens_mode == HEXFC_LENS_SCREEN) {
        dist = screen_lens_dist(x, y, a.sp);
        in_lens = in_lens || !(dist >= 1.f);
    }
    Window<KW> w;
    w.init(&S.window[0][threadIdx.x]);
    uint32_t zs = kNoDepth;   // nearest boundary fragment (silhouettes)
    bool bad = false;
    bool done = x >= a.W || y >= a.H;   // nothing left to do for this pixel
    bool hidden = false;                // nothing behind shows: opaque, or left to the tail
    uint32_t m = 0;                     // the lane's remaining triangles of its chunk `ch`
    int ch = -1;
    uint32_t hi = 0, rel = 0;           // chunks taken by the warp, chunks released
    uint32_t step = 0;
    long long waited = 0;
    const uint32_t* zsuf = a.zsuf + beg / kChunk;
    for (;;) {
        while (m == 0 && !done && ch + 1 < (int)hi) {   // on to the pixel's next chunk
            ++ch;
            m = S.ring[ch & (kRing - 1)].mask[threadIdx.x];
            if (hidden) {
                // opaque: finished if every triangle from here on lies behind the last
                // blended fragment (out of order: the tail draws the pixel), and none
                // is a nearer boundary fragment
                const uint32_t zn = zsuf[ch];
                if ((!w.ok || (uint32_t)(w.last >> 32) <= zn) && (!kSil || zs <= zn)) {
                    done = true;
                    m = 0;
                }
            }
        }
        const bool act = __any_sync(kFull, m != 0);
        if (!act || (step++ & (kService - 1)) == 0) {
            // release the chunks every lane is past, stage the next one if its slot is free, take what is staged
            const uint32_t lo = __reduce_min_sync(kFull, done ? hi : (uint32_t)(m != 0 ? ch : ch + 1));
            __syncwarp();   // what the lanes read of those chunks comes before lane 0's release
            if (lo > rel) {
                rel = lo;
                if (lane == 0) store_release(&S.rel[warp], rel);
            }
            if (!kWide && mine < n_chunks && mine < min(slowest(), kGone - kRing) + kRing) stage();
            bool got = false;
            while (hi < n_chunks && hi < rel + kRing &&
                   __all_sync(kFull, mbar_test(&S.full[hi & (kRing - 1)], (hi / kRing) & 1u))) {
                ++hi;
                got = true;
            }
            if (got) {
                waited = 0;
                continue;
            }
            if (!act) {
                if (hi >= n_chunks || __all_sync(kFull, done)) break;   // no triangle left, or all finished
                // nothing to do until a chunk is staged
                const long long now = clock64();
                if (waited == 0) waited = now;
                if (__any_sync(kFull, now - waited > kWaitCycles)) {
                    if (lane == 0) atomicOr(a.err, kErrWait);
                    break;
                }
                __nanosleep(20);
                continue;
            }
        }
        const bool live = m != 0;   // (a lane without a triangle goes along)
        // (a lane without a triangle: the blank record of its slot; its results go
        // nowhere. Where there are many such lanes they read one of them)
        const ShadeRec& R = S.ring[!kWide || live ? ch & (kRing - 1) : 0].sh[next_place(m)];
        m &= m - 1;   // (0 stays 0)
        const uint4 zf = R.zf, ha = R.ha;
        const Sample q = sample_of(R, zf, ha, (uint32_t)lx << 8, (uint32_t)ly << 8, live, bad);
        const uint64_t key = ((uint64_t)(q.z + 1u) << 32) | zf.w;
        if (kSil && live && (ha.z & kRecBound)) zs = min(zs, q.z);
        const bool need = live && !hidden;
        if (live && hidden) w.ok = w.ok && key > w.last;
        // the least of the three forms of the shading that serves every lane
        float4 c;
        if (__any_sync(kFull, need && (in_lens || (ha.z & (kRecLens | kRecEdge))))) {
            if (__any_sync(kFull, need && (in_lens || (ha.z & kRecLens))))
                c = shade_fragment(R, zf.x >> 24, q.lam1, q.lam2, sx, sy, dist, a.sp);
            else
                c = shade_context<true>(R, zf.x >> 24, q.lam1, q.lam2, sx, sy, a.sp);
        } else {
            c = shade_context<false>(R, 0u, q.lam1, q.lam2, sx, sy, a.sp);
        }
        if (need) {
            w.push(key, c);
            hidden = !w.ok || (w.acc.t == 0.f && a.sp.bounded);
        }
        __syncwarp();
    }
    __syncwarp();
    if (lane == 0) store_release(&S.rel[warp], kGone);
    if (bad) atomicOr(a.err, kErrDepth);
    const int64_t q = (int64_t)tile * kTilePix + p;
    if (kSil) a.zsil[q] = zs;
    w.flush();
    int64_t o;
    if (x < a.W && y < a.H && out_index(a.win, x, y, o)) {   // (else an apron pixel: only its depth is used)
        if (w.ok) a.out[o] = finish(w.acc, a.sp);
        else a.redo[atomicAdd(a.redo_cursor, 1ull)] = (uint32_t)q;
    }
    // this warp's chunks are still to be staged for the others
    __syncwarp();
    if (!kWide) stage_rest();
}

template <int KW, bool kSil>
__global__ void __launch_bounds__(kTilePix, 3) k_draw(const __grid_constant__ DrawItem a)
{
    chain_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    draw_tile<KW, kSil, false>(*reinterpret_cast<DrawRing<KW, false>*>(smem), a, (int)a.order[blockIdx.x]);
}

// Few tiles with long lists (a large mesh drawn small): what a tile takes decides,
// not what the chip can issue, and most triangles of a chunk are not a warp's
// own. Eight warps draw, eight others stage, and 16 chunks ahead give the lanes
// more to go on with (96^3 at 320x180, 240 tiles: 0.95 ms with the form above, with
// 8 slots and 8 stagers 0.75, 16 and 16 0.67, 16 and 4 0.57, 16 and 8 0.53).
template <int KW, bool kSil>
__global__ void __launch_bounds__(kTilePix + 32 * stagers_of(true), 1) k_draw_wide(const __grid_constant__ DrawItem a)
{
    chain_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    draw_tile<KW, kSil, true>(*reinterpret_cast<DrawRing<KW, true>*>(smem), a, (int)a.order[blockIdx.x]);
}

// The drawing pass of several frames in one grid (a batch).
template <int KW, bool kSil>
__global__ void __launch_bounds__(kTilePix, 3) k_draw_batch(const __grid_constant__ DrawBatch b)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ DrawItem s_it;   // the frame's pointers and constants, read from shared memory
    const int i = batch_item(b.tile_begin, b.n, blockIdx.x);
    if (threadIdx.x == 0) s_it = b.it[i];
    __syncthreads();
    draw_tile<KW, kSil, false>(*reinterpret_cast<DrawRing<KW, false>*>(smem), s_it,
                               (int)s_it.order[blockIdx.x - b.tile_begin[i]]);
}

// ---------------------------------------------------------------- silhouettes

// White silhouettes of the boundary surface (Section "Blending Focus and
// Context": the boundary surface is rendered and fragments along sharp edges
// of its depth buffer are emphasised). zsil holds, per drawn pixel (tile-major),
// the 24-bit depth of its nearest boundary-face fragment (kNoDepth: none). An
// output pixel p with a depth is a silhouette pixel if a 4-neighbour inside the
// frame has none (exterior), or if for a neighbour q and the opposite q' (both
// with depths) D(q) - D(p) > T and |D(q) - 2 D(p) + D(q')| > T (interior: the
// near side of a depth jump; a plane, however steep, has no second
// difference); its colour and opacity move towards white by alpha. The drawn
// rectangle starts at frame pixel (fx0, fy0) and holds every in-frame
// neighbour of the output window (an apron around a sub-rectangle).
__device__ __forceinline__ uint32_t zsil_at(const uint32_t* __restrict__ zsil, int tiles_x, int x, int y)
{
    const int64_t t = (int64_t)(y / kTileH) * tiles_x + x / kTileW;
    return zsil[t * kTilePix + (y % kTileH) * kTileW + (x % kTileW)];
}

__global__ void __launch_bounds__(256) k_silhouette(const __grid_constant__ DrawItem a, int fx0, int fy0, int frame_w,
                                                    int frame_h, float alpha, int64_t T)
{
    chain_begin();
    const OutWin& win = a.win;
    const uint32_t* zsil = a.zsil;
    const int tiles_x = a.tiles_x;
    float4* out = a.out;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)win.w * win.h || !frame_allowed(a)) return;   // (a refused frame leaves its output alone)
    const int x = win.x0 + (int)(i % win.w), y = win.y0 + (int)(i / win.w);
    const uint32_t zp = zsil_at(zsil, tiles_x, x, y);
    if (zp == kNoDepth) return;
    const int dx[4] = {1, -1, 0, 0}, dy[4] = {0, 0, 1, -1};   // k ^ 1: the opposite side
    int64_t zq[4];
    bool has[4];
    bool sil = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int qx = x + dx[k], qy = y + dy[k];
        const bool inside = qx + fx0 >= 0 && qy + fy0 >= 0 && qx + fx0 < frame_w && qy + fy0 < frame_h;
        const uint32_t z = inside ? zsil_at(zsil, tiles_x, qx, qy) : kNoDepth;
        has[k] = z != kNoDepth;
        zq[k] = (int64_t)z;
        sil = sil || (inside && !has[k]);   // exterior: the surface ends here
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int o = k ^ 1;
        if (has[k] && has[o]) {
            const int64_t d1 = zq[k] - (int64_t)zp, d2 = zq[k] - 2 * (int64_t)zp + zq[o];
            sil = sil || (d1 > T && (d2 > T || -d2 > T));   // interior: the near side of a jump
        }
    }
    if (!sil) return;
    float4 c = out[i];
    c.x = fmaf(alpha, 1.f - c.x, c.x);
    c.y = fmaf(alpha, 1.f - c.y, c.y);
    c.z = fmaf(alpha, 1.f - c.z, c.z);
    c.w = fmaf(alpha, 1.f - c.w, c.w);
    out[i] = c;
}

// ---------------------------------------------------------------- debug gather

// Sorted lists of requested pixels written at dst_off[i], a block each, by the
// routine that draws pixels out of order.
__device__ __forceinline__ int64_t pixel_index(int x, int y, int tiles_x)
{
    return ((int64_t)(y / kTileH) * tiles_x + x / kTileW) * kTilePix + (y % kTileH) * kTileW + (x % kTileW);
}

__global__ void __launch_bounds__(kTilePix) k_debug_lists(const __grid_constant__ DrawItem a, const DrawnCorners dc,
                                                          const int32_t* __restrict__ px,
                                                          const int32_t* __restrict__ py,
                                                          const uint64_t* __restrict__ dst_off,
                                                          uint64_t* __restrict__ out_key,
                                                          float4* __restrict__ out_rgba)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int64_t i = blockIdx.x;
    const int64_t q = pixel_index(px[i], py[i], a.tiles_x);
    const uint32_t n = a.cnt[q];
    if (n == 0 || n > (uint32_t)HEXFC_MAX_LIST) return;
    bool bad = false;
    (void)block_list<true>(a, dc, pixel_ref(q, a.tiles_x), n, *reinterpret_cast<PixelList*>(smem), out_key + dst_off[i],
                           out_rgba + dst_off[i], bad);
    if (bad) atomicOr(a.err, kErrDepth);
}

__global__ void k_debug_counts(const uint32_t* __restrict__ cnt, const int32_t* __restrict__ px,
                               const int32_t* __restrict__ py, int64_t n_req, int tiles_x,
                               uint32_t* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_req) out[i] = cnt[pixel_index(px[i], py[i], tiles_x)];
}

constexpr unsigned kTailBlocks = 3 * 152;   // persistent: blocks stride over the queue

// f(kernel tag) for the instantiation of a window size and silhouette variant.
template <template <int, bool> class K, class F>
cudaError_t for_variant(int window, bool sil, F&& f)
{
    if (window == 8) return sil ? f(K<8, true>{}) : f(K<8, false>{});
    if (window == 4) return sil ? f(K<4, true>{}) : f(K<4, false>{});
    return sil ? f(K<2, true>{}) : f(K<2, false>{});
}
template <int KW, bool kSil>
struct DrawKernel {
    static constexpr auto fn = &k_draw<KW, kSil>;
    static constexpr int smem = sizeof(DrawRing<KW, false>);
};
template <int KW, bool kSil>
struct DrawWideKernel {
    static constexpr auto fn = &k_draw_wide<KW, kSil>;
    static constexpr int smem = sizeof(DrawRing<KW, true>);
};
template <int KW, bool kSil>
struct DrawBatchKernel {
    static constexpr auto fn = &k_draw_batch<KW, kSil>;
    static constexpr int smem = sizeof(DrawRing<KW, false>);
};

}  // namespace

cudaError_t prepare_draw_kernels()
{
    for (int window : {2, 4, 8})
        for (bool sil : {false, true}) {
            auto set = [](auto k) {
                return cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem);
            };
            cudaError_t e = for_variant<DrawKernel>(window, sil, set);
            if (e == cudaSuccess) e = for_variant<DrawBatchKernel>(window, sil, set);
            if (e == cudaSuccess) e = for_variant<DrawWideKernel>(window, sil, set);
            if (e != cudaSuccess) return e;
        }
    const cudaError_t e = cudaFuncSetAttribute(k_draw_tail, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(PixelList));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_debug_lists, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PixelList));
}

cudaError_t launch_draw(const DrawItem& a, int64_t n_tiles, uint64_t n_bins, int window, cudaStream_t s)
{
    // The wide form, one block an SM, for a frame that has the chip to itself, lists
    // of some length, and no more tiles than the other form holds at once, or not
    // many more and long lists (sides measured, wide / other, ms a frame: 96^3 at
    // 240 tiles 0.71 / 0.94, 2040 tiles 0.67 / 0.71; 64^3 at 920 tiles 0.30 / 0.32,
    // 2040 tiles equal; 16^3 at 240 tiles 0.076 / 0.080, 920 tiles 0.114 / 0.102; 4^3
    // and 8^3 at 200 tiles, 26 and 78 entries a list: 2-3% slower). In a batch frames
    // fill each other's gaps: 48 thumbnails 16.1 / 14.4 ms.
    const uint64_t t = (uint64_t)n_tiles;
    const bool few = n_bins >= 96 * t && (t <= 2 * 152 || (t < 10000 && t * t * t <= 3200 * n_bins));
    if (a.chained && few)
        return for_variant<DrawWideKernel>(window, a.zsil != nullptr, [&](auto k) {
            return launch_chained(k.fn, (unsigned)n_tiles, kTilePix + 32 * stagers_of(true), k.smem, s, a.chained, a);
        });
    return for_variant<DrawKernel>(window, a.zsil != nullptr, [&](auto k) {
        return launch_chained(k.fn, (unsigned)n_tiles, kTilePix, k.smem, s, a.chained, a);
    });
}

cudaError_t launch_draw_batch(const DrawBatch& b, bool sil, int window, cudaStream_t s)
{
    if (b.n == 0 || b.tile_begin[b.n] == 0) return cudaSuccess;
    return for_variant<DrawBatchKernel>(window, sil, [&](auto k) {
        k.fn<<<b.tile_begin[b.n], kTilePix, k.smem, s>>>(b);
        return cudaGetLastError();
    });
}

cudaError_t launch_draw_tail(const DrawItem& a, cudaStream_t s)
{
    return launch_chained(k_draw_tail, kTailBlocks, kTilePix, sizeof(PixelList), s, a.chained, a);
}

cudaError_t launch_silhouette(const DrawItem& a, int fx0, int fy0, int frame_w, int frame_h, float alpha, float threshold,
                              cudaStream_t s)
{
    const int64_t n = (int64_t)a.win.w * a.win.h;
    if (n == 0) return cudaSuccess;
    return launch_chained(k_silhouette, (unsigned)((n + 255) / 256), 256, 0, s, a.chained, a, fx0, fy0, frame_w, frame_h, alpha,
                          (int64_t)threshold);
}

cudaError_t launch_debug_gather(const DrawItem& a, const DrawnCorners& dc, const int32_t* d_px, const int32_t* d_py, int64_t n,
                                const uint64_t* d_dst_off, uint64_t* d_keys, float4* d_rgba, uint32_t* d_counts,
                                cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (d_counts) {
        k_debug_counts<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a.cnt, d_px, d_py, n, a.tiles_x, d_counts);
        return cudaGetLastError();
    }
    k_debug_lists<<<(unsigned)n, kTilePix, sizeof(PixelList), s>>>(a, dc, d_px, d_py, d_dst_off, d_keys, d_rgba);
    return cudaGetLastError();
}

}  // namespace hexfc

