// Internal declarations of the hexfc CUDA library (not part of the C ABI).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "hexfc.h"
#include "vertex_stage.h"

namespace hexfc {

#ifndef HEXFC_TILE_W
#define HEXFC_TILE_W 16
#endif
constexpr int kTilePix = 256;                  // pixels (= threads) per tile CTA
constexpr int kTileW = HEXFC_TILE_W;           // raster tile width in pixels (a build-time choice)
constexpr int kTileH = kTilePix / kTileW;      // raster tile height
static_assert(kTileW == 8 || kTileW == 16 || kTileW == 32, "tiles of 8x32, 16x16 or 32x8 pixels");
constexpr int kLongList = 256;             // lists longer than this are counted in the frame's statistics
constexpr uint64_t kPadKey = ~0ull;
constexpr int kChunk = 32;                // triangles per raster chunk (one coverage bit each)
constexpr uint32_t kPadBin = 0xFFFFFFFFu; // empty slot: tile lists are padded to whole chunks

// Focus+context constants of the fragment stage (float).
struct ShadeParams {
    int lens_mode;
    float lens_c[3];
    float lens_inv_r;
    float w_base;
    int lod;
    float delta, s;
    float alpha_min, alpha_span;   // alpha_hat = alpha_min + alpha_span * t
    float tf_lo, tf_inv;           // t = clamp((imp - tf_lo) * tf_inv, 0, 1)
    float bg[3];
    float accent_beta, halo_scale, darken, g_min, g_max;
    float zref;
    int ortho;
    float accent_r2;   // (256 * 2/3 * w_base)^2: accentuation radius squared, 1/256-pixel units
    float desat;       // depth cue strength (0 = off)
    bool bounded;      // every style and lens constant is finite and below 1e15: no product of a zero is NaN
    int px_off, py_off;   // drawn rectangle's offset in the frame: pixel (x, y) is frame pixel (x + px_off, ...)
};

// A face as two 64-byte records: the per-frame one (window corners, depths,
// flags, eye depths), written by the face stage of every frame into the
// rendering context's buffers, and the static one (corner importance and world
// position), owned by the mesh and rewritten in place only when importance
// changes, so that contexts can render one resident mesh at the same time.
struct __align__(64) FaceFrame {
    int4 X, Y;            // corner window position, 16.8 fixed point
    uint4 Z;              // bits 0-23: corner window depth (z24). Bits 24-31 of Z.x: edge flags (bits 0-3
                          // visible in focus, 4-7 visible in context); of Z.y: face flags (kFace...)
    float4 q;             // 1 / corner eye depth (1 in an orthographic view)
};
// What a triangle's shading record needs besides, found once per face instead of
// for every tile it touches where there is room for it.
struct __align__(32) FaceExtra {
    float4 nl;            // -1 / squared length of window edge k -> k+1 (0: degenerate)
    uint4 area;           // triangle 0, 1: twice the area if below 2^26, else 0; 1 / the same (float bits)
};
struct __align__(64) FaceStatic {
    float4 imp;           // corner importance
    float4 px, py, pz;    // corner world position
};
static_assert(sizeof(FaceFrame) == 64 && sizeof(FaceStatic) == 64, "two sectors each");
constexpr uint32_t kZ24 = 0xFFFFFFu;
constexpr int32_t kVertexValid = 1 << 24;   // of a projected vertex' depth word
// Face flags, bit t for triangle t where shifted by it.
constexpr uint32_t kFaceDrawn = 1u;      // << t: triangle drawn
constexpr uint32_t kFaceBoundary = 4u;   // a face of one cell
constexpr uint32_t kFaceSwapped = 8u;    // << t: vertices 1 and 2 swapped to wind it to positive area
constexpr uint32_t kFaceOut = 32u;       // << t: wholly outside the sphere lens

// Device scalars of a frame (FrameBufs::scal): 0-2 count pass (fragments,
// longest list, lists longer than kLongList), 3 cursor of the
// drawing pass's queue, 5 device error bits (kept across frames), 6 tiles
// above their chosen capacity, 8-10 tile scan (bin entries, ...), 11-13
// capacity scan (regions' total, ...), 14 records taken from the pool, 15 tiles
// counted. The count pass's statistics follow them: kStatCopies copies of
// (fragments, longest list, long lists, unused), one per tile % kStatCopies
// (tiles adding into one address would queue on it), summed by its last block.
constexpr int kScal = 24;
constexpr int kStatCopies = 32;
constexpr int kScalAll = kScal + 4 * kStatCopies;
__host__ __device__ inline uint32_t face_edge_flags(const uint4& z) { return z.x >> 24; }
__host__ __device__ inline uint32_t face_flags(const uint4& z) { return z.y >> 24; }
__host__ __device__ inline uint32_t face_tris(const uint4& z) { return (z.y >> 24) & 3u; }
constexpr uint32_t kNoDepth = 0xFFFFFFFFu;   // no boundary fragment at a pixel

// Resident mesh (device pointers), see hexfc_upload_mesh.
struct DevMesh {
    int64_t n_verts = 0, n_cells = 0, n_faces = 0, n_edges = 0;
    float* verts = nullptr;        // [V*3]
    int32_t* cells = nullptr;      // [C*8]
    int32_t* cell_edges = nullptr; // [C*12] unique edge id per cell edge
    float* cell_imp = nullptr;     // [C]
    int32_t* vkey = nullptr;       // [V] ordered-int max of incident importance
    int32_t* ekey = nullptr;       // [E]
    float* eattr = nullptr;        // [E]
    uint8_t* elevel = nullptr;     // [E]
    int4* fverts = nullptr;        // [F] canonical corners
    int4* fedges = nullptr;        // [F] unique edge id of local edge k = (c_k, c_k+1)
    uint8_t* fbound = nullptr;     // [F] 1: a boundary face (one cell)
    FaceStatic* fstat = nullptr;   // [F] static face records
};

// An importance as an int of the same order (vkey, ekey), so that atomicMax on
// int is a float max; an unreferenced vertex or edge (INT32_MIN) has 0.
__device__ __forceinline__ int32_t importance_key(float f)
{
    const int32_t i = __float_as_int(f);
    return i >= 0 ? i : (i ^ 0x7FFFFFFF);
}
__device__ __forceinline__ float importance_of(int32_t k)
{
    return k == INT32_MIN ? 0.f : __int_as_float(k >= 0 ? k : (k ^ 0x7FFFFFFF));
}

// Tile-capacity network (4 -> 64 -> 64 -> 1): FP32 master weights, the FP16
// copy the kernels use, Adam moments, and per-tile training values.
constexpr int kCapIn = 4, kCapHid = 64;
constexpr int kCapParams = kCapHid * kCapIn + kCapHid + kCapHid * kCapHid + kCapHid + kCapHid + 1;
struct CapNet {
    float* w = nullptr;
    __half* w16 = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* grad = nullptr;        // [kCapParams + 1]; the last value is the loss
    float* part = nullptr;        // shares of the gradient (cap_partials())
    float* x = nullptr;           // [4 * tiles] features handed in by the caller
    uint32_t* t = nullptr;        // [tiles] counts handed in by the caller
    int64_t tiles = 0;            // capacity of the per-tile arrays
    int64_t step = 0;             // Adam steps taken
    bool ready = false;           // weights set
};

// Per-frame buffers owned by the context.
struct FrameBufs {
    // vertex stage
    // {X, Y, z24 | kVertexValid, importance key}: the key is the frame's own copy, so that its fragments can
    // be found again (hexfc_debug_pixels) after the mesh's importance has changed
    int4* vproj = nullptr;
    float* ved = nullptr;    // eye depth
    int64_t v_cap = 0;
    // faces
    FaceFrame* fframe = nullptr;    // [F] per-frame face records
    uint32_t* tzsum = nullptr;      // [2F] per triangle (2 face + tri): its depths (pack_depths)
    int64_t f_cap = 0;
    // binning of triangles that touch at most 2x2 tiles: each pair's place in its tile's list is found
    // with its count (nullptr: all places are found in a second pass)
    uint2* trange = nullptr;        // [2F] the triangle's tiles (kRange...), its place in the first one's list
    uint4* slots = nullptr;         // [2F] places in the lists of its 2x2 tiles, if more than one
    FaceExtra* fextra = nullptr;    // [F]
    int64_t slot_cap = 0;           // faces of these three
    uint64_t slots_refused = 0;     // the budget that had no room for them
    // tiles
    uint32_t* tile_cnt = nullptr;   // [T+1] pairs whose place is known
    uint32_t* tile_big = nullptr;   // [T+1] the others
    uint32_t* tile_skip = nullptr;  // [T+1] pairs of triangles that cover no sample (with places only)
    uint64_t* tile_off = nullptr;   // [T+1]
    uint32_t* tile_cur = nullptr;   // [T] the binning's places without counts, then the tiles' chunks
    uint32_t* tile_order = nullptr; // [T] tiles by decreasing chunk count
    uint32_t* tile_frag = nullptr;  // [T] exact fragments per tile (the count's)
    float* cap_x = nullptr;         // [4T] capacity-network features of the frame
    uint32_t* tile_cap = nullptr;   // [T+1] chosen fragment capacity per tile (predicted frames)
    uint64_t* cap_off = nullptr;    // [T+1] its exclusive prefix
    int64_t cap_cap = 0;
    int64_t t_cap = 0;
    uint32_t* bins = nullptr;       // face2tri ids grouped by tile, each tile padded to whole chunks
    uint32_t* bins_tmp = nullptr;   // scratch of the depth order of long tile lists (same layout)
    bool scal_fresh = false;        // scal just allocated (undefined contents)
    bool chained = false;           // the frame's kernels follow each other on one stream (launch_chained)
    uint64_t bin_limit = ~0ull;     // bins that there is room for: with more (scal[8]) the later passes do nothing
    uint64_t bins_seen = 0;         // bins of the last frame
    int64_t bin_cap = 0;
    uint32_t* masks = nullptr;      // per chunk of a tile list: 256 per-pixel coverage masks
    uint32_t* zsuf = nullptr;       // per chunk: a lower bound of the depths of its tile's triangles from it on
    int64_t zsuf_cap = 0;
    int64_t mask_cap = 0;
    // pixels (tile-major)
    uint32_t* cnt = nullptr;        // [P]
    int64_t p_cap = 0;
    uint64_t* part = nullptr;       // scan partials
    uint32_t* part_max = nullptr;
    int64_t part_cap = 0;
    uint32_t* zsil = nullptr;       // [P] depth of the nearest boundary fragment (silhouettes), kNoDepth if none
    uint32_t* redo = nullptr;       // [P] queue of the pixels that met their fragments out of order
    // fragments: the drawing pass stores none; what a frame's lists would take (24 bytes a fragment) is
    // accounted against the memory budget and the chosen capacities
    int64_t frag_cap = 0;
    bool frag_sized = false;
    uint64_t* scal = nullptr;       // kScalAll device scalars (slots: see kScal)
    uint64_t* h_scal = nullptr;     // pinned mirror
};

// The pixels of the drawn rectangle that go to the output image: [x0, x0 + w) x
// [y0, y0 + h), written at out[(y - y0) w + (x - x0)] (the rest is an apron whose
// depths the silhouettes read).
struct OutWin {
    int x0, y0, w, h;
};

// ---- batched launches: the tiles of up to kBatchLaunchMax frames in one grid ------------
// Each block finds its frame from the frames' first tile (tile_begin, in the
// kernel's parameters) and takes that frame's tile in its tile order.
constexpr int kBatchLaunchMax = 64;
struct CountItem {
    const uint64_t* tile_off;
    const uint32_t* tile_chunks;
    const uint32_t* bins;
    const FaceFrame* fframe;
    const uint32_t* order;
    uint32_t* cnt;
    uint32_t* masks;
    uint32_t* tile_frag;
    unsigned long long* scal;
    uint64_t* h_scal;     // pinned host copy of scal[0..2] and [5], nullptr: not wanted
    uint64_t bin_limit;   // see FrameBufs
    int tiles_x, W, H, n_tiles;
};
struct CountBatch {
    CountItem it[kBatchLaunchMax];
    uint32_t tile_begin[kBatchLaunchMax + 1];
    int n;
};
// A frame's kernels can be launched while the one before still runs
// (programmatic dependent launch): each begins with chain_begin, which waits for
// the whole of the kernel before and lets the next one be launched, so that a
// launch's latency hides behind the kernel before it (4^3 at 256x256, nine
// kernels: 65 -> 55 us a frame; 64^3 at 1920x1080: 1.19 -> 1.16 ms). All of a
// kernel's blocks are running by the time the next one's appear, in what they
// leave free: where that would crowd the next kernel's few, long blocks onto some
// of the SMs, the kernel only waits (chain_wait), and the next is launched as its
// last blocks end (the drawing pass after the count: 96^3 at 320x180 1.33 ms, with
// the early launch 1.70, without either 1.40).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_begin()
{
    chain_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Launch of a kernel that begins with either; chained: after another of the frame's, on the same stream.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s, bool chained,
                           A&&... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// What the drawing pass needs of a frame.
struct DrawItem {
    const uint64_t* tile_off;
    const uint32_t* tile_chunks;   // chunks of the tile's list that are drawn
    const uint32_t* bins;
    const uint32_t* masks;
    const uint32_t* zsuf;
    const FaceFrame* fframe;
    const FaceStatic* fstat;
    const FaceExtra* fextra;   // nullptr: not kept
    const uint32_t* order;
    const uint32_t* cnt;
    uint32_t* zsil;   // nullptr: no silhouettes
    float4* out;
    uint32_t* redo;   // queue of the pixels that met their fragments out of order
    unsigned long long* redo_cursor;
    const unsigned long long* scal;
    unsigned long long* err;
    uint64_t limit;       // most fragments the frame may have (memory budget)
    uint64_t bin_limit;   // see FrameBufs
    bool chained;         // see FrameBufs
    ShadeParams sp;
    OutWin win;
    int tiles_x, W, H;
};
struct DrawBatch {
    DrawItem it[kBatchLaunchMax];
    uint32_t tile_begin[kBatchLaunchMax + 1];
    int n;
};
// The frame of block b in a batched launch: the last with begin[i] <= b.
__device__ __forceinline__ int batch_item(const uint32_t* begin, int n, uint32_t b)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (begin[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
static_assert(sizeof(DrawBatch) < 30000 && sizeof(CountBatch) < 30000,
              "a batch's parameters fit a kernel's parameter space");

// cudaMalloc of the library (api.cu; HEXFC_OPT_DEBUG_FAIL_ALLOC); *p is null if it fails.
cudaError_t device_alloc(void** p, size_t bytes);

// ---- launches (each returns cudaGetLastError()) -----------------------------------------
cudaError_t launch_cell_quality(const DevMesh& m, int metric, float* out, cudaStream_t s);
// Vertex and edge importance (max over cells) and the faces' static records;
// positions: also the corners' world positions (once, at the upload).
// From m.cell_imp; chained: see launch_chained.
cudaError_t launch_importance(const DevMesh& m, bool positions, bool chained, cudaStream_t s);

cudaError_t launch_vertex_setup(const DevMesh& m, const CamParams& cam, FrameBufs& fb, int64_t n_tiles, cudaStream_t s);
cudaError_t launch_face_setup(const DevMesh& m, const CamParams& cam, const ShadeParams& sp, FrameBufs& fb,
                              int tiles_x, int tiles_y, int reverse, cudaStream_t s);
// Tile offsets (whole chunks) and their total into scal[8]; true in *ordered if the tile order is done too.
cudaError_t launch_tile_scan(FrameBufs& fb, int64_t n_tiles, bool* ordered, cudaStream_t s);
cudaError_t launch_bin_fill(const DevMesh& m, FrameBufs& fb, int tiles_x, int W, int H, cudaStream_t s);
// Constants of the capacity network's features (CapFeatures::X == nullptr: not wanted).
struct CapFeatures {
    const uint32_t* prev;   // the previous frame's tile counts, nullptr: none
    float* X;
    float lens_x, lens_y, inv_diag, motion;
    int tiles_x;
};
// Kernel attributes (dynamic shared memory limits), once per device context.
cudaError_t prepare_raster_kernels();
cudaError_t prepare_draw_kernels();

cudaError_t launch_bin_sort(FrameBufs& fb, int64_t n_tiles, int64_t n_bins, int buckets, const CapFeatures& cf,
                            cudaStream_t s);
cudaError_t launch_tile_order(FrameBufs& fb, int n_tiles, cudaStream_t s);
CountItem count_item(const FrameBufs& fb, int tiles_x, int tiles_y, int W, int H);
// Blocks a tile (the cluster size) of a frame's count.
unsigned count_slices(int64_t n_tiles, int64_t n_bins);
cudaError_t launch_count(FrameBufs& fb, int tiles_x, int tiles_y, int W, int H, int64_t n_bins, cudaStream_t s,
                         bool to_host = true);
// The count and the drawing pass of several frames, each one launch.
cudaError_t launch_count_batch(const CountBatch& b, cudaStream_t s);
cudaError_t launch_draw_batch(const DrawBatch& b, bool sil, int window, cudaStream_t s);
// The drawing pass of a frame, and its second pass (pixels out of order).
// n_bins: the frame's bins, about (they pick the form of the pass)
cudaError_t launch_draw(const DrawItem& a, int64_t n_tiles, uint64_t n_bins, int window, cudaStream_t s);
cudaError_t launch_draw_tail(const DrawItem& a, cudaStream_t s);
// Tile capacities from the previous frame's exact counts, or `uniform` (> 0) per tile.
cudaError_t launch_capacity_from_previous(FrameBufs& fb, int64_t n_tiles, float margin, uint32_t pad,
                                          uint32_t uniform, cudaStream_t s);
// The frame's exact tile counts against the chosen capacities.
cudaError_t launch_capacity_check(FrameBufs& fb, int64_t n_tiles, cudaStream_t s);
cudaError_t launch_cap_forward(const CapNet& net, FrameBufs& fb, int64_t n_tiles, float margin, uint32_t pad,
                               cudaStream_t s);
cudaError_t prepare_capacity_kernels();
int64_t cap_partials();   // floats of CapNet::part
// Loss and gradient into net.grad, and (lr > 0) an Adam step.
// chained: after another step on the same stream
cudaError_t launch_cap_grad(CapNet& net, const float* X, const uint32_t* counts, int64_t n, float lr, bool chained,
                            cudaStream_t s);
cudaError_t launch_cap_to_half(CapNet& net, cudaStream_t s);
// White silhouettes over the output (Section "Blending Focus and Context"):
// from the boundary surface's depths zsil of the drawn rectangle, which sits
// at (fx0, fy0) of a frame_w x frame_h frame.
cudaError_t launch_silhouette(const DrawItem& a, int fx0, int fy0, int frame_w, int frame_h, float alpha, float threshold,
                              cudaStream_t s);
// What a frame keeps of its faces' corners: their vertices, and the vertices as it projected them.
struct DrawnCorners {
    const int4* fverts;
    const int4* vproj;
};
// The sorted lists of n pixels of a frame drawn as `a` with corners dc (or their lengths, if d_counts).
cudaError_t launch_debug_gather(const DrawItem& a, const DrawnCorners& dc, const int32_t* d_px, const int32_t* d_py, int64_t n,
                                const uint64_t* d_dst_off, uint64_t* d_keys, float4* d_rgba, uint32_t* d_counts,
                                cudaStream_t s);

// scans
cudaError_t scan_u32_to_u64(const uint32_t* in, uint64_t* out, int64_t n, uint64_t* part,
                            uint32_t* part_max, uint64_t* total_and_max, uint32_t long_threshold,
                            cudaStream_t s, uint32_t round_to = 0, const uint32_t* in2 = nullptr, const uint32_t* in3 = nullptr);
int64_t scan_partials_needed(int64_t n);

}  // namespace hexfc
