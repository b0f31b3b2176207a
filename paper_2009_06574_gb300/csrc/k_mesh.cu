// Unique faces and edges of a hexahedral mesh on the device: the tables of
// mesh_host.cpp (which defines them), for meshes whose vertices have ordinary
// valences. A table's ids are the ranks of sorted vertex tuples, so the records of
// all cells go into one bucket per least vertex (counted, scanned, placed), each
// bucket is sorted and its distinct records numbered by a warp, and a scan of the
// buckets' numbers gives the ids.
//
// Sorting 83,000 faces and 166,000 edges (24^3 cells) on the host took 14 ms of the
// 16 ms from a new context to its first frame; the upload with the kernels here
// takes 0.7 ms. Bound by the launches (18) and allocations around them.
#include "hexfc_internal.cuh"
#include "mesh_device.h"

namespace hexfc {
namespace {

// cyclic corners of the six faces of a VTK hexahedron, the cell edges between them, the ends of the twelve edges
__constant__ uint8_t c_face[6][4] = {{0, 1, 2, 3}, {4, 5, 6, 7}, {0, 1, 5, 4}, {1, 2, 6, 5}, {2, 3, 7, 6}, {3, 0, 4, 7}};
__constant__ uint8_t c_side[6][4] = {{0, 1, 2, 3}, {4, 5, 6, 7}, {0, 9, 4, 8}, {1, 10, 5, 9}, {2, 11, 6, 10}, {3, 8, 7, 11}};
__constant__ uint8_t c_edge[12][2] = {{0, 1}, {1, 2}, {2, 3}, {3, 0}, {4, 5}, {5, 6},
                                      {6, 7}, {7, 4}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};

constexpr uint32_t kFirst = 1u << 31;   // the first of equal records
constexpr uint32_t kMostInBucket = 1024;   // (ranks are counted: the square of it, 32 at a time)
constexpr unsigned kFull = 0xffffffffu;

inline unsigned grid_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

__device__ __forceinline__ void order2(int32_t& a, int32_t& b)
{
    const int32_t t = min(a, b);
    b = max(a, b);
    a = t;
}
// The vertices of face i % 6 of cell i / 6 in cyclic order, and in ascending order.
__device__ __forceinline__ int4 face_corners(const int32_t* __restrict__ cells, uint32_t i)
{
    const int32_t* cv = cells + 8 * (int64_t)(i / 6);
    const uint8_t* f = c_face[i % 6];
    return make_int4(cv[f[0]], cv[f[1]], cv[f[2]], cv[f[3]]);
}
__device__ __forceinline__ int4 ascending(int4 q)
{
    order2(q.x, q.y);
    order2(q.z, q.w);
    order2(q.x, q.z);
    order2(q.y, q.w);
    order2(q.y, q.z);
    return q;
}
__device__ __forceinline__ int2 edge_ends(const int32_t* __restrict__ cells, uint32_t i)
{
    const int32_t* cv = cells + 8 * (int64_t)(i / 12);
    const uint8_t* e = c_edge[i % 12];
    int2 r = make_int2(cv[e[0]], cv[e[1]]);
    order2(r.x, r.y);
    return r;
}

// Thread per record (6 faces, then 12 edges a cell): how many each vertex is the least of.
__global__ void __launch_bounds__(256) k_mesh_count(const int32_t* __restrict__ cells, int64_t n_cells,
                                                    uint32_t* __restrict__ fcnt, uint32_t* __restrict__ ecnt)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < 6 * n_cells) {
        const int4 q = face_corners(cells, (uint32_t)i);
        atomicAdd(&fcnt[min(min(q.x, q.y), min(q.z, q.w))], 1u);
    } else if (i < 18 * n_cells) {
        atomicAdd(&ecnt[edge_ends(cells, (uint32_t)(i - 6 * n_cells)).x], 1u);
    }
}

// The records into their buckets, in any order; the counts run down to 0.
__global__ void __launch_bounds__(256) k_mesh_place(const int32_t* __restrict__ cells, int64_t n_cells,
                                                    uint32_t* __restrict__ fcnt, const uint64_t* __restrict__ foff,
                                                    uint4* __restrict__ frec, uint32_t* __restrict__ ecnt,
                                                    const uint64_t* __restrict__ eoff, uint2* __restrict__ erec)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < 6 * n_cells) {
        const int4 s = ascending(face_corners(cells, (uint32_t)i));
        frec[foff[s.x] + atomicSub(&fcnt[s.x], 1u) - 1u] = make_uint4((uint32_t)s.y, (uint32_t)s.z, (uint32_t)s.w, (uint32_t)i);
    } else if (i < 18 * n_cells) {
        const uint32_t k = (uint32_t)(i - 6 * n_cells);
        const int2 e = edge_ends(cells, k);
        erec[eoff[e.x] + atomicSub(&ecnt[e.x], 1u) - 1u] = make_uint2((uint32_t)e.y, k);
    }
}

__device__ __forceinline__ bool same(const uint4& a, const uint4& b) { return a.x == b.x && a.y == b.y && a.z == b.z; }
__device__ __forceinline__ bool less(const uint4& a, const uint4& b)
{
    return a.x != b.x ? a.x < b.x : a.y != b.y ? a.y < b.y : a.z != b.z ? a.z < b.z : a.w < b.w;
}
__device__ __forceinline__ bool same(const uint2& a, const uint2& b) { return a.x == b.x; }
__device__ __forceinline__ bool less(const uint2& a, const uint2& b) { return a.x != b.x ? a.x < b.x : a.y < b.y; }

// A warp's bucket [beg, beg + n): sorted from rec to out, and per record the
// number of distinct ones before it (kFirst: it is the first of its kind).
template <class R>
__device__ __forceinline__ void sort_bucket(const R* __restrict__ rec, R* out, uint32_t* __restrict__ number, uint64_t beg,
                                            uint32_t n, uint32_t* __restrict__ distinct, int lane)
{
    for (uint32_t i = lane; i < n; i += 32) {
        const R r = rec[beg + i];
        uint32_t rank = 0;
        for (uint32_t j = 0; j < n; ++j) rank += less(rec[beg + j], r) ? 1u : 0u;
        out[beg + rank] = r;
    }
    __syncwarp();
    uint32_t before = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += 32) {
        const uint32_t i = i0 + lane;
        const bool first = i < n && (i == 0 || !same(out[beg + i], out[beg + i - 1]));
        const unsigned b = __ballot_sync(kFull, first);
        if (i < n) number[beg + i] = (before + __popc(b & (kFull >> (31 - lane))) - 1u) | (first ? kFirst : 0u);
        before += __popc(b);
    }
    if (lane == 0) *distinct = before;
}

// Warp per vertex: its bucket of faces, or of edges (the second half of the grid).
__global__ void __launch_bounds__(256) k_mesh_sort(int64_t n_verts, int64_t n_cells, const uint64_t* __restrict__ foff,
                                                   const uint4* __restrict__ frec, uint4* __restrict__ fsort,
                                                   uint32_t* __restrict__ fnum, uint32_t* __restrict__ fcnt,
                                                   const uint64_t* __restrict__ eoff, const uint2* __restrict__ erec,
                                                   uint2* __restrict__ esort, uint32_t* __restrict__ enum_,
                                                   uint32_t* __restrict__ ecnt, uint64_t* __restrict__ flags)
{
    const int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= 2 * n_verts) return;
    const bool edges = w >= n_verts;
    const int64_t v = edges ? w - n_verts : w;
    const uint64_t* off = edges ? eoff : foff;
    const uint64_t beg = off[v], end = v + 1 < n_verts ? off[v + 1] : (uint64_t)(edges ? 12 : 6) * (uint64_t)n_cells;
    const uint32_t n = (uint32_t)(end - beg);
    if (n > kMostInBucket) {
        if (lane == 0) *flags = 1;
        return;
    }
    if (edges) sort_bucket(erec, esort, enum_, beg, n, ecnt + v, lane);
    else sort_bucket(frec, fsort, fnum, beg, n, fcnt + v, lane);
}

// Thread per sorted edge record: the cell edge's id; the first of a kind takes the
// largest of its cells' levels.
__global__ void __launch_bounds__(256) k_mesh_edges(const int32_t* __restrict__ cells, int64_t n, const uint2* __restrict__ esort,
                                                    const uint32_t* __restrict__ num, const uint64_t* __restrict__ base,
                                                    const uint8_t* __restrict__ level, int32_t* __restrict__ cell_edges,
                                                    uint8_t* __restrict__ elevel)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = esort[i].y, u = num[i];
    const uint64_t id = base[edge_ends(cells, k).x] + (u & ~kFirst);
    cell_edges[k] = (int32_t)id;
    if (u & kFirst) {
        uint8_t most = level ? level[k] : (uint8_t)0;
        for (int64_t j = i + 1; level && j < n && !(num[j] & kFirst); ++j) most = max(most, level[esort[j].y]);
        elevel[id] = most;
    }
}

// The quad of face record i: its least vertex first, then the smaller of its
// neighbours; side k (corner k to k + 1) is cell edge e[k].
__device__ __forceinline__ void quad_of(const int32_t* __restrict__ cells, uint32_t i, int32_t (&c)[4], int (&e)[4])
{
    const int4 v = face_corners(cells, i);
    const int32_t q[4] = {v.x, v.y, v.z, v.w};
    int m = 0;
    int32_t least = q[0];
#pragma unroll
    for (int k = 1; k < 4; ++k)
        if (q[k] < least) {
            least = q[k];
            m = k;
        }
    auto at = [&](int k) { k &= 3; return k == 0 ? q[0] : k == 1 ? q[1] : k == 2 ? q[2] : q[3]; };
    const bool fwd = at(m + 1) < at(m + 3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        c[k] = fwd ? at(m + k) : at(m - k + 4);
        e[k] = c_side[i % 6][(fwd ? m + k : m - k + 3) & 3];
    }
}

// Thread per sorted face record: the first of a kind writes the face. Equal
// records with other quads (repeated or crossed corners) are left to the host.
__global__ void __launch_bounds__(256) k_mesh_faces(const int32_t* __restrict__ cells, int64_t n, const uint4* __restrict__ fsort,
                                                    const uint32_t* __restrict__ num, const uint64_t* __restrict__ base,
                                                    const int32_t* __restrict__ cell_edges, int4* __restrict__ fverts,
                                                    int4* __restrict__ fedges, uint8_t* __restrict__ fbound,
                                                    uint64_t* __restrict__ flags)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const uint32_t r = fsort[i].w, u = num[i];
    int32_t c[4];
    int e[4];
    quad_of(cells, r, c, e);
    if (u & kFirst) {
        const uint64_t id = base[c[0]] + (u & ~kFirst);
        const int32_t* ce = cell_edges + 12 * (int64_t)(r / 6);
        fverts[id] = make_int4(c[0], c[1], c[2], c[3]);
        fedges[id] = make_int4(ce[e[0]], ce[e[1]], ce[e[2]], ce[e[3]]);
        fbound[id] = i + 1 == n || (num[i + 1] & kFirst) ? 1 : 0;
    } else {
        int32_t p[4];
        quad_of(cells, fsort[i - 1].w, p, e);
        if (c[0] != p[0] || c[1] != p[1] || c[2] != p[2] || c[3] != p[3]) *flags = 1;
    }
}

}  // namespace

MeshScratch::~MeshScratch() { cudaFree(block); }

cudaError_t MeshScratch::number(const int32_t* cells, int64_t n_cells, int64_t n_verts, uint64_t* n_faces, uint64_t* n_edges,
                                bool* host)
{
    const size_t V = (size_t)n_verts, F = 6 * (size_t)n_cells, E = 12 * (size_t)n_cells;
    const int64_t parts = scan_partials_needed(n_verts) + 1;
    size_t used = 0;
    auto room = [&](size_t bytes) {
        const size_t at = used;
        used = (used + bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_scal = room(16 * sizeof(uint64_t)), o_fcnt = room(V * 4), o_ecnt = room(V * 4), zero = used;
    const size_t o_foff = room((V + 1) * 8), o_eoff = room((V + 1) * 8), o_frec = room(F * 16), o_fsort = room(F * 16),
                 o_erec = room(E * 8), o_esort = room(E * 8), o_fnum = room(F * 4), o_enum = room(E * 4),
                 o_part = room(2 * (size_t)parts * 8), o_max = room(2 * (size_t)parts * 4);
    cudaError_t e = device_alloc(&block, used);
    if (e != cudaSuccess) return e;
    auto at = [&](size_t o) { return static_cast<unsigned char*>(block) + o; };
    scal = (uint64_t*)at(o_scal);
    uint32_t *fcnt = (uint32_t*)at(o_fcnt), *ecnt = (uint32_t*)at(o_ecnt);
    foff = (uint64_t*)at(o_foff);
    eoff = (uint64_t*)at(o_eoff);
    fsort = (uint4*)at(o_fsort);
    esort = (uint2*)at(o_esort);
    fnum = (uint32_t*)at(o_fnum);
    enum_ = (uint32_t*)at(o_enum);
    uint64_t* part = (uint64_t*)at(o_part);
    uint32_t* most = (uint32_t*)at(o_max);
    if ((e = cudaMemsetAsync(block, 0, zero, 0)) != cudaSuccess) return e;
    const unsigned grid = grid_for(18 * n_cells, 256);
    k_mesh_count<<<grid, 256>>>(cells, n_cells, fcnt, ecnt);
    if ((e = scan_u32_to_u64(fcnt, foff, n_verts, part, most, scal, 0xFFFFFFFFu, 0)) != cudaSuccess) return e;
    if ((e = scan_u32_to_u64(ecnt, eoff, n_verts, part, most, scal + 3, 0xFFFFFFFFu, 0)) != cudaSuccess) return e;
    k_mesh_place<<<grid, 256>>>(cells, n_cells, fcnt, foff, (uint4*)at(o_frec), ecnt, eoff, (uint2*)at(o_erec));
    k_mesh_sort<<<grid_for(2 * n_verts, 8), 256>>>(n_verts, n_cells, foff, (const uint4*)at(o_frec), fsort, fnum, fcnt, eoff,
                                                   (const uint2*)at(o_erec), esort, enum_, ecnt, scal + 12);
    // (the offsets are not needed any more: the ids of the buckets' first records take their place)
    if ((e = scan_u32_to_u64(fcnt, foff, n_verts, part, most, scal + 6, 0xFFFFFFFFu, 0)) != cudaSuccess) return e;
    if ((e = scan_u32_to_u64(ecnt, eoff, n_verts, part, most, scal + 9, 0xFFFFFFFFu, 0)) != cudaSuccess) return e;
    uint64_t h[13];
    if ((e = cudaMemcpy(h, scal, sizeof(h), cudaMemcpyDeviceToHost)) != cudaSuccess) return e;
    *n_faces = h[6];
    *n_edges = h[9];
    *host = h[12] != 0;
    return cudaGetLastError();
}

cudaError_t MeshScratch::write(const int32_t* cells, int64_t n_cells, const uint8_t* level, int32_t* cell_edges, uint8_t* elevel,
                               int4* fverts, int4* fedges, uint8_t* fbound, bool* host)
{
    k_mesh_edges<<<grid_for(12 * n_cells, 256), 256>>>(cells, 12 * n_cells, esort, enum_, eoff, level, cell_edges, elevel);
    k_mesh_faces<<<grid_for(6 * n_cells, 256), 256>>>(cells, 6 * n_cells, fsort, fnum, foff, cell_edges, fverts, fedges, fbound,
                                                      scal + 12);
    uint64_t flags = 0;
    const cudaError_t e = cudaMemcpy(&flags, scal + 12, sizeof(flags), cudaMemcpyDeviceToHost);
    *host = flags != 0;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace hexfc
