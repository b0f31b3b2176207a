// Per-cell quality (Jacobian of the cube-to-cell map) and importance max-reduce.
//
// Quality: the paper names the Jacobian-based deformation measures (Section
// "Introduction"; Section "Results and Analysis": per-cell scaled Jacobian
// ratio) without printing a formula. Evaluated here: the Jacobian at the 8
// corners (three edge vectors to the corner's neighbours) and at the cell
// centre (the three principal axes, sums of the four parallel edges):
//   scaled Jacobian = min det of the unit-length vectors,
//   Jacobian ratio  = min det / max det (centre axes scaled by 1/4),
//   importance      = clamp(1 - scaled Jacobian, 0, 1).
// Importance: every vertex and every edge takes the maximum importance of the
// cells sharing it (Section "Method Overview").
#include "hexfc_internal.cuh"

namespace hexfc {
namespace {

__device__ __forceinline__ float det3f(float3 a, float3 b, float3 c)
{
    return a.x * (b.y * c.z - b.z * c.y) + a.y * (b.z * c.x - b.x * c.z) + a.z * (b.x * c.y - b.y * c.x);
}
__device__ __forceinline__ float3 sub3(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 add3(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float len3(float3 a) { return sqrtf(a.x * a.x + a.y * a.y + a.z * a.z); }

// One thread a cell, the metric at compile time (the ratio needs no lengths), all
// indices too (the corners stay in registers). The 12 edges' lengths are taken
// once: the two corners of an edge see it with the same length, bit for bit.
// 262,144 cells: 11.0 -> 7.1 us (scaled Jacobian), 11.0 -> 4.3 us (ratio); with caches
// cold 17 -> 15 and 17 -> 11. Bound by the gathers' latency, then by the 9 divisions
// and 15 square roots a cell; cells, vertices and results are 13 MB, 2 us at the copy
// rate. (64 registers, 8 blocks an SM: 8.8 us.)
template <int kMetric>
__global__ void __launch_bounds__(128) k_cell_quality(const float* __restrict__ verts, const int32_t* __restrict__ cells,
                                                      int64_t n_cells, float* __restrict__ out)
{
    // neighbours of corner k of a VTK hexahedron, right-handed, and the edges to them
    constexpr int kNb[8][3] = {{1, 3, 4}, {2, 0, 5}, {3, 1, 6}, {0, 2, 7}, {7, 5, 0}, {4, 6, 1}, {5, 7, 2}, {6, 4, 3}};
    constexpr int kEdge[8][3] = {{0, 3, 8}, {1, 0, 9}, {2, 1, 10}, {3, 2, 11}, {7, 4, 8}, {4, 5, 9}, {5, 6, 10}, {6, 7, 11}};
    constexpr int kEnds[12][2] = {{0, 1}, {1, 2}, {2, 3}, {3, 0}, {4, 5}, {5, 6}, {6, 7}, {7, 4}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};
    constexpr bool kRatio = kMetric == HEXFC_METRIC_JACOBIAN_RATIO;
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_cells) return;
    const int4* cc = reinterpret_cast<const int4*>(cells + 8 * c);
    int4 a = __ldg(cc), b = __ldg(cc + 1);
    int id[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    float3 p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        p[k] = make_float3(__ldg(verts + 3 * (int64_t)id[k]), __ldg(verts + 3 * (int64_t)id[k] + 1),
                           __ldg(verts + 3 * (int64_t)id[k] + 2));
    float len[12];
    if (!kRatio) {
#pragma unroll
        for (int e = 0; e < 12; ++e) len[e] = len3(sub3(p[kEnds[e][1]], p[kEnds[e][0]]));
    }
    float sj = 3.0e38f, dmin = 3.0e38f, dmax = -3.0e38f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float3 e0 = sub3(p[kNb[k][0]], p[k]);
        float3 e1 = sub3(p[kNb[k][1]], p[k]);
        float3 e2 = sub3(p[kNb[k][2]], p[k]);
        float d = det3f(e0, e1, e2);
        if (kRatio) {
            dmin = fminf(dmin, d);
            dmax = fmaxf(dmax, d);
        } else {
            float l = len[kEdge[k][0]] * len[kEdge[k][1]] * len[kEdge[k][2]];
            float nd = l > 0.f ? d / l : 0.f;
            sj = fminf(sj, nd);
        }
    }
    {
        float3 X0 = add3(add3(sub3(p[1], p[0]), sub3(p[2], p[3])), add3(sub3(p[5], p[4]), sub3(p[6], p[7])));
        float3 X1 = add3(add3(sub3(p[3], p[0]), sub3(p[2], p[1])), add3(sub3(p[7], p[4]), sub3(p[6], p[5])));
        float3 X2 = add3(add3(sub3(p[4], p[0]), sub3(p[5], p[1])), add3(sub3(p[6], p[2]), sub3(p[7], p[3])));
        float d = det3f(X0, X1, X2);
        if (kRatio) {
            float dc = d * (1.0f / 64.0f);
            dmin = fminf(dmin, dc);
            dmax = fmaxf(dmax, dc);
        } else {
            float l = len3(X0) * len3(X1) * len3(X2);
            float nd = l > 0.f ? d / l : 0.f;
            sj = fminf(sj, nd);
        }
    }
    float v;
    if (kMetric == HEXFC_METRIC_SCALED_JACOBIAN) v = sj;
    else if (kRatio) v = dmax > 0.f ? dmin / dmax : -1.f;
    else v = fminf(fmaxf(1.f - sj, 0.f), 1.f);
    out[c] = v;
}

// Importance of every vertex and edge, the largest of its cells': keys cleared,
// scattered with an atomic each (bound by them: 20 a cell), and written where the
// frames read them. Three launches, each behind the one before, instead of
// four (64^3 cells: 36 -> 29 us, caches cold 48 -> 40).

// The keys of vertices, then edges.
__global__ void __launch_bounds__(256) k_init_keys(int32_t* __restrict__ a, int64_t na, int32_t* __restrict__ b, int64_t nb,
                                                   int32_t v)
{
    chain_begin();
    int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < na) a[i] = v;
    else if (i - na < nb) b[i - na] = v;
}

// Thread per cell.
__global__ void __launch_bounds__(256) k_importance_scatter(const int32_t* __restrict__ cells,
                                                            const int32_t* __restrict__ cell_edges,
                                                            const float* __restrict__ cell_imp,
                                                            int64_t n_cells, int32_t* __restrict__ vkey,
                                                            int32_t* __restrict__ ekey)
{
    chain_begin();
    const int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (c >= n_cells) return;
    const float v = cell_imp[c];
    const int4* p = reinterpret_cast<const int4*>(cells) + 2 * c;
    const int4* q = reinterpret_cast<const int4*>(cell_edges) + 3 * c;
    const int4 a[2] = {p[0], p[1]}, b[3] = {q[0], q[1], q[2]};
    const int32_t k = importance_key(v);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        atomicMax(vkey + a[j].x, k);
        atomicMax(vkey + a[j].y, k);
        atomicMax(vkey + a[j].z, k);
        atomicMax(vkey + a[j].w, k);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        atomicMax(ekey + b[j].x, k);
        atomicMax(ekey + b[j].y, k);
        atomicMax(ekey + b[j].z, k);
        atomicMax(ekey + b[j].w, k);
    }
}

// Thread per face: the importances of its corners in its static record, and with
// `positions` (a new record) their world positions; then a thread per edge.
__global__ void __launch_bounds__(256) k_face_static(const int4* __restrict__ fverts, const int32_t* __restrict__ vkey,
                                                     const float* __restrict__ verts, int64_t n_faces, bool positions,
                                                     FaceStatic* __restrict__ fstat, const int32_t* __restrict__ ekey,
                                                     int64_t n_edges, float* __restrict__ eattr)
{
    chain_begin();
    const int64_t f = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (f >= n_faces) {
        const int64_t e = f - n_faces;
        if (e < n_edges) eattr[e] = importance_of(ekey[e]);
        return;
    }
    const int4 c = fverts[f];
    const int id[4] = {c.x, c.y, c.z, c.w};
    FaceStatic& r = fstat[f];
    r.imp = make_float4(importance_of(vkey[id[0]]), importance_of(vkey[id[1]]), importance_of(vkey[id[2]]),
                        importance_of(vkey[id[3]]));
    if (!positions) return;
    float x[4], y[4], z[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[k] = verts[3 * (int64_t)id[k]];
        y[k] = verts[3 * (int64_t)id[k] + 1];
        z[k] = verts[3 * (int64_t)id[k] + 2];
    }
    r.px = make_float4(x[0], x[1], x[2], x[3]);
    r.py = make_float4(y[0], y[1], y[2], y[3]);
    r.pz = make_float4(z[0], z[1], z[2], z[3]);
}

inline unsigned grid_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

cudaError_t launch_cell_quality(const DevMesh& m, int metric, float* out, cudaStream_t s)
{
    if (m.n_cells == 0) return cudaSuccess;
    auto go = [&](auto kernel) { kernel<<<grid_for(m.n_cells, 128), 128, 0, s>>>(m.verts, m.cells, m.n_cells, out); };
    if (metric == HEXFC_METRIC_SCALED_JACOBIAN) go(k_cell_quality<HEXFC_METRIC_SCALED_JACOBIAN>);
    else if (metric == HEXFC_METRIC_JACOBIAN_RATIO) go(k_cell_quality<HEXFC_METRIC_JACOBIAN_RATIO>);
    else go(k_cell_quality<HEXFC_METRIC_IMPORTANCE>);
    return cudaGetLastError();
}

cudaError_t launch_importance(const DevMesh& m, bool positions, bool chained, cudaStream_t s)
{
    cudaError_t e = launch_chained(k_init_keys, grid_for(m.n_verts + m.n_edges, 256), 256, 0, s, false, m.vkey, m.n_verts, m.ekey,
                                   m.n_edges, INT32_MIN);
    if (e == cudaSuccess)
        e = launch_chained(k_importance_scatter, grid_for(m.n_cells, 256), 256, 0, s, chained, m.cells, m.cell_edges, m.cell_imp,
                           m.n_cells, m.vkey, m.ekey);
    if (e == cudaSuccess)
        e = launch_chained(k_face_static, grid_for(m.n_faces + m.n_edges, 256), 256, 0, s, chained, m.fverts, m.vkey, m.verts,
                           m.n_faces, positions, m.fstat, m.ekey, m.n_edges, m.eattr);
    return e;
}

}  // namespace hexfc
