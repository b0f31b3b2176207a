// Tile-capacity network: per raster tile, a 4 -> 64 -> 64 -> 1 ReLU network
// predicts y ~ log(1 + fragments of the tile) from four features, so that
// fragment storage can be divided among the tiles before a frame is counted.
// Weights are used in FP16 (staged in shared memory), sums in FP32; training
// keeps an FP32 master copy and Adam moments. No counterpart in the paper.
//
// The features (left by the depth order of the tile lists): log1p(previous
// frame's count) / 12, the depth range of its triangles, the distance from the
// tile to the lens on screen / screen diagonal, the camera's motion since the
// previous frame.
//
//   k_cap_forward   per tile: y and the capacity expm1(y) (1 + margin) + pad
//   k_cap_backward  mean-squared loss on log1p(exact count) and the gradient, a
//                   share per block
//   k_cap_sum       the shares summed; an Adam step on the master copy, FP16 copy
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "hexfc_internal.cuh"

namespace hexfc {
namespace {

constexpr int kIn = kCapIn, kHid = kCapHid;
constexpr int oW1 = 0, oB1 = oW1 + kHid * kIn, oW2 = oB1 + kHid, oB2 = oW2 + kHid * kHid, oW3 = oB2 + kHid,
              oB3 = oW3 + kHid;
static_assert(oB3 + 1 == kCapParams, "parameter layout");

inline unsigned grid_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// ---- layers on a group of kGroup tiles, 256 threads
//
// A thread per tile left 120 of 152 SMs idle at 8160 tiles and walked 8,500
// multiply-adds alone: 75 us forward and backward, and 32 us to sum the gradient
// from 8 MB of stored layer values. Here a block takes 32 tiles; the three 64 x 64
// products (layer 2, its gradient, the error back through it) are register tiles
// over operands in shared memory, the gradient's sums stay in registers over the
// block's groups, and what leaves the block is its share of the gradient, summed
// in a fixed order (so a training step gives the same bits every time). Then the
// weights' loads were a third of a step and the transposed stores went into one
// bank: all loads at once, rows apart. Backward 75 + 32 us -> 15 + 4.4; 8 Adam steps
// at 1920x1080, weights set and read: 0.93 -> 0.30 -> 0.19 ms. Bound by shared-memory
// reads (9 of the 15 us) and the phases' barriers.
constexpr int kGroup = 32;
constexpr int kCapThreads = 256;
constexpr int kCapBlocks = 304;   // two blocks an SM at most; more tiles than kGroup * 304: several groups each

constexpr int kPartStride = (kCapParams + 1 + 3) / 4 * 4;   // a block's share: the gradient, the loss
static_assert(oW2 % 4 == 0, "16-byte stores");

struct NetSmem {
    float w1[kHid * kIn], b1[kHid], b2[kHid], w3[kHid];
    float w2[kHid][kHid + 16];  // [j][i] (rows apart for the stores of net_load)
    float w2t[kHid][kHid + 4];  // [i][j]
    float x[kGroup][kIn];
    float h1[kGroup][kHid];     // [t][i]
    float h1t[kHid][kGroup + 2];   // [i][t] (written along i: without the 2, all into one bank)
    float da[kGroup][kHid];     // [t][j]: errors of layer 2, then [t][i]: of layer 1
    float dat[kHid][kGroup + 2];   // [j][t]
    float red[2][16][kHid];     // sums over the groups of tiles at the end
    float dy[16][2];
    float b3;
};
// (read 16 bytes at a time, the transposed ones 8)
static_assert(offsetof(NetSmem, b2) % 16 == 0 && offsetof(NetSmem, w3) % 16 == 0 && offsetof(NetSmem, w2) % 16 == 0 &&
                  offsetof(NetSmem, w2t) % 16 == 0 && offsetof(NetSmem, h1) % 16 == 0 &&
                  offsetof(NetSmem, da) % 16 == 0 && offsetof(NetSmem, h1t) % 8 == 0 &&
                  offsetof(NetSmem, dat) % 8 == 0,
              "alignment of the vector reads");

// The weights into shared memory: all of a thread's loads in flight at once (one
// after another they were a third of a training step).
__device__ __forceinline__ void net_load(NetSmem& S, const __half* __restrict__ w16)
{
    static_assert(kCapThreads == 4 * kHid && kHid == 64 && oW2 % 8 == 0, "a quarter of a row of W2 each");
    const int tid = threadIdx.x, j = tid >> 2, c = (tid & 3) * 4;
    uint2 r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] = *reinterpret_cast<const uint2*>(w16 + oW2 + j * kHid + 16 * k + c);
    const __half w1 = w16[oW1 + tid];
    const int at = tid < kHid ? oB1 + tid : tid < 2 * kHid ? oB2 + tid - kHid : tid < 3 * kHid ? oW3 + tid - 2 * kHid : oB3;
    const __half rest = w16[at];
    S.w1[tid] = __half2float(w1);
    const float v = __half2float(rest);
    if (tid < kHid) S.b1[tid] = v;
    else if (tid < 2 * kHid) S.b2[tid - kHid] = v;
    else if (tid < 3 * kHid) S.w3[tid - 2 * kHid] = v;
    else if (tid == 3 * kHid) S.b3 = v;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&r[k].x)),
                     hi = __half22float2(*reinterpret_cast<const __half2*>(&r[k].y));
        const int i = 16 * k + c;
        *reinterpret_cast<float4*>(&S.w2[j][i]) = make_float4(lo.x, lo.y, hi.x, hi.y);
        S.w2t[i][j] = lo.x;
        S.w2t[i + 1][j] = lo.y;
        S.w2t[i + 2][j] = hi.x;
        S.w2t[i + 3][j] = hi.y;
    }
}

// Layers 1 and 2 of tiles t0 .. t0 + 31 (rows past n are zero): this thread's
// values before the second ReLU, a[u][v] of tile 2 (tid / 16) + u and hidden
// unit 4 (tid % 16) + v, and the output y[u] of its two tiles.
template <bool kTrain>
__device__ __forceinline__ void net_forward(NetSmem& S, const float* __restrict__ X, int64_t n, int64_t t0, float (&a)[2][4],
                                            float (&y)[2])
{
    const int tid = threadIdx.x, jq = tid & 15, tp = tid >> 4;
    __syncthreads();   // the last group is done with the arrays (and the weights are loaded)
    if (tid < kGroup * kIn) {
        const int64_t at = t0 * kIn + tid;
        S.x[tid / kIn][tid % kIn] = at < n * kIn ? X[at] : 0.f;
    }
    __syncthreads();
    {
        const int i = tid & 63, t8 = (tid >> 6) * 8;
        const float* w = S.w1 + i * kIn;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float* x = S.x[t8 + k];
            const float h = fmaxf(fmaf(w[3], x[3], fmaf(w[2], x[2], fmaf(w[1], x[1], fmaf(w[0], x[0], S.b1[i])))), 0.f);
            S.h1t[i][t8 + k] = h;
            if (kTrain) S.h1[t8 + k][i] = h;
        }
    }
    __syncthreads();
    const float4 b = *reinterpret_cast<const float4*>(&S.b2[4 * jq]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        a[u][0] = b.x; a[u][1] = b.y; a[u][2] = b.z; a[u][3] = b.w;
    }
#pragma unroll 8
    for (int i = 0; i < kHid; ++i) {
        const float2 h = *reinterpret_cast<const float2*>(&S.h1t[i][2 * tp]);
        const float4 w = *reinterpret_cast<const float4*>(&S.w2t[i][4 * jq]);
        a[0][0] = fmaf(w.x, h.x, a[0][0]); a[0][1] = fmaf(w.y, h.x, a[0][1]);
        a[0][2] = fmaf(w.z, h.x, a[0][2]); a[0][3] = fmaf(w.w, h.x, a[0][3]);
        a[1][0] = fmaf(w.x, h.y, a[1][0]); a[1][1] = fmaf(w.y, h.y, a[1][1]);
        a[1][2] = fmaf(w.z, h.y, a[1][2]); a[1][3] = fmaf(w.w, h.y, a[1][3]);
    }
    const float4 w3 = *reinterpret_cast<const float4*>(&S.w3[4 * jq]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        float v = fmaf(w3.x, fmaxf(a[u][0], 0.f), w3.y * fmaxf(a[u][1], 0.f)) +
                  fmaf(w3.z, fmaxf(a[u][2], 0.f), w3.w * fmaxf(a[u][3], 0.f));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        y[u] = v + S.b3;
    }
}

__global__ void __launch_bounds__(kCapThreads) k_cap_forward(const float* __restrict__ X, int64_t n,
                                                             const __half* __restrict__ w16, float margin,
                                                             uint32_t pad, uint32_t* __restrict__ cap)
{
    extern __shared__ __align__(16) unsigned char net_smem[];
    NetSmem& S = *reinterpret_cast<NetSmem*>(net_smem);
    net_load(S, w16);
    for (int64_t t0 = (int64_t)blockIdx.x * kGroup; t0 < n; t0 += (int64_t)gridDim.x * kGroup) {
        float a[2][4], y[2];
        net_forward<false>(S, X, n, t0, a, y);
        const int64_t t = t0 + 2 * (threadIdx.x >> 4);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if ((threadIdx.x & 15) == 0 && t + u < n) {
                const float c = expm1f(fminf(y[u], 20.f)) * (1.f + margin) + (float)pad;
                cap[t + u] = (uint32_t)fminf(fmaxf(c, 0.f), 4.0e9f);
            }
    }
}

// Loss (mean over the n tiles of (y - log1p(count))^2) and gradient: block b's
// shares into part[b][kPartStride].
__global__ void __launch_bounds__(kCapThreads) k_cap_backward(const float* __restrict__ X,
                                                              const uint32_t* __restrict__ counts, int64_t n,
                                                              const __half* __restrict__ w16,
                                                              float* __restrict__ part)
{
    extern __shared__ __align__(16) unsigned char net_smem[];
    NetSmem& S = *reinterpret_cast<NetSmem*>(net_smem);
    chain_begin();
    net_load(S, w16);
    const int tid = threadIdx.x, q = tid & 15, g = tid >> 4;
    float gw2[4][4] = {}, gw3[4] = {}, gb2[4] = {}, gw1 = 0.f, gb1 = 0.f, gb3 = 0.f, loss = 0.f;
    const float inv_n = 1.f / (float)n;
    for (int64_t t0 = (int64_t)blockIdx.x * kGroup; t0 < n; t0 += (int64_t)gridDim.x * kGroup) {
        float a[2][4], y[2];
        net_forward<true>(S, X, n, t0, a, y);
        const float4 w3 = *reinterpret_cast<const float4*>(&S.w3[4 * q]);
        const float w3v[4] = {w3.x, w3.y, w3.z, w3.w};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t t = t0 + 2 * g + u;
            const float e = t < n ? y[u] - log1pf((float)counts[t]) : 0.f;
            const float dy = 2.f * e * inv_n;
            if (q == 0) {
                loss = fmaf(e * inv_n, e, loss);
                gb3 += dy;
            }
            float d[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                gw3[v] = fmaf(dy, fmaxf(a[u][v], 0.f), gw3[v]);
                d[v] = a[u][v] > 0.f ? dy * w3v[v] : 0.f;
                gb2[v] += d[v];
                S.dat[4 * q + v][2 * g + u] = d[v];
            }
            *reinterpret_cast<float4*>(&S.da[2 * g + u][4 * q]) = make_float4(d[0], d[1], d[2], d[3]);
        }
        __syncthreads();
        // gradient of W2: units j = 4 g + u, i = 4 q + v
#pragma unroll 4
        for (int t = 0; t < kGroup; ++t) {
            const float4 d = *reinterpret_cast<const float4*>(&S.da[t][4 * g]);
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[t][4 * q]);
            const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) gw2[u][v] = fmaf(dv[u], hv[v], gw2[u][v]);
        }
        // errors of layer 1: tiles 2 g + u, units i = 4 q + v
        float e1[2][4] = {};
#pragma unroll 8
        for (int j = 0; j < kHid; ++j) {
            const float2 d = *reinterpret_cast<const float2*>(&S.dat[j][2 * g]);
            const float4 w = *reinterpret_cast<const float4*>(&S.w2[j][4 * q]);
            e1[0][0] = fmaf(w.x, d.x, e1[0][0]); e1[0][1] = fmaf(w.y, d.x, e1[0][1]);
            e1[0][2] = fmaf(w.z, d.x, e1[0][2]); e1[0][3] = fmaf(w.w, d.x, e1[0][3]);
            e1[1][0] = fmaf(w.x, d.y, e1[1][0]); e1[1][1] = fmaf(w.y, d.y, e1[1][1]);
            e1[1][2] = fmaf(w.z, d.y, e1[1][2]); e1[1][3] = fmaf(w.w, d.y, e1[1][3]);
        }
        __syncthreads();   // da has been read
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[2 * g + u][4 * q]);
            *reinterpret_cast<float4*>(&S.da[2 * g + u][4 * q]) =
                make_float4(h.x > 0.f ? e1[u][0] : 0.f, h.y > 0.f ? e1[u][1] : 0.f, h.z > 0.f ? e1[u][2] : 0.f,
                            h.w > 0.f ? e1[u][3] : 0.f);
        }
        __syncthreads();
        // gradients of W1 and b1: unit tid / 4, input tid % 4
#pragma unroll 8
        for (int t = 0; t < kGroup; ++t) {
            const float d = S.da[t][tid >> 2];
            gw1 = fmaf(d, S.x[t][tid & 3], gw1);
            gb1 += d;
        }
    }
    float* P = part + (int64_t)blockIdx.x * kPartStride;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        *reinterpret_cast<float4*>(P + oW2 + (4 * g + u) * kHid + 4 * q) = make_float4(gw2[u][0], gw2[u][1], gw2[u][2], gw2[u][3]);
    P[oW1 + tid] = gw1;
    if ((tid & 3) == 0) P[oB1 + (tid >> 2)] = gb1;
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        S.red[0][g][4 * q + v] = gw3[v];
        S.red[1][g][4 * q + v] = gb2[v];
    }
    if (q == 0) {
        S.dy[g][0] = gb3;
        S.dy[g][1] = loss;
    }
    __syncthreads();
    if (tid < 2 * kHid) {
        const int which = tid / kHid, j = tid % kHid;
        float v = 0.f;
        for (int k = 0; k < 16; ++k) v += S.red[which][k][j];
        P[(which == 0 ? oW3 : oB2) + j] = v;
    }
    if (tid < 2) {
        float v = 0.f;
        for (int k = 0; k < 16; ++k) v += S.dy[k][tid];
        P[tid == 0 ? oB3 : kCapParams] = v;
    }
}

// The blocks' shares summed, 16 threads a parameter; with `adam`, an Adam step on
// the master copy and its FP16 copy. Bound by the latency of its loads, so all
// that can be are in flight together.
constexpr int kSumWarps = 16;
__global__ void __launch_bounds__(32 * kSumWarps) k_cap_sum(const float* __restrict__ part, int blocks, float* __restrict__ grad,
                                                            bool adam, float* __restrict__ w, __half* __restrict__ w16,
                                                            float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                                                            float b2, float eps, float c1, float c2)
{
    __shared__ float s[kSumWarps][32];
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
    const bool step = adam && k == 0 && p < kCapParams;
    const float m0 = step ? m[p] : 0.f, v0 = step ? v[p] : 0.f, w0 = step ? w[p] : 0.f;   // (the last step's: complete)
    chain_begin();
    float sum = 0.f;
    if (p <= kCapParams) {
        constexpr int kMost = (kCapBlocks + kSumWarps - 1) / kSumWarps;
        float x[kMost];
#pragma unroll
        for (int i = 0; i < kMost; ++i) {
            const int b = k + i * kSumWarps;
            x[i] = b < blocks ? part[(int64_t)b * kPartStride + p] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kMost; ++i) sum += x[i];
    }
    s[k][lane] = sum;
    __syncthreads();
    if (k != 0 || p > kCapParams) return;
    float g = 0.f;
#pragma unroll
    for (int i = 0; i < kSumWarps; ++i) g += s[i][lane];
    grad[p] = g;
    if (!step) return;
    const float mm = fmaf(b1, m0, (1.f - b1) * g);
    const float vv = fmaf(b2, v0, (1.f - b2) * g * g);
    m[p] = mm;
    v[p] = vv;
    const float wn = w0 - lr * (mm * c1) / (sqrtf(vv * c2) + eps);
    w[p] = wn;
    w16[p] = __float2half_rn(wn);
}

__global__ void k_cap_to_half(const float* __restrict__ w, __half* __restrict__ w16)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < kCapParams) w16[p] = __float2half_rn(w[p]);
}

// Capacities from the previous frame's exact tile counts: prev * (1 + margin)
// + pad; or, given a uniform count (> 0), that count for every tile instead.
__global__ void k_capacity_from_previous(const uint32_t* __restrict__ prev, int64_t n_tiles, float margin,
                                         uint32_t pad, uint32_t uniform, uint32_t* __restrict__ cap)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tiles) return;
    const float c = uniform ? (float)uniform : (float)prev[t];
    cap[t] = (uint32_t)fminf(c * (1.f + margin) + (float)pad, 4.0e9f);
}

// The exact tile counts against the chosen capacities: a tile's lists go to its
// region [cap_off[t], cap_off[t+1]), or to the pool after all regions (scal[14]
// records taken, scal[6] tiles) if they do not fit; a frame whose pool runs out
// is not drawn (error bit kErrPool) but drawn again without capacities.
constexpr unsigned long long kErrPool = 16ull;
__global__ void k_capacity_check(const uint32_t* __restrict__ tile_frag, const uint64_t* __restrict__ cap_off,
                                 int64_t n_tiles, uint64_t frag_cap, unsigned long long* __restrict__ scal)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tiles) return;
    const uint64_t total = tile_frag[t], region = cap_off[t];
    if (region + total <= cap_off[t + 1] && region + total <= frag_cap) return;
    const uint64_t p = atomicAdd(&scal[14], (unsigned long long)total);
    atomicAdd(&scal[6], 1ull);
    if (cap_off[n_tiles] + p + total > frag_cap) atomicOr(&scal[5], kErrPool);
}

}  // namespace

cudaError_t launch_capacity_from_previous(FrameBufs& fb, int64_t n_tiles, float margin, uint32_t pad, uint32_t uniform,
                                          cudaStream_t s)
{
    k_capacity_from_previous<<<grid_for(n_tiles, 256), 256, 0, s>>>(fb.tile_frag, n_tiles, margin, pad, uniform,
                                                                     fb.tile_cap);
    return cudaGetLastError();
}

cudaError_t launch_capacity_check(FrameBufs& fb, int64_t n_tiles, cudaStream_t s)
{
    k_capacity_check<<<grid_for(n_tiles, 256), 256, 0, s>>>(fb.tile_frag, fb.cap_off, n_tiles, (uint64_t)fb.frag_cap,
                                                            reinterpret_cast<unsigned long long*>(fb.scal));
    return cudaGetLastError();
}

cudaError_t prepare_capacity_kernels()
{
    const cudaError_t e = cudaFuncSetAttribute(k_cap_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(NetSmem));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_cap_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NetSmem));
}

int64_t cap_partials() { return (int64_t)kCapBlocks * kPartStride; }

static unsigned cap_grid(int64_t n) { return (unsigned)std::min<int64_t>((n + kGroup - 1) / kGroup, kCapBlocks); }

cudaError_t launch_cap_forward(const CapNet& net, FrameBufs& fb, int64_t n_tiles, float margin, uint32_t pad,
                               cudaStream_t s)
{
    k_cap_forward<<<cap_grid(n_tiles), kCapThreads, sizeof(NetSmem), s>>>(fb.cap_x, n_tiles, net.w16, margin, pad,
                                                                           fb.tile_cap);
    return cudaGetLastError();
}

cudaError_t launch_cap_grad(CapNet& net, const float* X, const uint32_t* counts, int64_t n, float lr, bool chained,
                            cudaStream_t s)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const bool adam = lr > 0.f;
    if (adam) net.step += 1;
    const float c1 = 1.f / (1.f - std::pow(b1, (float)net.step)), c2 = 1.f / (1.f - std::pow(b2, (float)net.step));
    const unsigned blocks = cap_grid(n);
    cudaError_t e = launch_chained(k_cap_backward, blocks, kCapThreads, sizeof(NetSmem), s, chained, X, counts, n, net.w16,
                                   net.part);
    if (e != cudaSuccess) return e;
    return launch_chained(k_cap_sum, grid_for(kCapParams + 1, 32), 32 * kSumWarps, 0, s, chained, net.part, (int)blocks,
                          net.grad, adam, net.w, net.w16, net.m, net.v, lr, b1, b2, eps, c1, c2);
}

cudaError_t launch_cap_to_half(CapNet& net, cudaStream_t s)
{
    k_cap_to_half<<<grid_for(kCapParams, 256), 256, 0, s>>>(net.w, net.w16);
    return cudaGetLastError();
}

}  // namespace hexfc
