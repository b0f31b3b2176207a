// Fragment shading of the focus+context renderer (Section "Focus+Context",
// Eqs. 1-4), used by the drawing kernels of this library.
#pragma once
#include "raster_common.cuh"

namespace hexfc {

// Shading and depth inputs of one triangle of a tile's list (vertices in wound
// order), read by the lanes 16 bytes at a time. Eleven vectors, an odd stride
// in 16-byte units, so the lanes of a quarter warp that read different
// triangles of a chunk share banks only when the triangles' indices agree
// modulo 8. The first eight are what a sample outside the lens needs; the last
// three (the lens distance) are read only where the lens may reach.
// Coordinates are in 1/256-pixel units; integers below 2^24 are exact in float.
//
// Perspective-correct interpolation of an attribute a with vertex weights
// lam_k (lam_0 = 1 - lam_1 - lam_2) is sum lam_k a_k / w_k over
// sum lam_k / w_k (w = eye depth). Both sums are affine in (lam_1, lam_2), so
// each is kept as its value at vertex 0 and two differences: with q_k = 1/w_k,
// Q = q0 + lam_1 dq1 + lam_2 dq2 and sum lam_k a_k q_k = A0 + lam_1 dA1 + lam_2 dA2.
// Orthographic views use q_k = 1.
struct ShadeRec {
    float4 nx, ny;   // face corners, negated
    float4 nl;       // -1 / squared length of face edge k -> k+1 (0: degenerate)
    float4 qa;       // q0, dq1, dq2 (1 / eye depth); a0 (importance / eye depth)
    uint4 aw;        // da1, da2 (float bits); low words of the edge functions of vertices 1, 2 at the tile's first sample
    int4 ev;         // dx, dy of the edges opposite vertices 1 and 2 (16.8)
    uint4 zf;        // window depth of vertex 0 | face edge flags << 24; depths of vertices 1, 2 less it (int); f2t
    uint4 ha;        // the same differences (float bits); twice the area A if below 2^26 else 0, with kRecLens,
                     // kRecEdge, kRecBound; 1 / A (float bits), or if A is larger its low word
    float4 p0;       // p0.x, p0.y, p0.z (p = (world position - sphere lens centre) / eye depth); dp1.x
    float4 p1;       // dp1.y, dp1.z; dp2.x, dp2.y
    uint4 p2;        // dp2.z (float bits); high words of the two edge functions and of A
};
static_assert(sizeof(ShadeRec) == 11 * 16, "eleven 16-byte vectors");
constexpr uint32_t kRecLens = 1u << 31;    // the sphere lens may reach the triangle
constexpr uint32_t kRecEdge = 1u << 30;    // an edge of the face is visible in context
constexpr uint32_t kRecBound = 1u << 29;   // a boundary face
constexpr uint32_t kRecArea = (1u << 26) - 1u;

// -1 / the squared lengths of a face's window edges, k -> k + 1.
__device__ __forceinline__ float4 edge_scales(const int4& X, const int4& Y)
{
    const int32_t FX[4] = {X.x, X.y, X.z, X.w}, FY[4] = {Y.x, Y.y, Y.z, Y.w};
    float nl[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int32_t ex = FX[(k + 1) & 3] - FX[k], ey = FY[(k + 1) & 3] - FY[k];
        const float l2 = u64_to_f32((uint64_t)((int64_t)ex * ex + (int64_t)ey * ey));
        nl[k] = l2 > 0.f ? -__frcp_rn(l2) : 0.f;
    }
    return make_float4(nl[0], nl[1], nl[2], nl[3]);
}

// The record of triangle f2t (from the records F, S of its face, E if kept) for
// the tile whose first pixel is (px0, py0). The positions are read only where
// the sphere lens may reach.
__device__ __forceinline__ void make_record(const FaceFrame& F, const FaceStatic& S, const FaceExtra* E, uint32_t f2t,
                                            int px0, int py0, const ShadeParams& sp, ShadeRec& R)
{
    const Pair16 fa = load32(&F.X), fb = load32(&F.Z);
    const int4 X = as_int4(fa.a), Y = as_int4(fa.b);
    const uint4 Z = fb.a;
    const float4 fq = as_float4(fb.b), imp = S.imp;
    Pair16 ex{};
    if (E) ex = load32(E);
    const bool second = f2t & 1u;
    const uint32_t flags = face_flags(Z) >> (f2t & 1u);   // this triangle's bits in triangle 0's places
    // |coordinate| <= 2^22: exact in float
    R.nx = make_float4(-(float)X.x, -(float)X.y, -(float)X.z, -(float)X.w);
    R.ny = make_float4(-(float)Y.x, -(float)Y.y, -(float)Y.z, -(float)Y.w);
    R.nl = E ? as_float4(ex.a) : edge_scales(X, Y);
    // vertices 1 and 2: corners (1, 2) or (2, 3), swapped if the triangle winds the other way
    const bool sw = flags & kFaceSwapped;
    auto pick = [&](auto b, auto c, auto d, auto& v1, auto& v2) {
        const auto u = second ? c : b, w = second ? d : c;
        v1 = sw ? w : u;
        v2 = sw ? u : w;
    };
    int32_t x1, x2, y1, y2;
    uint32_t z1, z2;
    float q1, q2, i1, i2;
    pick(X.y, X.z, X.w, x1, x2);
    pick(Y.y, Y.z, Y.w, y1, y2);
    pick(Z.y & kZ24, Z.z & kZ24, Z.w & kZ24, z1, z2);
    pick(fq.y, fq.z, fq.w, q1, q2);
    pick(imp.y, imp.z, imp.w, i1, i2);
    const uint32_t z0 = Z.x & kZ24;
    const float a0 = __fmul_rn(imp.x, fq.x), a1 = __fmul_rn(i1, q1), a2 = __fmul_rn(i2, q2);
    R.qa = make_float4(fq.x, q1 - fq.x, q2 - fq.x, a0);
    const int32_t dx1 = X.x - x2, dy1 = Y.x - y2;   // edge opposite vertex 1: 2 -> 0
    const int32_t dx2 = x1 - X.x, dy2 = y1 - Y.x;   // edge opposite vertex 2: 0 -> 1
    // edge functions at the tile's first sample, low words: exact modulo 2^32,
    // and at a covered sample of a small triangle the value itself lies in [0, area]
    const int32_t sx = 256 * px0 + 128, sy = 256 * py0 + 128;
    const uint32_t e1 = (uint32_t)dx1 * (uint32_t)(sy - y2) - (uint32_t)dy1 * (uint32_t)(sx - x2);
    const uint32_t e2 = (uint32_t)dx2 * (uint32_t)(sy - Y.x) - (uint32_t)dy2 * (uint32_t)(sx - X.x);
    R.aw = make_uint4(__float_as_uint(a1 - a0), __float_as_uint(a2 - a0), e1, e2);
    R.ev = make_int4(dx1, dy1, dx2, dy2);
    const int32_t d1 = (int32_t)(z1 - z0), d2 = (int32_t)(z2 - z0);
    R.zf = make_uint4(z0 | (face_edge_flags(Z) << 24), (uint32_t)d1, (uint32_t)d2, f2t);
    const bool lens = !(flags & kFaceOut) && sp.lens_mode == HEXFC_LENS_SPHERE;
    uint32_t area, iw;
    if (E) {
        const uint4 A = ex.b;
        area = second ? A.y : A.x;
        iw = second ? A.w : A.z;
    } else {
        const uint64_t twice = (uint64_t)edge_fn(X.x, Y.x, x1, y1, x2, y2);
        area = twice < (1ull << 26) ? (uint32_t)twice : 0u;
        iw = __float_as_uint(__frcp_rn((float)area));
    }
    uint4 p2 = make_uint4(0u, 0u, 0u, 0u);
    if (area == 0) {   // a large triangle: 64-bit edge functions and area (wound: positive)
        const int64_t f1 = edge_fn(x2, y2, X.x, Y.x, sx, sy), f2 = edge_fn(X.x, Y.x, x1, y1, sx, sy);
        const uint64_t big = (uint64_t)edge_fn(X.x, Y.x, x1, y1, x2, y2);
        p2 = make_uint4(0u, (uint32_t)((uint64_t)f1 >> 32), (uint32_t)((uint64_t)f2 >> 32), (uint32_t)(big >> 32));
        iw = (uint32_t)big;
    }
    R.ha = make_uint4(__float_as_uint((float)d1), __float_as_uint((float)d2),
                      area | (lens ? kRecLens : 0u) | ((Z.x >> 28) ? kRecEdge : 0u) |
                          ((face_flags(Z) & kFaceBoundary) ? kRecBound : 0u),
                      iw);
    if (lens) {
        // offsets from the lens' centre
        const float4 wx = S.px, wy = S.py, wz = S.pz;
        float ox1, ox2, oy1, oy2, oz1, oz2;
        pick(wx.y - sp.lens_c[0], wx.z - sp.lens_c[0], wx.w - sp.lens_c[0], ox1, ox2);
        pick(wy.y - sp.lens_c[1], wy.z - sp.lens_c[1], wy.w - sp.lens_c[1], oy1, oy2);
        pick(wz.y - sp.lens_c[2], wz.z - sp.lens_c[2], wz.w - sp.lens_c[2], oz1, oz2);
        const float P0 = __fmul_rn(wx.x - sp.lens_c[0], fq.x), P1 = __fmul_rn(wy.x - sp.lens_c[1], fq.x),
                    P2 = __fmul_rn(wz.x - sp.lens_c[2], fq.x);
        R.p0 = make_float4(P0, P1, P2, __fmul_rn(ox1, q1) - P0);
        R.p1 = make_float4(__fmul_rn(oy1, q1) - P1, __fmul_rn(oz1, q1) - P2, __fmul_rn(ox2, q2) - P0,
                           __fmul_rn(oy2, q2) - P1);
        p2.x = __float_as_uint(__fmul_rn(oz2, q2) - P2);
    }
    R.p2 = p2;
}

// A covered sample of a triangle: its weights and exact depth. (sx8, sy8): the
// pixel in its tile, 1/256-pixel units.
struct Sample {
    float lam1, lam2;
    uint32_t z;
};
// The parts of sample_of that few samples need: a large triangle (64-bit
// weights), or a depth whose float estimate q was off (remainder r).
static __device__ __noinline__ Sample sample_rare(const ShadeRec& R, Sample s, int32_t r, uint32_t sx8, uint32_t sy8, bool& bad)
{
    const uint4 zf = R.zf, ha = R.ha, aw = R.aw, hw = R.p2;
    const int32_t area = (int32_t)(ha.z & kRecArea);
    if (area != 0) {
#pragma unroll 1
        for (int it = 0; it < 16 && r < 0; ++it) { --s.z; r += area; }
#pragma unroll 1
        for (int it = 0; it < 16 && r >= area; ++it) { ++s.z; r -= area; }
        if ((uint32_t)r >= (uint32_t)area) bad = true;
        return s;
    }
    const int4 ev = R.ev;
    const int64_t big = (int64_t)(((uint64_t)hw.w << 32) | ha.w);
    const float ia = 1.f / u64_to_f32((uint64_t)big);
    const int64_t l1 = (int64_t)(((uint64_t)hw.y << 32) | aw.z) + (int64_t)ev.x * (int32_t)sy8 -
                       (int64_t)ev.y * (int32_t)sx8;
    const int64_t l2 = (int64_t)(((uint64_t)hw.z << 32) | aw.w) + (int64_t)ev.z * (int32_t)sy8 -
                       (int64_t)ev.w * (int32_t)sx8;
    s.lam1 = __fmul_rn(u64_to_f32((uint64_t)l1), ia);
    s.lam2 = __fmul_rn(u64_to_f32((uint64_t)l2), ia);
    s.z = sample_depth_lam(zf.x & kZ24, (int32_t)zf.y, (int32_t)zf.z, l1, l2, big, s.lam1, s.lam2,
                           __uint_as_float(ha.x), __uint_as_float(ha.y), bad);
    return s;
}

// A triangle with twice its area A below 2^26 (16.8 units squared: below 512
// square pixels) takes its weights in 32-bit arithmetic, exact modulo 2^32: at a
// covered sample 0 <= l <= A < 2^26. Its depth: with lam within 5 ulp and 0 <=
// lam <= 1, |d| < 2^24, the float estimate is within 8 of the quotient
// floor((l1 d1 + l2 d2) / A), so the exact remainder lies within (-9, 9) A, below
// 2^30 in magnitude, and its value modulo 2^32 read as a signed integer is exact.
__device__ __forceinline__ Sample sample_of(const ShadeRec& R, const uint4& zf, const uint4& ha, uint32_t sx8,
                                            uint32_t sy8, bool live, bool& bad)
{
    Sample s;
    const uint4 aw = R.aw;
    const int4 ev = R.ev;
    const uint32_t area = ha.z & kRecArea;
    const float ia = __uint_as_float(ha.w);
    const uint32_t l1 = aw.z + (uint32_t)ev.x * sy8 - (uint32_t)ev.y * sx8;
    const uint32_t l2 = aw.w + (uint32_t)ev.z * sy8 - (uint32_t)ev.w * sx8;
    s.lam1 = __fmul_rn((float)l1, ia);
    s.lam2 = __fmul_rn((float)l2, ia);
    const int32_t q = __float2int_rd(fmaf(s.lam1, __uint_as_float(ha.x), __fmul_rn(s.lam2, __uint_as_float(ha.y))));
    const int32_t r = (int32_t)(l1 * zf.y + l2 * zf.z - (uint32_t)q * area);
    s.z = (zf.x & kZ24) + (uint32_t)q;
    if ((uint32_t)r >= area && live) s = sample_rare(R, s, r, sx8, sy8, bad);   // (r < 0, and A = 0: large, too)
    return s;
}

// Square root of x >= 0 (0 at 0), the hardware approximation (a few units in
// the last place).
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Distance of pixel (px, py) from the screen lens, 1 at its border.
__device__ __forceinline__ float screen_lens_dist(int px, int py, const ShadeParams& sp)
{
    // (frame pixel coordinates, so that a drawn rectangle shades as the frame does)
    const float dx = ((float)(px + sp.px_off) + 0.5f) - sp.lens_c[0];
    const float dy = ((float)(py + sp.py_off) + 0.5f) - sp.lens_c[1];
    return sqrt_approx(fmaf(dx, dx, __fmul_rn(dy, dy))) * sp.lens_inv_r;
}

// Squared distances (1/256-pixel units) of the sample (sx, sy) to the face's
// four edge segments. The closest point of edge k is corner k + t e_k, t =
// clamp(v_k . e_k / |e_k|^2, 0, 1), with v_k = sample - corner k and e_k =
// corner k+1 - corner k (both exact). Two edges at a time (packed
// single-precision operations, each lane of which rounds as the scalar one).
__device__ __forceinline__ float4 edge_dist2(const ShadeRec& t, float sx, float sy)
{
    const float4 nx = t.nx, ny = t.ny, nl = t.nl;
    const float2 s2x = make_float2(sx, sx), s2y = make_float2(sy, sy);
    const float2 vxa = __fadd2_rn(s2x, make_float2(nx.x, nx.y)), vxb = __fadd2_rn(s2x, make_float2(nx.z, nx.w));
    const float2 vya = __fadd2_rn(s2y, make_float2(ny.x, ny.y)), vyb = __fadd2_rn(s2y, make_float2(ny.z, ny.w));
    // -e_k = v_{k+1} - v_k
    const float2 exa = make_float2(vxa.y - vxa.x, vxb.x - vxa.y), exb = make_float2(vxb.y - vxb.x, vxa.x - vxb.y);
    const float2 eya = make_float2(vya.y - vya.x, vyb.x - vya.y), eyb = make_float2(vyb.y - vyb.x, vya.x - vyb.y);
    const float2 da = __ffma2_rn(vxa, exa, __fmul2_rn(vya, eya)), db = __ffma2_rn(vxb, exb, __fmul2_rn(vyb, eyb));
    const float2 ta = make_float2(__saturatef(__fmul_rn(da.x, nl.x)), __saturatef(__fmul_rn(da.y, nl.y)));
    const float2 tb = make_float2(__saturatef(__fmul_rn(db.x, nl.z)), __saturatef(__fmul_rn(db.y, nl.w)));
    const float2 xa = __ffma2_rn(ta, exa, vxa), ya = __ffma2_rn(ta, eya, vya);
    const float2 xb = __ffma2_rn(tb, exb, vxb), yb = __ffma2_rn(tb, eyb, vyb);
    const float2 d2a = __ffma2_rn(xa, xa, __fmul2_rn(ya, ya)), d2b = __ffma2_rn(xb, xb, __fmul2_rn(yb, yb));
    return make_float4(d2a.x, d2a.y, d2b.x, d2b.y);
}

// The least of the distances d, and of those whose bit k of `bits` is set (else infinity).
__device__ __forceinline__ float least(const float4& d) { return fminf(fminf(d.x, d.y), fminf(d.z, d.w)); }
__device__ __forceinline__ float least_of(const float4& d, uint32_t bits)
{
    return least(make_float4((bits & 1u) ? d.x : INFINITY, (bits & 2u) ? d.y : INFINITY, (bits & 4u) ? d.z : INFINITY,
                             (bits & 8u) ? d.w : INFINITY));
}

// Eqs. 1-4 for one fragment of triangle t at sample (sx, sy) (1/256-pixel
// units); lam1, lam2 are the screen-space barycentric weights of vertices 1
// and 2, flags the face's edge flags, dist the screen lens distance of the
// pixel (the sphere lens' is found here). Returns the premultiplied RGBA of Eq. 4.
__device__ __forceinline__ float4 shade_fragment(const ShadeRec& t, uint32_t flags, float lam1, float lam2, float sx,
                                                 float sy, float dist, const ShadeParams& sp)
{
    const float4 qa = t.qa;
    const float Q = fmaf(lam2, qa.z, fmaf(lam1, qa.y, qa.x));   // 1 / eye depth of the fragment
    const float iQ = __fdividef(1.f, Q);
    const float g = sp.ortho ? 1.f : fminf(fmaxf(sp.zref * Q, sp.g_min), sp.g_max);   // z_ref / z_eye
    const uint2 da = make_uint2(t.aw.x, t.aw.y);
    const float t_imp = fmaf(lam2, __uint_as_float(da.y), fmaf(lam1, __uint_as_float(da.x), qa.w)) * iQ;
    if (sp.lens_mode != HEXFC_LENS_SCREEN) {
        // the interpolated offset from the centre, P - C = D / Q (D affine in lam)
        const float4 p0 = t.p0, p1 = t.p1;
        const float Dx = fmaf(lam2, p1.z, fmaf(lam1, p0.w, p0.x));
        const float Dy = fmaf(lam2, p1.w, fmaf(lam1, p1.x, p0.y));
        const float Dz = fmaf(lam2, __uint_as_float(t.p2.x), fmaf(lam1, p1.y, p0.z));
        dist = sqrt_approx(fmaf(Dx, Dx, fmaf(Dy, Dy, __fmul_rn(Dz, Dz)))) * (iQ * sp.lens_inv_r);
        if (!(t.ha.z & kRecLens)) dist = 1.f;   // outside the lens (no p in the record): any distance from 1 on
    }
    // focus = 1 - smoothstep(0.7, 1, dist)
    const float st = __saturatef((dist - 0.7f) * (1.f / 0.3f));
    const float focus = fmaf(-__fmul_rn(st, st), fmaf(-2.f, st, 3.f), 1.f);
    const float4 d2 = edge_dist2(t, sx, sy);
    const float a2 = least(d2), f2 = least_of(d2, flags), c2 = least_of(d2, flags >> 4);
    // Eq. 1 with the depth-dependent width w, halo band h (focus edges); the
    // tests compare squared distances in 1/256-pixel units. Edges visible in
    // context are visible in focus too (c2 >= f2), so an edge in context
    // (alpha 1) is one in focus, and an edge in focus or in the halo band has
    // alpha = focus (in the band with focus 0 that is 0 as well).
    const float wg = __fmul_rn(256.f * sp.w_base, g);            // >= 0: w_base, g_min, halo_scale >= 0
    const float w256 = fmaf(0.3f * focus, wg, wg);
    const float wh256 = fmaf((0.3f + sp.halo_scale) * focus, wg, wg);
    const float w2 = __fmul_rn(w256, w256);
    const bool band = f2 <= __fmul_rn(wh256, wh256);
    const bool halo = band && f2 > w2 && focus > 0.f;
    const float alpha_e = c2 <= w2 ? 1.f : (band ? focus : 0.f);
    // colour table ctf = (t, 0, 1 - t); Eq. 2: accentuated faces (s_e = s > 1)
    // move the face colour towards white by beta
    const float tt = __saturatef((t_imp - sp.tf_lo) * sp.tf_inv);
    const bool accent = a2 <= sp.accent_r2;
    const float s_e = accent ? sp.s : 1.f;
    const float beta = s_e > 1.f ? sp.accent_beta : 0.f;
    const float dk = fmaf(-sp.darken, focus, 1.f);
    const float er = halo ? 1.f : __fmul_rn(tt, dk), eg = halo ? 1.f : 0.f, eb = halo ? 1.f : __fmul_rn(1.f - tt, dk);
    // Eq. 3 and Eq. 4
    const float ahat = fmaf(sp.alpha_span, tt, sp.alpha_min);
    const float dc = fminf(dist, 1.f);
    const float dc2 = dc * dc;
    const float af = fminf(s_e * (ahat * (dc2 * dc2)), 1.f);
    const float wf = __fmul_rn(1.f - alpha_e, af);
    float4 c = make_float4(fmaf(alpha_e, er, __fmul_rn(wf, fmaf(beta, 1.f - tt, tt))),
                           fmaf(alpha_e, eg, __fmul_rn(wf, beta)),
                           fmaf(alpha_e, eb, __fmul_rn(wf, fmaf(beta, tt, 1.f - tt))), alpha_e + wf);
    // depth cue (Section "Evaluation"): in focus and beyond the reference
    // depth, the colour moves towards its luma; opacity unchanged
    if (sp.desat > 0.f) {
        const float k = sp.desat * focus * fminf(fmaxf(1.f - g, 0.f), 1.f);
        const float y = fmaf(0.114f, c.z, fmaf(0.299f, c.x, __fmul_rn(0.587f, c.y)));
        c.x = fmaf(k, y - c.x, c.x);
        c.y = fmaf(k, y - c.y, c.y);
        c.z = fmaf(k, y - c.z, c.z);
    }
    return c;
}

// shade_fragment for a sample outside the lens (dist >= 1, sp.bounded), bit for
// bit: there the focus is exactly 0, so an edge is opaque or absent, halo,
// darkening and depth cue do nothing and Eq. 3's dist^4 is 1. It needs neither
// the lens distance nor the edges visible in focus; with kEdges false, none of
// the face's edges is visible in context either, and only the face is left.
template <bool kEdges>
__device__ __forceinline__ float4 shade_context(const ShadeRec& t, uint32_t flags, float lam1, float lam2, float sx,
                                                float sy, const ShadeParams& sp)
{
    const float4 qa = t.qa;
    const float Q = fmaf(lam2, qa.z, fmaf(lam1, qa.y, qa.x));
    const float iQ = __fdividef(1.f, Q);
    const uint2 da = make_uint2(t.aw.x, t.aw.y);
    const float t_imp = fmaf(lam2, __uint_as_float(da.y), fmaf(lam1, __uint_as_float(da.x), qa.w)) * iQ;
    const float4 d2 = edge_dist2(t, sx, sy);
    const float tt = __saturatef((t_imp - sp.tf_lo) * sp.tf_inv);
    const bool accent = least(d2) <= sp.accent_r2;
    const float s_e = accent ? sp.s : 1.f;
    const float beta = s_e > 1.f ? sp.accent_beta : 0.f;
    const float ahat = fmaf(sp.alpha_span, tt, sp.alpha_min);
    const float af = fminf(s_e * ahat, 1.f);
    float4 c = make_float4(__fmul_rn(af, fmaf(beta, 1.f - tt, tt)), __fmul_rn(af, beta),
                           __fmul_rn(af, fmaf(beta, tt, 1.f - tt)), af);
    if (kEdges) {
        const float g = sp.ortho ? 1.f : fminf(fmaxf(sp.zref * Q, sp.g_min), sp.g_max);
        const float wg = __fmul_rn(256.f * sp.w_base, g);
        if (least_of(d2, flags >> 4) <= __fmul_rn(wg, wg)) c = make_float4(tt, 0.f, 1.f - tt, 1.f);
    }
    return c;
}

}  // namespace hexfc
