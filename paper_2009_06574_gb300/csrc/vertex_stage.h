// The vertex stage: camera transform of one vertex in double precision in a fixed
// order (the definition), and the same results from pairs of floats where those
// decide them. Compiles for the device and, for tests, for the host (without
// floating-point contraction).
#pragma once
#include <stdint.h>

#include <cmath>
#include <cstring>

#if defined(__CUDACC__)
#define HEXFC_HD __device__ __forceinline__
#define HEXFC_HD_COLD static __device__ __noinline__
#else
#define HEXFC_HD inline
#define HEXFC_HD_COLD inline
#endif

namespace hexfc {

// Camera constants of the vertex stage (double, evaluated without FMA).
struct CamParams {
    double eye[3], R[3], U[3], F[3];
    double focal, scale, cx, cy, znear, zfar, zf_over;
    int ortho, W, H;   // W, H: size of the drawn rectangle (the frame's unless a sub-rectangle is drawn)
    int ox, oy;   // drawn rectangle's offset in the frame (pixels): window positions are shifted by it
};

// A projected vertex: window position (16.8), window depth, eye depth.
struct ProjVertex {
    int32_t x, y, z, valid;
    float depth;
};

#if !defined(__CUDACC__)
// the device's names for correctly rounded operations
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __frcp_rn(float a) { return 1.f / a; }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __ddiv_rn(double a, double b) { return a / b; }
inline int32_t float_bits(float v) { int32_t b; std::memcpy(&b, &v, 4); return b; }
inline float float_of(int32_t b) { float v; std::memcpy(&v, &b, 4); return v; }
#else
HEXFC_HD int32_t float_bits(float v) { return __float_as_int(v); }
HEXFC_HD float float_of(int32_t b) { return __int_as_float(b); }
#endif

// A value as the unevaluated sum of two floats (about 48 bits), and its
// operations (Dekker 1971, Knuth TAOCP 2; the products by fma).
struct F2 {
    float h, l;
};
HEXFC_HD F2 f2_fast(float a, float b)   // |a| >= |b|
{
    const float h = __fadd_rn(a, b);
    return F2{h, __fsub_rn(b, __fsub_rn(h, a))};
}
HEXFC_HD F2 f2_sum(float a, float b)
{
    const float h = __fadd_rn(a, b), t = __fsub_rn(h, a);
    return F2{h, __fadd_rn(__fsub_rn(a, __fsub_rn(h, t)), __fsub_rn(b, t))};
}
HEXFC_HD F2 f2_add(F2 a, F2 b)
{
    const F2 s = f2_sum(a.h, b.h), t = f2_sum(a.l, b.l);
    const F2 v = f2_fast(s.h, __fadd_rn(s.l, t.h));
    return f2_fast(v.h, __fadd_rn(t.l, v.l));
}
HEXFC_HD F2 f2_mul(F2 a, F2 b)
{
    const float h = __fmul_rn(a.h, b.h);
    const float e = fmaf(a.h, b.h, -h);
    return f2_fast(h, __fadd_rn(e, fmaf(a.h, b.l, __fmul_rn(a.l, b.h))));
}
HEXFC_HD F2 f2_neg(F2 a) { return F2{-a.h, -a.l}; }
HEXFC_HD F2 f2_rcp(F2 a)   // one Newton step from the float reciprocal
{
    const float y = __frcp_rn(a.h);
    const F2 e = f2_add(F2{1.f, 0.f}, f2_neg(f2_mul(a, F2{y, 0.f})));   // 1 - a y
    return f2_add(F2{y, 0.f}, f2_mul(e, F2{y, 0.f}));
}
// rint(v) if no value within `margin` of v rounds otherwise.
HEXFC_HD bool f2_rint(F2 v, float margin, int32_t& out)
{
    const float r = rintf(v.h);
    const float d = __fadd_rn(__fsub_rn(v.h, r), v.l);   // v - r: the difference is exact
    const float k = rintf(d);
    out = (int32_t)r + (int32_t)k;
    return fabsf(__fsub_rn(d, k)) < 0.5f - margin - 0x1p-23f;   // (d itself is rounded)
}
// Camera constants of the vertex stage in pairs of floats.
struct CamPairs {
    F2 eye[3], R[3], U[3], F[3];
    F2 focal, cx, cy, znear, zfar, zf_over, inv_range;   // focal: the scale in an orthographic view
    bool usable;   // every constant is within the floats' range
};

// The vertex stage in double, in the order that defines it.
HEXFC_HD_COLD void vertex_double(float px, float py, float pz, const CamParams& cam, ProjVertex& o)
{
    double dx = __dsub_rn((double)px, cam.eye[0]);
    double dy = __dsub_rn((double)py, cam.eye[1]);
    double dz = __dsub_rn((double)pz, cam.eye[2]);
    double ex = __dadd_rn(__dadd_rn(__dmul_rn(dx, cam.R[0]), __dmul_rn(dy, cam.R[1])), __dmul_rn(dz, cam.R[2]));
    double ey = __dadd_rn(__dadd_rn(__dmul_rn(dx, cam.U[0]), __dmul_rn(dy, cam.U[1])), __dmul_rn(dz, cam.U[2]));
    double ed = __dadd_rn(__dadd_rn(__dmul_rn(dx, cam.F[0]), __dmul_rn(dy, cam.F[1])), __dmul_rn(dz, cam.F[2]));
    double xw, yw, z;
    if (cam.ortho) {
        xw = __dadd_rn(cam.cx, __dmul_rn(ex, cam.scale));
        yw = __dsub_rn(cam.cy, __dmul_rn(ey, cam.scale));
        z = __ddiv_rn(__dsub_rn(ed, cam.znear), __dsub_rn(cam.zfar, cam.znear));
    } else {
        xw = __dadd_rn(cam.cx, __dmul_rn(__ddiv_rn(ex, ed), cam.focal));
        yw = __dsub_rn(cam.cy, __dmul_rn(__ddiv_rn(ey, ed), cam.focal));
        z = __dmul_rn(cam.zf_over, __dsub_rn(1.0, __ddiv_rn(cam.znear, ed)));
    }
    bool valid = (ed > cam.znear) && (ed < cam.zfar) && (fabs(xw) <= 16384.0) && (fabs(yw) <= 16384.0);
    o = ProjVertex{0, 0, 0, 0, (float)ed};
    if (valid) {
        z = fmin(fmax(z, 0.0), 1.0);
        // snapped in frame coordinates, then moved by whole pixels into the drawn
        // rectangle: coverage, depth and edge distances are those of the frame
        o.x = (int32_t)rint(__dmul_rn(xw, 256.0)) - 256 * cam.ox;
        o.y = (int32_t)rint(__dmul_rn(yw, 256.0)) - 256 * cam.oy;
        o.z = (int32_t)(uint32_t)rint(__dmul_rn(z, 16777215.0));
        o.valid = 1;
    }
}

// The same from pairs of floats, where that decides it: every result is a
// rounding or a comparison of a value that the pairs give to about 2^-44, so it
// is taken from them unless the value lies within a margin of where the result
// changes (2^-42 of each operation's largest operand, several times what the
// pairs and the double evaluation differ by); false if some result does.
HEXFC_HD bool vertex_pairs(float vx, float vy, float vz, const CamPairs& c, const CamParams& cam, ProjVertex& o)
{
    constexpr float u = 0x1p-42f;
    const F2 dx = f2_add(F2{vx, 0.f}, f2_neg(c.eye[0])), dy = f2_add(F2{vy, 0.f}, f2_neg(c.eye[1])),
             dz = f2_add(F2{vz, 0.f}, f2_neg(c.eye[2]));
    auto dot = [&](const F2 (&B)[3]) { return f2_add(f2_add(f2_mul(dx, B[0]), f2_mul(dy, B[1])), f2_mul(dz, B[2])); };
    const F2 ex = dot(c.R), ey = dot(c.U), ed = dot(c.F);
    // |ex|, |ey|, |ed| are known to within 4 u D (the basis vectors have components of at most 1)
    const float D = fabsf(dx.h) + fabsf(dy.h) + fabsf(dz.h) + fabsf(vx) + fabsf(vy) + fabsf(vz);
    const float m = 4.f * u * D;
    F2 xw, yw, z;
    float mx, my, mz;
    if (cam.ortho) {
        const F2 px = f2_mul(ex, c.focal), py = f2_mul(ey, c.focal);
        xw = f2_add(c.cx, px);
        yw = f2_add(c.cy, f2_neg(py));
        z = f2_mul(f2_add(ed, f2_neg(c.znear)), c.inv_range);
        mx = fmaf(m, fabsf(c.focal.h), u * (fabsf(px.h) + c.cx.h));
        my = fmaf(m, fabsf(c.focal.h), u * (fabsf(py.h) + c.cy.h));
        mz = (m + u * (fabsf(ed.h) + fabsf(c.znear.h))) * fabsf(c.inv_range.h) + 4.f * u;
    } else {
        const F2 r = f2_rcp(ed);
        const F2 qx = f2_mul(ex, r), qy = f2_mul(ey, r);
        const F2 px = f2_mul(qx, c.focal), py = f2_mul(qy, c.focal);
        xw = f2_add(c.cx, px);
        yw = f2_add(c.cy, f2_neg(py));
        const F2 nz = f2_mul(c.znear, r);
        z = f2_mul(c.zf_over, f2_add(F2{1.f, 0.f}, f2_neg(nz)));
        const float rel = fmaf(m, fabsf(r.h), u);   // relative error of r, and the absolute one of ex r + |q| u
        mx = fmaf(c.focal.h * rel, 1.f + 2.f * fabsf(qx.h), u * c.cx.h);
        my = fmaf(c.focal.h * rel, 1.f + 2.f * fabsf(qy.h), u * c.cy.h);
        mz = fabsf(c.zf_over.h) * fmaf(2.f * fabsf(nz.h), rel, 2.f * u);
    }
    // the comparisons: each has to be clear of its margin
    const F2 a = f2_add(ed, f2_neg(c.znear)), b = f2_add(c.zfar, f2_neg(ed));
    bool sure = fabsf(a.h) > m + u * fabsf(c.znear.h) && fabsf(b.h) > m + u * fabsf(c.zfar.h) &&
                fabsf(fabsf(xw.h) - 16384.f) > mx + 0.002f && fabsf(fabsf(yw.h) - 16384.f) > my + 0.002f;
    const bool valid = a.h > 0.f && b.h > 0.f && fabsf(xw.h) <= 16384.f && fabsf(yw.h) <= 16384.f;
    o = ProjVertex{0, 0, 0, 0, ed.h};
    if (valid) {
        const F2 w{256.f * xw.h, 256.f * xw.l}, v{256.f * yw.h, 256.f * yw.l};   // exact
        sure = f2_rint(w, 256.f * mx, o.x) && sure;
        sure = f2_rint(v, 256.f * my, o.y) && sure;
        sure = f2_rint(f2_mul(z, F2{16777215.f, 0.f}), 16777216.f * (mz + 2.f * u), o.z) && sure;
        if (!(z.h > mz && z.h < 1.f - mz)) sure = false;   // (clamped)
        o.x -= 256 * cam.ox;
        o.y -= 256 * cam.oy;
        o.valid = 1;
    }
    // the eye depth to float: the pair's high part unless the low one is near half
    // a unit of its last place (a quarter below a power of two)
    const int32_t eb = float_bits(fabsf(ed.h));
    const float half = float_of((eb & 0x7F800000) - (((eb & 0x7FFFFF) ? 24 : 25) << 23));
    sure = sure && fabsf(ed.l) + m < half;
    // (NaN, overflow and tiny values fail one of these)
    return sure && D < 1e15f && fabsf(ed.h) > 1e-12f;
}

inline F2 pair_of(double v) { return F2{(float)v, (float)(v - (double)(float)v)}; }

inline CamPairs cam_pairs(const CamParams& c)
{
    CamPairs p{};
    p.usable = true;
    auto put = [&](double v) {
        p.usable = p.usable && std::fabs(v) < 1e15;   // (not NaN)
        return pair_of(v);
    };
    for (int d = 0; d < 3; ++d) {
        p.eye[d] = put(c.eye[d]);
        p.R[d] = put(c.R[d]);
        p.U[d] = put(c.U[d]);
        p.F[d] = put(c.F[d]);
    }
    p.focal = put(c.ortho ? c.scale : c.focal);
    p.cx = put(c.cx);
    p.cy = put(c.cy);
    p.znear = put(c.znear);
    p.zfar = put(c.zfar);
    p.zf_over = put(c.ortho ? 0.0 : c.zf_over);
    p.inv_range = put(1.0 / (c.zfar - c.znear));
    return p;
}

}  // namespace hexfc
