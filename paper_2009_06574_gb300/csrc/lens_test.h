// Whether a triangle lies wholly outside the sphere lens. Compiles for the device
// and, for tests, for the host.
#pragma once
#include <cmath>

#if defined(__CUDACC__)
#define HEXFC_LENS_FN __device__ __forceinline__
#else
#define HEXFC_LENS_FN inline
#endif

namespace hexfc {

#if !defined(__CUDACC__)
// the device's names
inline float rsqrtf(float v) { return 1.f / std::sqrt(v); }
inline float __fdividef(float a, float b) { return a / b; }
using std::fabs;
using std::fmax;
using std::fmin;
#endif

// The triangle's corners have offsets o[k] from the lens' centre and eye depths
// e[k]; inv_r: 1 / the lens' radius. The offsets, projected on the direction of
// their sum, are all above the radius, so every point of the triangle is. The
// margin covers the rounding of a sample's distance (affine sums of offset / w and
// 1 / w in float: below 12 * 2^-24 of the largest offset, times the ratio of the
// eye depths), so that the computed distance is at least 1 too, and the sample's
// focus exactly 0. The answer is no wherever it is not certain: offsets that
// cancel (the centre is the triangle's centroid) or nearly vanish give no
// direction, offsets beyond 1e15 squares that overflow, and every comparison fails
// on a NaN.
HEXFC_LENS_FN bool outside_lens(const float (&o)[3][3], const float (&e)[3], bool ortho, float inv_r)
{
    const float mx = o[0][0] + o[1][0] + o[2][0], my = o[0][1] + o[1][1] + o[2][1],
                mz = o[0][2] + o[1][2] + o[2][2];
    const float m2 = mx * mx + my * my + mz * mz, im = rsqrtf(m2);
    float near[3], far = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        near[k] = (o[k][0] * mx + o[k][1] * my + o[k][2] * mz) * im;
        far = fmaxf(far, fabsf(o[k][0]) + fabsf(o[k][1]) + fabsf(o[k][2]));
    }
    const float e_lo = fminf(e[0], fminf(e[1], e[2])), e_hi = fmaxf(e[0], fmaxf(e[1], e[2]));
    const float ratio = ortho ? 1.f : fmaxf(__fdividef(e_hi, e_lo), 1.f);
    const float bound = 1.0001f + 8e-6f * far * inv_r * ratio;
    return (ortho || e_lo > 0.f) && m2 > 1e-30f && far < 1e15f && near[0] * inv_r >= bound && near[1] * inv_r >= bound &&
           near[2] * inv_r >= bound;
}

}  // namespace hexfc
