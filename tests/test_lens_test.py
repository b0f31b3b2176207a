"""Triangles outside the sphere lens (csrc/lens_test.h), compiled for the host: the
answer is never yes where a point of the triangle lies within the lens, in 64
bits, or where the distance that the shading finds in float is below 1; lenses on
the triangles (centroids, corners, edges), scales from 1e-18 to 1e18, both
projections."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_06574_gb300", "csrc")

SOURCE = r"""
#include "lens_test.h"
#include <cmath>
using namespace hexfc;
// off: n x 3 x 3 corner offsets, depth: n x 3, w: m x 2 weights of corners 1 and 2.
// Counts the triangles taken for outside (found) that have a point inside (wrong).
extern "C" long check(const float* off, const float* depth, long n, int ortho, const float* inv_r, const float* w, long m,
                      long* found)
{
    long wrong = 0;
    *found = 0;
    for (long i = 0; i < n; ++i) {
        float o[3][3], e[3];
        for (int k = 0; k < 3; ++k) {
            e[k] = depth[3 * i + k];
            for (int d = 0; d < 3; ++d) o[k][d] = off[9 * i + 3 * k + d];
        }
        if (!outside_lens(o, e, ortho != 0, inv_r[i])) continue;
        ++*found;
        bool bad = false;
        float q[3], P[3][3];
        for (int k = 0; k < 3; ++k) {
            q[k] = ortho ? 1.f : 1.f / e[k];
            for (int d = 0; d < 3; ++d) P[k][d] = o[k][d] * q[k];
        }
        for (long s = 0; s < m; ++s) {
            const float a = w[2 * s], b = w[2 * s + 1];
            // the point itself
            const double c = 1.0 - (double)a - (double)b;
            const double W[3] = {c / (ortho ? 1.0 : e[0]), (double)a / (ortho ? 1.0 : e[1]), (double)b / (ortho ? 1.0 : e[2])};
            double d2 = 0.0;
            for (int d = 0; d < 3; ++d) {
                const double v = (W[0] * o[0][d] + W[1] * o[1][d] + W[2] * o[2][d]) / (W[0] + W[1] + W[2]);
                d2 += v * v;
            }
            bad = bad || !(std::sqrt(d2) * inv_r[i] >= 1.0);
            // its distance as the shading has it: sums affine in the weights
            const float Q = fmaf(b, q[2] - q[0], fmaf(a, q[1] - q[0], q[0]));
            float D[3];
            for (int d = 0; d < 3; ++d) D[d] = fmaf(b, P[2][d] - P[0][d], fmaf(a, P[1][d] - P[0][d], P[0][d]));
            const float dist = sqrtf(fmaf(D[0], D[0], fmaf(D[1], D[1], D[2] * D[2]))) * ((1.f / Q) * inv_r[i]);
            bad = bad || !(dist >= 1.f);
        }
        wrong += bad;
    }
    return wrong;
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("lens")
    src, lib = d / "l.cpp", d / "l.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).check
    fn.restype = ctypes.c_long

    def run(off, depth, ortho, inv_r, seed=0):
        rng = np.random.default_rng(seed)
        w = rng.random((60, 2))
        w = np.where(w.sum(1, keepdims=True) > 1, 1 - w, w)
        w = np.concatenate([w, [[0, 0], [1, 0], [0, 1], [.5, .5], [.5, 0], [0, .5], [1 / 3, 1 / 3]]])
        a = [np.ascontiguousarray(v, dtype=np.float32) for v in (off, depth, inv_r, w)]
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in a]
        found = ctypes.c_long(0)
        wrong = fn(p[0], p[1], ctypes.c_long(len(off)), int(ortho), p[2], p[3], ctypes.c_long(len(w)), ctypes.byref(found))
        return wrong, found.value

    return run


@pytest.mark.parametrize("ortho", [False, True])
@pytest.mark.parametrize("corners,centre,radius", [
    ([(0, 0, 0), (.75, 0, 0), (0, .75, 0)], (.25, .25, 0), 1.0),       # the offsets' sum is exactly 0
    ([(0, 0, 0), (3, 0, 0), (3, 3, 0)], (2, 1, 0), 10.0),
    ([(0, 0, 0), (3, 0, 0), (3, 3, 0)], (2, 1, 0), 0.25),              # (the corners outside of it)
    ([(1e19, 0, 0), (1e19, 1e18, 0), (1e19, 0, 1e18)], (0, 0, 0), 1e20),   # a squared sum that overflows
    ([(1e-20, 0, 0), (0, 1e-20, 0), (0, 0, 1e-20)], (0, 0, 0), 1e-14),     # one that underflows
    ([(-1e-16, 0, 0), (1e-16, 0, 0), (0, 0, 1e-30)], (0, 0, 0), 1e-12),
])
def test_lens_on_the_triangle(check, ortho, corners, centre, radius):
    off = np.asarray(corners, np.float32) - np.asarray(centre, np.float32)
    wrong, found = check(off[None], np.array([[1.0, 1.25, 1.5]]), ortho, np.array([1.0 / radius]))
    assert (wrong, found) == (0, 0)


@pytest.mark.parametrize("ortho", [False, True])
@pytest.mark.parametrize("scale", [1e-18, 1e-6, 1.0, 1e6, 1e18])
def test_never_outside_with_a_point_inside(check, ortho, scale):
    rng = np.random.default_rng(int(np.log10(scale)) + 100 + ortho)
    n = 40000
    size = 10.0 ** rng.uniform(-3, 1, (n, 1, 1))
    tri = np.where(rng.random((n, 1, 1)) < .5, rng.integers(-4, 5, (n, 3, 3)) / 4.0, rng.uniform(-1, 1, (n, 3, 3))) * size
    # the lens: anywhere, on a corner, on an edge, on the centroid, or just off the plane
    k = rng.integers(0, 5, n)
    centre = rng.uniform(-1, 1, (n, 3)) * size[:, 0]
    centre[k == 1] = tri[k == 1, 0]
    centre[k == 2] = tri[k == 2, :2].mean(1)
    centre[k == 3] = tri[k == 3].mean(1)
    centre[k == 4] += 2.0 * size[k == 4, 0]
    off = ((tri - centre[:, None]) * scale).astype(np.float32)
    # radii about the distances
    d = np.abs(off.astype(np.float64)).sum(2).min(1)
    radius = np.maximum(d * 10.0 ** rng.uniform(-1, 1, n), 2e-15)
    depth = 10.0 ** rng.uniform(-1, 1, (n, 1)) * rng.uniform(1, 3, (n, 3))
    wrong, found = check(off, depth, ortho, 1.0 / radius, seed=3)
    assert wrong == 0
    if 1e-15 < scale < 1e15:
        assert found > n // 20
