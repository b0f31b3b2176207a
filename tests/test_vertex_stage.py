"""The vertex stage from pairs of floats (csrc/vertex_stage.h) against its
definition in double precision, compiled for the host: whatever the pairs claim
to decide equals the double evaluation bit for bit, over cameras of every kind
(scales from 1e-4 to 1e4, far offsets, wide and long lenses, both projections,
drawn rectangles) and vertices on and off the lattices that put window positions
exactly on rounding boundaries."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_06574_gb300", "csrc")

SOURCE = r"""
#include "vertex_stage.h"
using namespace hexfc;
extern "C" long check(const float* v, long n, const double* c, int ortho, int ox, int oy, long* undecided)
{
    CamParams cam{};
    for (int d = 0; d < 3; ++d) { cam.eye[d] = c[d]; cam.R[d] = c[3 + d]; cam.U[d] = c[6 + d]; cam.F[d] = c[9 + d]; }
    cam.focal = c[12]; cam.scale = c[13]; cam.cx = c[14]; cam.cy = c[15];
    cam.znear = c[16]; cam.zfar = c[17]; cam.zf_over = c[18];
    cam.ortho = ortho; cam.ox = ox; cam.oy = oy;
    const CamPairs p = cam_pairs(cam);
    long wrong = 0;
    *undecided = 0;
    for (long i = 0; i < n; ++i) {
        ProjVertex a, b;
        vertex_double(v[3 * i], v[3 * i + 1], v[3 * i + 2], cam, a);
        if (!p.usable || !vertex_pairs(v[3 * i], v[3 * i + 1], v[3 * i + 2], p, cam, b)) { ++*undecided; continue; }
        wrong += a.x != b.x || a.y != b.y || a.z != b.z || a.valid != b.valid || float_bits(a.depth) != float_bits(b.depth);
    }
    return wrong;
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("vertex")
    src, lib = d / "v.cpp", d / "v.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).check
    fn.restype = ctypes.c_long
    return fn


def _camera(eye, target, fovy, half, n, f, W, H):
    eye, F = np.asarray(eye, float), np.asarray(target, float) - eye
    F = F / np.linalg.norm(F)
    R = np.cross(F, (0.0, 1.0, 0.0))
    R /= np.linalg.norm(R)
    ortho = not fovy > 0
    focal, scale = (0.0, 0.5 * H / half) if ortho else (0.5 * H / np.tan(np.radians(fovy) / 2), 0.0)
    c = np.concatenate([eye, R, np.cross(R, F), F, [focal, scale, 0.5 * W, 0.5 * H, n, f, f / (f - n)]])
    return np.ascontiguousarray(c), int(ortho)


def _run(check, verts, cam, ortho, ox=0, oy=0):
    v = np.ascontiguousarray(verts, np.float32)
    und = ctypes.c_long(0)
    wrong = check(v.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(v)), cam.ctypes.data_as(ctypes.c_void_p), ortho, ox,
                  oy, ctypes.byref(und))
    return wrong, und.value / len(v)


@pytest.mark.parametrize("ortho", [False, True])
@pytest.mark.parametrize("log_scale", [-4, 0, 4])
def test_pairs_equal_double(check, ortho, log_scale):
    rng = np.random.default_rng(10 * log_scale + ortho + 100)
    undecided = []
    for k in range(12):
        s = 10.0 ** log_scale
        off = rng.normal(size=3) * s * 10.0 ** rng.uniform(-2, 2)
        v = rng.uniform(-0.5, 0.5, (40000, 3)) * s + off
        if k % 3 == 0:   # a lattice
            v = np.round(v / s * 64) / 64 * s
        W, H = int(rng.integers(1, 16385)), int(rng.integers(1, 16385))
        cam, o = _camera(off + rng.normal(size=3) * s * rng.uniform(0.1, 3), off, 0 if ortho else rng.uniform(0.5, 170),
                         s * rng.uniform(0.3, 2), s * 10.0 ** rng.uniform(-4, -0.3), s * 10.0 ** rng.uniform(0.3, 3), W, H)
        wrong, u = _run(check, v, cam, o, int(rng.integers(0, W)), int(rng.integers(0, H)))
        assert wrong == 0
        undecided.append(u)
    assert np.median(undecided) < 0.01   # the pairs decide nearly all


def test_rounding_boundaries_and_limits(check):
    """Vertices exactly on half steps of the window grid, on the near and far
    planes, at the guard band, at the eye and beyond the floats' precision."""
    cam, o = _camera((0, 0, 3), (0, 0, 0), 0, 0.5, 1.0, 5.0, 256, 256)
    half = np.arange(-4096, 4096) / (2 * 256 * 256.0)
    v = np.stack([half, -half, np.zeros_like(half)], axis=1)
    assert _run(check, v, cam, o)[0] == 0
    cam, o = _camera((0, 0, 3), (0, 0, 0), 60, 1, 1.0, 5.0, 1000, 700)
    z = np.array([2.0, np.nextafter(np.float32(2), 0), np.nextafter(np.float32(2), 3), -2.0, 3.0, 4.0, 2.999999, 1e30, -1e30,
                  1e-40, 0.0])
    v = np.array([(x, y, w) for w in z for x in (0.0, 1e-7, 0.3, 27.0567, 1e20) for y in (0.0, -0.3, 27.0567)])
    assert _run(check, v, cam, o)[0] == 0
    far = cam.copy()
    far[12] = 1e18   # constants beyond the pairs' range: everything in double
    assert _run(check, v, far, o) == (0, 1.0)
