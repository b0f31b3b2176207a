"""The covered runs of a tile's rows (csrc/row_span.h) against the edge functions
evaluated in 64 bits at every sample, compiled for the host: triangles of every
size around the limit of the 32-bit values, edges through samples, parallel to
the rows and all but so, slivers, clipped tiles."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_06574_gb300", "csrc")

SOURCE = r"""
#include "row_span.h"
using namespace hexfc;
// tris: n x (x0 x1 x2 y0 y1 y2); returns the number of wrong samples
extern "C" long check(const int32_t* tris, long n, int cols, int rows, int tw, long* covered, long* large)
{
    long wrong = 0;
    *covered = *large = 0;
    for (long i = 0; i < n; ++i) {
        const int32_t *x = tris + 6 * i, *y = x + 3;
        int4 e[3];
        const uint32_t box = stage_edges(x, y, cols, rows, e, 1);
        uint32_t got[33] = {0};
        for (int r = 0; r < 2 * box_pairs(box); ++r) {
            int lo = box_lx0(box), hi = box_lx1(box);
            if (box & kBoxBig) { const int2 s = row_span_big(e, 1, tw, r, lo, hi); lo = s.x; hi = s.y; }
            else row_span(e, r, lo, hi);
            if (lo <= hi) got[box_ly0(box) + r] = ((2u << (hi - lo)) - 1u) << lo;
        }
        *large += (box & kBoxBig) != 0;
        int o[3] = {0, 1, 2};
        int64_t area = (int64_t)(x[1] - x[0]) * (y[2] - y[0]) - (int64_t)(y[1] - y[0]) * (x[2] - x[0]);
        if (area < 0) { o[1] = 2; o[2] = 1; }
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c) {
                bool in = area != 0;
                for (int k = 0; k < 3; ++k) {
                    const int a = o[(k + 1) % 3], b = o[(k + 2) % 3];
                    const int64_t dx = x[b] - x[a], dy = y[b] - y[a];
                    const int64_t v = dx * (256 * r + 128 - y[a]) - dy * (256 * c + 128 - x[a]);
                    in = in && (v > 0 || (v == 0 && (dy < 0 || (dy == 0 && dx > 0))));
                }
                *covered += in;
                wrong += in != (bool)((got[r] >> c) & 1u);
            }
    }
    return wrong;
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, lib = d / "r.cpp", d / "r.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).check
    fn.restype = ctypes.c_long
    return fn


@pytest.mark.parametrize("tw,cols,rows", [(16, 16, 16), (16, 7, 10), (8, 8, 32), (32, 32, 8), (32, 31, 5)])
@pytest.mark.parametrize("reach", [300, 3000, 16384, 16500, 60000, 1 << 23])
def test_runs_equal_the_edge_functions(check, tw, cols, rows, reach):
    rng = np.random.default_rng(reach + tw)
    n = 60000
    t = rng.integers(-reach, reach + 1, (n, 6), dtype=np.int64)
    t[:, :3] += 128 * tw
    near = rng.random((n, 6)) < 0.4                      # corners in the tile
    t = np.where(near, rng.integers(-256, 256 * tw + 256, (n, 6)), t)
    snap = rng.random(n) < 0.3                           # corners on sample centres
    t[snap] = (t[snap] // 256) * 256 + 128
    flat = rng.random(n) < 0.15                          # edges parallel to the rows, or all but so
    t[flat, 4] = t[flat, 3] + rng.integers(-1, 2, flat.sum())
    edge = rng.random(n) < 0.2                           # corners at the limit of the 32-bit values
    t[edge] = np.clip(t[edge], -16384, 16384)
    t = np.ascontiguousarray(np.clip(t, -(1 << 23), 1 << 23), dtype=np.int32)
    covered, large = ctypes.c_long(0), ctypes.c_long(0)
    wrong = check(t.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(n), cols, rows, tw, ctypes.byref(covered),
                  ctypes.byref(large))
    assert wrong == 0
    assert covered.value > 0
    assert (large.value > 0) == (reach + 128 * tw > 16384)
