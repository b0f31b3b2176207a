"""The drawing pass's waits are bounded one by one, not over a tile: a library
built with a bound of about an eighth of a millisecond draws a tile that takes
several times that, in the form whose finished warps go on staging (a batch), and
reports nothing."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2009_06574_gb300 import synth

pytestmark = pytest.mark.gpu

TESTS = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(TESTS)
LAYERS = 8000


def column(layers=LAYERS):
    """2 x 2 x layers cells along the view direction, wider than the frame: every
    pixel's list has a fragment of every layer."""
    x, z = np.array([-2.0, 0.0, 2.0]), np.linspace(-1.0, 1.0, layers + 1)
    zz, yy, xx = np.meshgrid(z, x, x, indexing="ij")
    verts = np.stack([xx.ravel(), yy.ravel(), zz.ravel()], axis=1).astype(np.float32)
    k, j, i = np.meshgrid(np.arange(layers), np.arange(2), np.arange(2), indexing="ij")
    at = lambda a, b, c: ((i + a) + 3 * ((j + b) + 3 * (k + c))).ravel()
    corners = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]
    return verts, np.stack([at(*c) for c in corners], axis=1).astype(np.int32)


def draw_twice():
    import torch
    from paper_2009_06574_gb300 import hexfc as hx
    verts, cells = column()
    # half of the tile's warps lie outside of the frame and are finished at once; no pixel becomes opaque
    view = synth.View(eye=(0, 0, 3), target=(0, 0, 0), ortho_half_h=1.0, znear=0.5, zfar=5.0, width=8, height=16)
    lens = synth.Lens(mode=synth.LENS_SCREEN, center=(-1e6, 0.0, 0.0), radius=1.0)
    style = synth.plain(synth.Style(lod=100, delta=2.0, alpha_min=1e-5, alpha_max=1e-4))
    r = hx.Renderer(0)
    r.set_option(hx.HEXFC_OPT_DEPTH_BUCKETS, 4096)   # two layers a bucket: no pixel meets its fragments out of order
    r.set_option(hx.HEXFC_OPT_COMPOSITE_WINDOW, 8)   # and is left to the pass after
    mid = r.upload_mesh(verts, cells, np.zeros(len(cells), np.float32))
    out = torch.zeros((16, 8, 4), device="cuda")
    for _ in range(2):   # a frame's drawing pass is reported by the next call on its buffers
        _, status, stats = r.render_batch([(mid, view, lens, style, out)], check=False)
        torch.cuda.synchronize()
        assert status == [0], hx.status_string(status[0])
        assert stats[0]["max_list"] > LAYERS
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    r.render_batch([(mid, view, lens, style, out)])
    end.record()
    torch.cuda.synchronize()
    img = out.cpu().numpy()
    r.close()
    return img, start.elapsed_time(end)


CHILD = """
import sys
sys.path.insert(0, {root!r})
sys.path.insert(0, {tests!r})
import numpy as np
from paper_2009_06574_gb300 import build
build.build(extra=["-DHEXFC_WAIT_CYCLES=(1ll<<18)"])
import test_wait_bound_gpu as t
img, ms = t.draw_twice()
assert ms > 0.4, ms   # several times the bound
np.save({out!r}, img)
"""


def test_a_tile_may_take_longer_than_a_wait(tmp_path):
    ref, _ = draw_twice()
    out = str(tmp_path / "img.npy")
    env = dict(os.environ, HEXFC_BUILD_DIR=str(tmp_path / "build"))
    p = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, tests=TESTS, out=out)], env=env, capture_output=True,
                       text=True, timeout=1200)
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
    np.testing.assert_array_equal(np.load(out), ref)
