"""hexfc_debug_pixels after a refused frame answers STATE, also when that call
had to draw the frame before it again: the lists' inputs are the refused frame's
by then."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

from test_wait_bound_gpu import column

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("redraw", [False, True])
def test_no_lists_after_a_refused_frame(redraw):
    from paper_2009_06574_gb300 import hexfc as hx
    mesh = synth.hex_grid(10, jitter=0.1, warp_amp=0.3, seed=6)
    r = hx.Renderer(0)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    verts, cells = column(hx.HEXFC_MAX_LIST + 8)
    long = r.upload_mesh(verts, cells, np.zeros(len(cells), np.float32))
    lens = synth.lissajous_lens(0, 120)
    r.set_lens(lens)
    out = torch.empty((120, 160, 4), device="cuda")
    near = synth.orbit_view(0, 120, 160, 120, radius=1.3)
    r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, 1)
    for view in [synth.orbit_view(0, 120, 160, 120, radius=4.0)] * 2 + ([near] if redraw else []):   # the pool runs out
        r.set_view(view)
        r.render(mid, out)
    last = r.last_stats["frame"]
    assert r.last_stats["pending"] == 1
    r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, 0)
    r.set_view(synth.View(eye=(0, 0, 3), target=(0, 0, 0), ortho_half_h=1.0, znear=0.5, zfar=5.0, width=8, height=16))
    assert r.render(long, torch.empty((16, 8, 4), device="cuda"), check=False) == hx.HEXFC_ERR_OVERFLOW
    assert r.completed_stats(last)["redrawn"] == int(redraw)
    with pytest.raises(hx.HexfcError) as e:
        r.debug_pixels([3], [4])
    assert e.value.status == hx.HEXFC_ERR_STATE
    r.set_view(near)   # and the context goes on
    r.render(mid, out)
    assert r.debug_pixels([80], [60])["counts"][0] > 0
    r.close()
