"""One context's frames on more than one stream."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

pytestmark = pytest.mark.gpu

LENS = synth.lissajous_lens(0, 120)
STYLE = synth.Style(w_base=1.5, lod=2)
VIEWS = [synth.orbit_view(0, 120, 160, 120, radius=4.0), synth.orbit_view(0, 120, 160, 120, radius=1.3)]


@pytest.fixture(scope="module")
def hx():
    from paper_2009_06574_gb300 import hexfc
    hexfc.load()
    return hexfc


def _context(hx, mesh):
    r = hx.Renderer(0)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    r.set_lens(LENS)
    r.set_style(STYLE)
    return r, mid


def _exact(hx, mesh, view):
    r, mid = _context(hx, mesh)
    r.set_view(view)
    out = torch.empty((view.height, view.width, 4), device="cuda")
    r.render(mid, out)
    torch.cuda.synchronize()
    r.close()
    return out.cpu().numpy()


def test_a_frame_on_another_stream_finds_the_pool_run_out(hx):
    """The frame before, on its own stream, is drawn again by that call: its error bits are cleared where that reads them."""
    mesh = synth.hex_grid(10, jitter=0.1, warp_amp=0.3, seed=6)
    want = [_exact(hx, mesh, v) for v in VIEWS]
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(20):
        r, mid = _context(hx, mesh)
        r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, 1)
        outs = [torch.empty((120, 160, 4), device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        for o, k in zip(outs[:3], (0, 0, 1)):
            r.set_view(VIEWS[k])
            r.render(mid, o, stream=a)
        jumped = r.last_stats["frame"]
        torch.cuda.synchronize()
        r.render(mid, outs[3], stream=b)
        assert r.completed_stats(jumped)["redrawn"] == 1
        assert r.finish()["redrawn"] == 0
        torch.cuda.synchronize()
        for o, k in zip(outs, (0, 0, 1, 1)):
            np.testing.assert_array_equal(o.cpu().numpy(), want[k])
        r.close()
