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
        r.render(mid, outs[3], stream=b)
        assert r.completed_stats(jumped)["redrawn"] == 1
        assert r.finish()["redrawn"] == 0
        torch.cuda.synchronize()
        for o, k in zip(outs, (0, 0, 1, 1)):
            np.testing.assert_array_equal(o.cpu().numpy(), want[k])
        r.close()


@pytest.mark.parametrize("mode", [0, 1, 3])
def test_frames_in_turn_on_two_streams(hx, mode):
    """Back to back, of two meshes and sizes, without a wait in between: a frame waits for the last one's kernels, whose
    buffers it writes."""
    meshes = [synth.hex_grid(24, jitter=0.1, warp_amp=0.3, seed=6), synth.hex_grid(7, jitter=0.1, seed=2)]
    views = [synth.orbit_view(3, 120, 640, 360, radius=1.4), synth.orbit_view(9, 120, 200, 150, radius=1.4)]
    want = [_exact(hx, m, v) for m, v in zip(meshes, views)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    r, big = _context(hx, meshes[0])
    small = r.upload_mesh(meshes[1].verts, meshes[1].cells, meshes[1].cell_scalar, meshes[1].edge_level)
    r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, mode)
    outs = [[torch.empty((v.height, v.width, 4), device="cuda") for v in views] for _ in range(12)]
    torch.cuda.synchronize()
    for pair in outs:
        for k in (0, 1):
            r.set_view(views[k])
            r.render((big, small)[k], pair[k], stream=streams[k])
    r.finish()
    torch.cuda.synchronize()
    for pair in outs:
        for k in (0, 1):
            np.testing.assert_array_equal(pair[k].cpu().numpy(), want[k])
    r.close()
