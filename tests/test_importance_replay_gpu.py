"""Importance updates captured into a CUDA graph: a replay, also after a plain
update, is what the next frame reads; the lists of a frame drawn before stay its
own; and no update allocates."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

pytestmark = pytest.mark.gpu

VIEW, LENS = synth.orbit_view(7, 120, 150, 110), synth.lissajous_lens(7, 120)
STYLE = synth.Style(w_base=1.5, lod=2)


def _renderer(hx, mesh, scalar):
    r = hx.Renderer(0)
    mid = r.upload_mesh(mesh.verts, mesh.cells, scalar, mesh.edge_level)
    r.set_view(VIEW)
    r.set_lens(LENS)
    r.set_style(STYLE)
    return r, mid


def _draw(r, mid):
    out = torch.empty((VIEW.height, VIEW.width, 4), device="cuda")
    r.render(mid, out)
    return out.cpu().numpy()


def _fresh(hx, mesh, scalar):
    r, mid = _renderer(hx, mesh, scalar)
    img = _draw(r, mid)
    r.close()
    return img


@pytest.mark.parametrize("render_first", [False, True])
def test_replay_after_a_plain_update(render_first):
    from paper_2009_06574_gb300 import hexfc as hx
    mesh = synth.hex_grid(9, jitter=0.12, warp_amp=0.3, seed=11)
    rng = np.random.default_rng(2)
    vals = [rng.random(mesh.n_cells).astype(np.float32) for _ in range(4)]
    r, mid = _renderer(hx, mesh, vals[0])
    if render_first:
        np.testing.assert_array_equal(_draw(r, mid), _fresh(hx, mesh, vals[0]))
    held = torch.from_numpy(vals[1]).cuda()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.set_cell_importance(mid, held)
    g.replay()
    np.testing.assert_array_equal(_draw(r, mid), _fresh(hx, mesh, vals[1]))
    px, py = (v.ravel().astype(np.int32) for v in np.meshgrid(np.arange(20, 130, 9), np.arange(10, 100, 9)))
    for k in (2, 3):
        r.set_cell_importance(mid, torch.from_numpy(vals[0]).cuda())
        drawn = _draw(r, mid)
        np.testing.assert_array_equal(drawn, _fresh(hx, mesh, vals[0]))
        lists = r.debug_pixels(px, py)
        assert lists["counts"].sum() > 1000
        held.copy_(torch.from_numpy(vals[k]))
        g.replay()
        torch.cuda.synchronize()
        kept = r.debug_pixels(px, py)   # of the frame drawn before the replay
        for name in ("counts", "keys", "rgba"):
            np.testing.assert_array_equal(kept[name], lists[name])
        np.testing.assert_array_equal(_draw(r, mid), _fresh(hx, mesh, vals[k]))
    r.close()


def test_updates_allocate_nothing():
    from paper_2009_06574_gb300 import hexfc as hx
    mesh = synth.hex_grid(40, seed=1)   # 12.6 MB of face records
    r, mid = _renderer(hx, mesh, mesh.cell_scalar)
    val = torch.from_numpy(mesh.cell_scalar).cuda()
    _draw(r, mid)
    r.set_cell_importance(mid, val)
    torch.cuda.synchronize()
    _draw(r, mid)
    r2, mid2 = _renderer(hx, mesh, mesh.cell_scalar)
    before = _draw(r2, mid2)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    r2.set_cell_importance(mid2, val)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    np.testing.assert_array_equal(_draw(r2, mid2), before)
    r.close()
    r2.close()
