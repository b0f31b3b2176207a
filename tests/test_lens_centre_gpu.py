"""The sphere lens exactly on a triangle's centroid: the triangle in the middle of
the focus is in focus, against the oracle, in both projections."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

from parity import check_sampled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fovy", [0.0, 50.0])
@pytest.mark.parametrize("radius", [0.5, 2.0, 20.0])
def test_lens_on_a_centroid(fovy, radius):
    from paper_2009_06574_gb300 import hexfc as hx
    mesh = synth.hex_grid(2, seed=4)
    mesh.verts = np.rint(mesh.verts * 6.0).astype(np.float32)   # corners at -3, 0, 3
    # the front faces' first triangles: corners (-3, -3, 3), (0, -3, 3), (0, 0, 3), so the centroid is (-1, -2, 3)
    lens = synth.Lens(mode=synth.LENS_SPHERE, center=(-1.0, -2.0, 3.0), radius=radius)
    view = synth.View(eye=(0.5, 0.25, 9.0), target=(0.0, 0.0, 0.0), fovy_deg=fovy, ortho_half_h=4.0, znear=0.5, zfar=30.0,
                      width=88, height=72)
    style = synth.Style(w_base=1.5, lod=1, delta=0.3)
    r = hx.Renderer(0)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    r.set_view(view)
    r.set_lens(lens)
    r.set_style(style)
    out = torch.empty((view.height, view.width, 4), device="cuda")
    r.render(mid, out)
    st = check_sampled(r, mesh, view, lens, style, out, n=3000, seed=1)
    assert st["fragments"] > 1000
    r.close()
