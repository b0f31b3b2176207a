"""Faces and edges found on the device against those built on the host (which an
upload falls back to when the device has no memory to sort them in): the same
numbers, the same fragments at every pixel, over cells with repeated corners,
repeated cells, faces of three cells, crossed faces and any numbering."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

from test_mesh_tables_gpu import _mesh

pytestmark = pytest.mark.gpu

# corners of a hexahedron drawn together: wedges, a pyramid, a tetrahedron, a quad, an edge, opposite corners, a point
REPEATS = [[0, 1, 2, 3, 4, 5, 5, 4], [0, 1, 1, 0, 4, 5, 6, 7], [0, 1, 2, 3, 4, 4, 4, 4], [0, 1, 2, 2, 4, 4, 4, 4],
           [0, 1, 2, 3, 0, 1, 2, 3], [0, 1, 1, 0, 0, 1, 1, 0], [0, 1, 0, 3, 4, 5, 6, 7], [0, 0, 0, 0, 0, 0, 0, 0]]


def _lists(mesh, host):
    from paper_2009_06574_gb300 import hexfc as hx
    r = hx.Renderer(0)
    if host:   # the third allocation is what the device would sort in
        r.set_option(hx.HEXFC_OPT_DEBUG_FAIL_ALLOC, 3)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    r.set_option(hx.HEXFC_OPT_DEBUG_FAIL_ALLOC, 0)
    view = synth.orbit_view(3, 120, 72, 54, radius=1.5)
    r.set_view(view)
    r.set_lens(synth.lissajous_lens(3, 120))
    r.set_style(synth.Style(lod=1, w_base=1.5))
    out = torch.empty((view.height, view.width, 4), device="cuda")
    r.render(mid, out)
    yy, xx = np.meshgrid(np.arange(view.height), np.arange(view.width), indexing="ij")
    g = r.debug_pixels(xx.ravel(), yy.ravel())
    info = r.mesh_info(mid)
    r.close()
    return info, g["counts"], g["keys"], g["rgba"], out.cpu().numpy()


@pytest.mark.parametrize("form", ["repeated corners", "repeated cells", "three cells a face", "crossed faces", "no levels"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_device_and_host_agree(form, seed):
    g = synth.hex_grid(5, jitter=0.1, warp_amp=0.2, seed=seed)
    rng = np.random.default_rng(seed)
    new = rng.permutation(len(g.verts))
    verts = np.empty_like(g.verts)
    verts[new] = g.verts
    cells = new[g.cells]
    some = rng.choice(len(cells), 40, replace=False)
    if form == "repeated corners":
        for k, c in enumerate(some):
            cells[c] = cells[c][REPEATS[k % len(REPEATS)]]
    elif form == "repeated cells":
        cells = np.concatenate([cells, cells[some], cells[some[:7]]])
    elif form == "three cells a face":   # a face of the cell, its other corners anywhere
        extra = cells[some].copy()
        extra[:, 4:] = rng.integers(0, len(verts), (len(some), 4))
        cells = np.concatenate([cells, extra])
    elif form == "crossed faces":
        cells[some] = cells[some][:, [0, 2, 1, 3, 4, 5, 6, 7]]
    mesh = _mesh(verts, cells[rng.permutation(len(cells))], seed=seed)
    if form == "no levels":
        mesh.edge_level = None
    device, host = _lists(mesh, False), _lists(mesh, True)
    assert device[0] == host[0] and host[1].sum() > 1000
    for a, b in zip(device[1:], host[1:]):
        np.testing.assert_array_equal(a, b)
