"""Unique faces and edges found on the device, and the meshes it leaves to the
host: against the oracle's, through the fragments of every pixel. Vertex numbers,
cell order and cell orientation in any order; a vertex whose faces fill a bucket
up to the device's limit and past it; cells that list a common face's corners in
different orders."""
import types

import numpy as np
import pytest

from paper_2009_06574_gb300 import synth

from parity import hex_rotations
from test_gpu_parity import hx, render_both  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mesh(verts, cells, level=None, seed=0):
    cells = np.ascontiguousarray(cells, np.int32)
    rng = np.random.default_rng(seed)
    level = rng.integers(0, 3, (len(cells), 12)).astype(np.uint8) if level is None else level
    return types.SimpleNamespace(verts=np.ascontiguousarray(verts, np.float32), cells=cells,
                                 cell_scalar=rng.random(len(cells)).astype(np.float32), edge_level=level)


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_any_numbering(hx, seed):  # noqa: F811
    g = synth.hex_grid(5, jitter=0.1, warp_amp=0.2, seed=seed)
    rng = np.random.default_rng(seed)
    new = rng.permutation(len(g.verts))
    verts = np.empty_like(g.verts)
    verts[new] = g.verts
    rot = np.array([s for s, _ in hex_rotations()])
    cells = new[g.cells][np.arange(len(g.cells))[:, None], rot[rng.integers(0, len(rot), len(g.cells))]]
    cells = cells[rng.permutation(len(cells))]
    st, _ = render_both(hx, _mesh(verts, cells, seed=seed), synth.orbit_view(9, 120, 70, 50),
                        synth.lissajous_lens(9, 120), synth.Style(lod=1, w_base=1.5))
    assert st["fragments"] > 1000


@pytest.mark.parametrize("n", [1, 341, 342, 400])   # 3 faces and 3 edges a cell in vertex 0's buckets (at most 1024)
def test_one_vertex_of_many_cells(hx, n):  # noqa: F811
    rng = np.random.default_rng(n)
    corner = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0], [0, 0, 1], [1, 0, 1], [1, 1, 1], [0, 1, 1]], float)
    verts, cells = [np.zeros(3)], []
    for i in range(n):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        q[:, 0] *= np.sign(np.linalg.det(q))
        verts += list(corner[1:] @ q.T * 0.12)
        cells.append([0] + [1 + 7 * i + k for k in range(7)])
    st, _ = render_both(hx, _mesh(np.array(verts), cells, seed=n), synth.orbit_view(3, 120, 60, 44, radius=1.6),
                        synth.lissajous_lens(3, 120), synth.Style(lod=1, w_base=1.5))
    assert st["fragments"] > 0


def test_repeated_and_crossed_corners(hx):  # noqa: F811
    verts = [[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0], [0, 0, 1], [1, 0, 1], [1, 1, 1], [0, 1, 1], [0, 0, 2], [1, 0, 2]]
    verts = (np.array(verts) - [0.5, 0.5, 1.0]) * 0.5
    cells = [[0, 1, 2, 3, 4, 5, 6, 7], [4, 5, 6, 7, 8, 9, 9, 8],   # a wedge
             [4, 6, 5, 7, 8, 9, 9, 8]]                              # the common face crossed
    r = hx.Renderer(0)
    m = _mesh(verts, cells)
    mid = r.upload_mesh(m.verts, m.cells, m.cell_scalar, m.edge_level)
    out = torch.zeros((48, 64, 4), device="cuda")
    r.set_view(synth.orbit_view(3, 120, 64, 48))
    r.set_lens(synth.lissajous_lens(3, 120))
    r.set_style(synth.Style(lod=0))
    r.render(mid, out)
    assert r.last_stats["fragments"] > 100 and torch.isfinite(out).all()
    r.close()
