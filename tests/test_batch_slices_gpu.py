"""Batches of one renderer whose frames need other launch shapes from batch to
batch (the count's blocks a tile change with the length of the lists): each the
same as the frame alone, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launch", [0, 1])
def test_lists_of_any_length_in_turn(launch):
    from paper_2009_06574_gb300 import hexfc as hx
    meshes = [synth.hex_grid(n, jitter=0.1, seed=n) for n in (3, 40, 12, 24)]
    lens, style = synth.lissajous_lens(5, 120), synth.Style(w_base=1.5, lod=2)
    views = [synth.orbit_view(f, 120, 64, 48, radius=1.6) for f in (3, 50)]
    r, alone = hx.Renderer(0), hx.Renderer(0)
    r.set_option(hx.HEXFC_OPT_BATCH_LAUNCH, launch)
    ids = [(r.upload_mesh(m.verts, m.cells, m.cell_scalar, m.edge_level),
            alone.upload_mesh(m.verts, m.cells, m.cell_scalar, m.edge_level)) for m in meshes]
    alone.set_lens(lens)
    alone.set_style(style)
    want = {}
    for k, (_, a) in enumerate(ids):
        for v, view in enumerate(views):
            out = torch.empty((48, 64, 4), device="cuda")
            alone.set_view(view)
            alone.render(a, out)
            want[k, v] = out.cpu().numpy()
    for k in (0, 1, 0, 2, 3, 1, 3, 0, 1):
        outs = [torch.empty((48, 64, 4), device="cuda") for _ in views]
        _, status, _ = r.render_batch([(ids[k][0], view, lens, style, o) for view, o in zip(views, outs)])
        torch.cuda.synchronize()
        assert status == [0, 0]
        for v, o in enumerate(outs):
            np.testing.assert_array_equal(o.cpu().numpy(), want[k, v])
    r.close()
    alone.close()
