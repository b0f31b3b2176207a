"""The binning's paths at their edges: frames of more tiles than the one-block
scan takes, triangles over many tiles and over at most 2x2, tile lists for each
size of the depth order's blocks and past the largest, meshes whose counts end
inside a warp. The image does not depend on how the triangles were binned, so
each is compared bit for bit with another way of drawing the same pixels."""
import numpy as np
import pytest

from paper_2009_06574_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_06574_gb300 import hexfc
    hexfc.load()
    return hexfc


def _renderer(hx, mesh, view, lens, style):
    r = hx.Renderer(0)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    r.set_view(view)
    r.set_lens(lens)
    r.set_style(style)
    return r, mid


@pytest.mark.parametrize("w,h", [(2048, 2048), (2064, 2048)])   # 16384 tiles (the scan's most) and 129 x 128
def test_many_tiles_equal_their_parts(hx, w, h):
    mesh = synth.hex_grid(5, jitter=0.1, warp_amp=0.2, seed=3)   # triangles over hundreds of tiles
    view = synth.orbit_view(11, 120, w, h, radius=1.5)
    r, mid = _renderer(hx, mesh, view, synth.lissajous_lens(11, 120), synth.Style(lod=1))
    full = torch.zeros((h, w, 4), device="cuda")
    r.render(mid, full)
    for (x0, y0, cw, ch) in [(0, 0, w, 700), (0, 700, w, h - 700), (801, 333, 517, 411)]:
        r.set_subrect(x0, y0, cw, ch)
        part = torch.full((ch, cw, 4), -1.0, device="cuda")
        r.render(mid, part)
        assert torch.equal(part, full[y0:y0 + ch, x0:x0 + cw])
    r.close()


# lists of a few entries, of 2 * 256 * 8 and more in few tiles, of more than 1024 * 16, of more than 768 on
# average over more than 1024 tiles
@pytest.mark.parametrize("n,w,h", [(1, 40, 40), (3, 33, 17), (16, 32, 32), (26, 32, 32), (48, 656, 480), (20, 300, 200)])
def test_depth_order_sizes(hx, n, w, h):
    mesh = synth.hex_grid(n, jitter=0.1, warp_amp=0.2, seed=5)
    view = synth.orbit_view(20, 120, w, h)
    r, mid = _renderer(hx, mesh, view, synth.lissajous_lens(20, 120), synth.Style(w_base=1.0))
    imgs = []
    for buckets in (2048, 256, 4096, 0):   # 0: no depth order, every list sorted by its keys
        r.set_option(hx.HEXFC_OPT_DEPTH_BUCKETS, buckets)
        out = torch.full((h, w, 4), -1.0, device="cuda")
        r.render(mid, out)
        imgs.append(out)
    for img in imgs[1:]:
        assert torch.equal(img, imgs[0])
    r.close()


@pytest.mark.parametrize("budget", [0, 6 << 20])   # with room for the binning's places, and without
def test_binning_with_and_without_places(hx, budget):
    mesh = synth.hex_grid(20, jitter=0.1, warp_amp=0.2, seed=7)
    view = synth.orbit_view(31, 120, 96, 80, radius=2.4)
    r, mid = _renderer(hx, mesh, view, synth.Lens(mode=0, center=(48.0, 40.0, 0.0), radius=20.0), synth.Style())
    ref = torch.zeros((80, 96, 4), device="cuda")
    r.render(mid, ref)
    r2 = hx.Renderer(0, frag_budget_bytes=budget)
    mid2 = r2.share_mesh(r, mid)
    r2.set_view(view)
    r2.set_lens(synth.Lens(mode=0, center=(48.0, 40.0, 0.0), radius=20.0))
    r2.set_style(synth.Style())
    out = torch.zeros((80, 96, 4), device="cuda")
    r2.render(mid2, out)
    assert torch.equal(out, ref)
    if budget:
        assert r2.frame_memory() <= budget
    r.close()
    r2.close()


def test_lists_survive_an_importance_update(hx):
    """hexfc_debug_pixels after importance updates gives the lists of the frame as it was drawn."""
    mesh = synth.hex_grid(6, jitter=0.1, warp_amp=0.2, seed=9)
    view = synth.orbit_view(5, 120, 64, 48, radius=1.6)
    r, mid = _renderer(hx, mesh, view, synth.lissajous_lens(5, 120), synth.Style(tf_hi=1.0))
    out = torch.zeros((48, 64, 4), device="cuda")
    r.render(mid, out)
    px, py = np.arange(20, 40, dtype=np.int32), np.full(20, 24, np.int32)
    a = r.debug_pixels(px, py)
    for k in range(3):
        r.set_cell_importance(mid, torch.full((len(mesh.cells),), 0.1 * k, device="cuda"))
        b = r.debug_pixels(px, py)
        np.testing.assert_array_equal(a["keys"], b["keys"])
        np.testing.assert_array_equal(a["rgba"], b["rgba"])
    again = torch.zeros_like(out)
    r.render(mid, again)
    assert not torch.equal(again, out)
    assert not np.array_equal(r.debug_pixels(px, py)["rgba"], a["rgba"])
    r.close()


# one block a tile's count, and clusters of 2 to 8 of them; lists that end inside a chunk, a run of chunks, a tile
@pytest.mark.parametrize("n,w,h", [(2, 32, 32), (14, 16, 16), (26, 47, 35), (40, 320, 180), (30, 640, 250)])
def test_counts_with_and_without_clusters(hx, n, w, h):
    mesh = synth.hex_grid(n, jitter=0.1, warp_amp=0.2, seed=11)
    view, lens, style = synth.orbit_view(9, 120, w, h), synth.lissajous_lens(9, 120), synth.Style(w_base=1.0)
    r, mid = _renderer(hx, mesh, view, lens, style)
    one = torch.full((h, w, 4), -1.0, device="cuda")
    r.render(mid, one)
    outs = [torch.full((h, w, 4), -1.0, device="cuda") for _ in range(2)]
    st, per, stats = r.render_batch([(mid, view, lens, style, o) for o in outs])   # one block a tile
    assert st == 0 and all(p == 0 for p in per)
    for o, s in zip(outs, stats):
        assert torch.equal(o, one)
        for k in ("fragments", "bin_entries", "max_list", "long_lists", "covered_pixels"):
            assert s[k] == r.last_stats[k], k
    r.close()


# meshes drawn so small that triangles lie between samples: set aside when binned, where places are kept
@pytest.mark.parametrize("n,w,h,radius", [(24, 33, 21, 2.0), (40, 64, 48, 2.6), (40, 16, 16, 8.0), (12, 1, 1, 2.0),
                                            (4, 16, 16, 40.0), (3, 40, 16, 25.0), (2, 33, 17, 8.0)])
def test_triangles_between_samples(hx, n, w, h, radius):
    mesh = synth.hex_grid(n, jitter=0.1, warp_amp=0.2, seed=13)
    view, lens, style = synth.orbit_view(17, 120, w, h, radius=radius), synth.lissajous_lens(17, 120), synth.Style()
    imgs, stats, weights = [], [], []
    budget = 0
    for kind in ("places", "budget", "noalloc"):
        r = hx.Renderer(0, frag_budget_bytes=budget if kind == "budget" else 0)
        mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
        r.set_view(view)
        r.set_lens(lens)
        r.set_style(style)
        out = torch.full((h, w, 4), -1.0, device="cuda")
        (r.render_noalloc if kind == "noalloc" else r.render)(mid, out)
        imgs.append(out)
        stats.append({k: r.last_stats[k] for k in ("fragments", "bin_entries", "max_list", "covered_pixels")})
        if kind != "noalloc":   # the network's features of the frame
            r.capacity_reset(5)
            r.capacity_train(4, lr=1e-2)
            weights.append(r.capacity_get_weights())
            budget = r.frame_memory() - 3 * n ** 3 * 16   # too little for the places (72 bytes a face)
        r.close()
    for img, st in zip(imgs[1:], stats[1:]):
        assert torch.equal(img, imgs[0])
        assert st == stats[0]
    np.testing.assert_allclose(weights[1], weights[0], rtol=1e-5, atol=1e-7)


def test_frames_whose_bins_outgrow_their_room(hx):
    """Launches go ahead with the last frame's room for bins: views that need less, more and far more of
    it, and meshes of other sizes in between, give what a fresh context gives."""
    meshes = [synth.hex_grid(n, jitter=0.1, warp_amp=0.2, seed=n) for n in (6, 20)]
    r = hx.Renderer(0)
    mids = [r.upload_mesh(m.verts, m.cells, m.cell_scalar, m.edge_level) for m in meshes]
    for k, (w, h, radius) in [(0, (64, 48, 3.0)), (0, (512, 400, 1.2)), (1, (64, 48, 3.0)), (1, (640, 480, 1.2)), (0, (33, 21, 2.0)),
                              (1, (900, 700, 1.1))]:
        view, lens, style = synth.orbit_view(7, 120, w, h, radius=radius), synth.lissajous_lens(7, 120), synth.Style(sil_alpha=0.5)
        imgs, stats = [], []
        for q, mid in ((r, mids[k]), (hx.Renderer(0), 0)):
            if q is not r:
                mid = q.upload_mesh(meshes[k].verts, meshes[k].cells, meshes[k].cell_scalar, meshes[k].edge_level)
            q.set_view(view)
            q.set_lens(lens)
            q.set_style(style)
            out = torch.full((h, w, 4), -1.0, device="cuda")
            q.render(mid, out)
            stats.append({n: q.last_stats[n] for n in ("fragments", "bin_entries", "max_list", "covered_pixels")})
            imgs.append(out)
            if q is not r:
                if k == 0:   # (fits the fixed scratch array)
                    imgs.append(torch.full((h, w, 4), -1.0, device="cuda"))
                    q.render_noalloc(mid, imgs[-1])
                q.close()
        assert stats[0] == stats[1]
        for img in imgs[1:]:
            assert torch.equal(img, imgs[0])
    r.close()


def test_refused_frames_leave_their_output_alone(hx):
    """A frame refused for its budget, silhouettes and all, after one of another view that was drawn."""
    mesh = synth.hex_grid(16, jitter=0.1, warp_amp=0.2, seed=15)
    r = hx.Renderer(0, frag_budget_bytes=24 << 20)
    mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
    r.set_lens(synth.lissajous_lens(3, 120))
    r.set_style(synth.Style(sil_alpha=0.7))
    small = torch.full((48, 64, 4), -1.0, device="cuda")
    r.set_view(synth.orbit_view(3, 120, 64, 48))
    r.render(mid, small)
    large = torch.full((480, 640, 4), -1.0, device="cuda")
    r.set_view(synth.orbit_view(3, 120, 640, 480))
    assert r.render(mid, large, check=False) != 0
    torch.cuda.synchronize()
    assert (large == -1.0).all()
    r.set_view(synth.orbit_view(3, 120, 64, 48))
    again = torch.full((48, 64, 4), -1.0, device="cuda")
    r.render(mid, again)
    assert torch.equal(again, small)
    r.close()
