"""A frame whose memory cannot be had is refused, and the context goes on: each
allocation of a frame made to fail in turn (HEXFC_OPT_DEBUG_FAIL_ALLOC), frames
small and large after it are the same bit for bit as without; through every call
that draws."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

pytestmark = pytest.mark.gpu

STYLE = synth.Style(w_base=1.5, lod=2)
LENS = synth.lissajous_lens(5, 120)
SMALL = (synth.hex_grid(5, jitter=0.1, seed=2), synth.orbit_view(5, 120, 64, 48))
LARGE = (synth.hex_grid(12, jitter=0.1, seed=3), synth.orbit_view(5, 120, 656, 500))   # (more tiles than the small frame leaves room for)


@pytest.fixture(scope="module")
def hx():
    from paper_2009_06574_gb300 import hexfc
    hexfc.load()
    return hexfc


class Context:
    def __init__(self, hx, kind):
        self.hx, self.kind = hx, kind
        self.r = hx.Renderer(0)
        self.ids = [self.r.upload_mesh(m.verts, m.cells, m.cell_scalar, m.edge_level) for m, _ in (SMALL, LARGE)]
        self.r.set_lens(LENS)
        self.r.set_style(STYLE)
        if kind == "predicted":
            self.r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, 3)   # (capacities for any size after the first frame)

    def draw(self, which):
        """Status and image (None if refused) of the small (0) or large (1) frame."""
        view = (SMALL, LARGE)[which][1]
        out = torch.full((view.height, view.width, 4), -1.0, device="cuda")
        if self.kind == "batch":
            st = self.r.render_batch([(self.ids[which], view, LENS, STYLE, out)] * 2, check=False)[0]
        else:
            self.r.set_view(view)
            if self.kind == "host":
                img = np.empty((view.height, view.width, 4), np.float32)
                st = self.r.render_host(self.ids[which], img, check=False)
                return st, img if st == 0 else None
            st = self.r.render(self.ids[which], out, check=False)
            if st == 0:
                self.r.finish()
        torch.cuda.synchronize()
        return st, out.cpu().numpy() if st == 0 else None

    def fail(self, k):
        self.r.set_option(self.hx.HEXFC_OPT_DEBUG_FAIL_ALLOC, k)


@pytest.fixture(scope="module")
def images(hx):
    c = Context(hx, "render")
    imgs = [c.draw(w)[1] for w in (0, 1)]
    c.r.close()
    return imgs


@pytest.mark.parametrize("kind", ["render", "host", "batch", "predicted"])
@pytest.mark.parametrize("first", [True, False])
def test_each_allocation_of_a_frame(hx, images, kind, first):
    refused = 0
    for k in range(1, 60):
        c = Context(hx, kind)
        if not first:   # (buffers of the small frame are there)
            st, img = c.draw(0)
            assert st == 0
        c.fail(k)
        st, _ = c.draw(1)
        c.fail(0)
        if st != 0:
            assert st in (hx.HEXFC_ERR_OOM, hx.HEXFC_ERR_CUDA)
            refused += 1
        for which in (0, 1, 0):
            st, img = c.draw(which)
            assert st == 0
            np.testing.assert_array_equal(img, images[which])
        c.r.close()
    assert refused >= 15


def _allocations(hx, draw):
    """The most that a frame's k-th allocation can be for the frame to be refused."""
    most = 0
    for k in range(1, 50):
        if draw(k) != 0:
            most = k
    return most


def test_trim_keeps_the_pinned_copy(hx):
    def fresh(k):
        c = Context(hx, "render")
        c.fail(k)
        st, _ = c.draw(1)
        c.fail(0)
        c.r.close()
        return st

    def trimmed(k):
        c = Context(hx, "render")
        c.draw(1)
        c.r.trim()
        c.fail(k)
        st, _ = c.draw(1)
        c.fail(0)
        c.r.close()
        return st

    assert _allocations(hx, trimmed) == _allocations(hx, fresh) - 1


def test_each_allocation_of_the_network(hx):
    """Weights whose memory cannot be had are refused; set again, they train as ever."""
    def train(k):
        c = Context(hx, "render")
        c.draw(0)
        c.fail(k)
        try:
            c.r.capacity_reset(3)
            refused = False
        except hx.HexfcError as e:
            assert e.status == hx.HEXFC_ERR_OOM
            refused = True
        c.fail(0)
        if refused:
            with pytest.raises(hx.HexfcError) as e:
                c.r.capacity_train(1)
            assert e.value.status == hx.HEXFC_ERR_STATE
            c.r.capacity_reset(3)
        c.r.capacity_train(2)
        w = c.r.capacity_get_weights()
        c.r.close()
        return refused, w

    _, want = train(0)
    refused = 0
    for k in range(1, 10):
        r, w = train(k)
        refused += r
        np.testing.assert_array_equal(w, want)
    assert refused == 6


def test_each_allocation_of_an_upload(hx):
    """A mesh is refused only for its own memory: what is allocated beside the sorting of its faces and edges is asked for
    again without that, and the same frame is drawn."""
    mesh, view = synth.hex_grid(20, jitter=0.1, seed=7), synth.orbit_view(5, 120, 150, 110)
    view_img = []

    def upload(k):
        r = hx.Renderer(0)
        r.set_option(hx.HEXFC_OPT_DEBUG_FAIL_ALLOC, k)
        try:
            mid = r.upload_mesh(mesh.verts, mesh.cells, mesh.cell_scalar, mesh.edge_level)
        except hx.HexfcError as e:
            assert e.status == hx.HEXFC_ERR_OOM
            mid = None
        r.set_option(hx.HEXFC_OPT_DEBUG_FAIL_ALLOC, 0)
        if mid is not None:
            r.set_view(view)
            r.set_lens(LENS)
            r.set_style(STYLE)
            out = torch.empty((view.height, view.width, 4), device="cuda")
            r.render(mid, out)
            view_img.append((out.cpu().numpy(), r.mesh_info(mid)))
        torch.cuda.synchronize()
        r.close()
        return mid is not None

    assert upload(0)
    free = torch.cuda.mem_get_info()[0]
    # vertices, cells | scratch, cell edges, levels, corners, sides, boundary, given levels | five arrays of values
    assert [upload(k) for k in range(1, 17)] == [False] * 2 + [True] * 7 + [False] * 5 + [True] * 2
    assert torch.cuda.mem_get_info()[0] == free
    for img, info in view_img[1:]:
        assert info == view_img[0][1]
        np.testing.assert_array_equal(img, view_img[0][0])
