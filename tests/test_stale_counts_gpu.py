"""The tile counts and features that a frame leaves belong to that frame, drawn or
refused, and go with their buffers: after hexfc_trim, after tile buffers that
could not be had, after a refused frame of another size."""
import numpy as np
import pytest
import torch

from paper_2009_06574_gb300 import synth

from test_alloc_failures_gpu import Context
from test_wait_bound_gpu import column

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hx():
    from paper_2009_06574_gb300 import hexfc
    hexfc.load()
    return hexfc


def _train(hx, r):
    """Weights after two steps from the same start, None: no frame to train on."""
    r.capacity_reset(5)
    try:
        r.capacity_train(2)
    except hx.HexfcError as e:
        assert e.status == hx.HEXFC_ERR_STATE
        return None
    return r.capacity_get_weights()


def test_nothing_is_left_after_a_trim(hx):
    c = Context(hx, "render")
    _, img = c.draw(1)
    want = _train(hx, c.r)
    assert want is not None
    c.r.trim()
    assert _train(hx, c.r) is None
    c.r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, 1)
    st, again = c.draw(1)   # no previous counts: drawn exactly
    assert st == 0 and c.r.last_stats["predicted"] == 0
    np.testing.assert_array_equal(again, img)
    np.testing.assert_array_equal(_train(hx, c.r), want)   # (the camera has not moved, and no counts before)
    c.draw(1)
    assert c.r.last_stats["predicted"] == 1
    for mode in (2, 3):   # these need only some earlier frame's total
        c.r.trim()
        c.r.set_option(hx.HEXFC_OPT_PREDICTED_CAPACITY, mode)
        st, again = c.draw(1)
        assert st == 0 and c.r.last_stats["predicted"] == 1
        np.testing.assert_array_equal(again, img)
    c.r.close()


def test_buffers_that_cannot_be_had(hx):
    gone = 0
    for k in range(1, 40):
        c = Context(hx, "render")
        c.draw(0)
        want = _train(hx, c.r)
        c.fail(k)
        st, _ = c.draw(1)
        c.fail(0)
        got = _train(hx, c.r)
        if st != 0:
            if got is None:
                gone += 1
            else:   # the tile buffers were not touched
                np.testing.assert_array_equal(got, want)
        else:
            assert got is not None
        c.r.close()
    assert gone >= 8


def test_a_refused_frame_leaves_its_own(hx):
    verts, cells = column(hx.HEXFC_MAX_LIST + 8)
    flat = np.zeros(len(cells), np.float32)
    size = lambda w, h: synth.View(eye=(0, 0, 3), target=(0, 0, 0), ortho_half_h=1.0, znear=0.5, zfar=5.0, width=w, height=h)
    got = []
    for before in (True, False):
        c = Context(hx, "render")
        mid = c.r.upload_mesh(verts, cells, flat)
        if before:   # another frame, with the same camera
            c.r.set_view(size(200, 30))
            c.r.render(c.ids[1], torch.empty((30, 200, 4), device="cuda"))
        c.r.set_view(size(40, 56))
        assert c.r.render(mid, torch.empty((56, 40, 4), device="cuda"), check=False) == hx.HEXFC_ERR_OVERFLOW
        got.append(_train(hx, c.r))
        assert got[-1] is not None
        c.r.close()
    np.testing.assert_array_equal(got[0], got[1])
