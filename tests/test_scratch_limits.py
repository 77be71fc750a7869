"""The least backward scratch (host only): the batch table, the counters and nine sums per
entry are enough, in the caller's scratch and in the static one. The room that the query
adds for the backward's own tile order (5633 to 16384 tiles) may be missing."""
import ctypes
import os

import numpy as np
import pytest

from paper_2509_07021_gb300 import build, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

P = ctypes.c_void_p
TABLE = 27 * 1024   # batch table and counters, rounded up


def _call(w, h, n):
    if not os.path.exists(build.library_path()):
        build.build()
    ds = DeviceScene.from_host(synth.make_scene(np.random.default_rng(0), 10, lobes=1), device="cpu")
    s = ds.struct()
    s.n = n   # sizes only: no pointer is read
    return s, sgsplat.camera_array([synth.make_camera(w, h, 100.0)]), sgsplat.grads_struct({})


@pytest.mark.parametrize("w,h", [(640, 480), (1392, 1040), (1920, 1080), (2048, 2048)])
def test_static_scratch_takes_as_many_entries_at_every_tile_count(w, h):
    n = (sgsplat.SG_NOALLOC_SCRATCH_BYTES - TABLE) // 36
    s, cams, g = _call(w, h, n)
    st = sgsplat.lib().sg_render_backward_noalloc(ctypes.byref(s), cams, 1, P(256), 1 << 10, P(256), P(256), P(256),
                                                  ctypes.byref(g), None)
    # past the scratch's size, the call is refused for the forward workspace of 1 KB
    assert st == sgsplat.SG_ERR_WORKSPACE and "fixed part" in sgsplat.sg_last_error()


@pytest.mark.parametrize("w,h", [(640, 480), (1392, 1040), (1920, 1080), (2048, 2048)])
def test_scratch_without_room_for_a_tile_order_is_enough(w, h):
    n = 5000
    s, cams, g = _call(w, h, n)

    def status(size):
        st = sgsplat.lib().sg_render_backward(ctypes.byref(s), cams, 1, P(256), 1 << 10, P(256), P(256), P(256), P(256),
                                              size, ctypes.byref(g), None)
        assert st == sgsplat.SG_ERR_WORKSPACE
        return sgsplat.sg_last_error()
    assert "fixed part" in status(36 * n + TABLE)
    assert "backward scratch" in status(36 * n)
