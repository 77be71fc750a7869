"""Camera values that binary32 or int32 cannot hold reach the library as C would convert
them, and the library, not the packing, decides on them (host only)."""
import math
import os

import numpy as np
import pytest

from paper_2509_07021_gb300 import build, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene


def _query(cam):
    if not os.path.exists(build.library_path()):
        build.build()
    ds = DeviceScene.from_host(synth.make_scene(np.random.default_rng(0), 10, lobes=1), device="cpu")
    return sgsplat.sg_workspace_query(ds, [cam], 10)


def test_near_plane_past_binary32_culls_everything():
    cam = synth.make_camera(64, 48, 60.0)
    cam.near = 1e39
    assert math.isinf(sgsplat.camera_struct(cam).near_plane)
    assert _query(cam)["n_tiles"] == 12


@pytest.mark.parametrize("field,value", [("fx", 1e39), ("fy", -1e300), ("cx", 1e39), ("width", 2**32 - 5)])
def test_values_out_of_range_are_refused_by_the_library(field, value):
    cam = synth.make_camera(64, 48, 60.0)
    setattr(cam, field, value)
    with pytest.raises(sgsplat.SGError) as e:
        _query(cam)
    assert e.value.status == sgsplat.SG_ERR_INVALID_ARG


def test_packing_agrees_with_the_fields():
    cam = synth.make_camera(640, 479, 512.25, bg=(0.1, 0.2, 0.3))
    cam.fx, cam.cy = np.float32(500.1), "239.5"
    c = sgsplat.camera_struct(cam)
    assert (c.width, c.height) == (640, 479)
    assert c.fx == np.float32(500.1) and c.fy == 512.25 and c.cy == 239.5
    assert list(c.bg) == [np.float32(x) for x in (0.1, 0.2, 0.3)]
    assert list(c.viewmat) == np.asarray(cam.viewmat, np.float32).reshape(12).tolist()
