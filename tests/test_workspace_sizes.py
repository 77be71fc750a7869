"""What a workspace costs (host only): ws_fixed_bytes is what a forward leaves per entry
and per tile plus its tables, without a share for pairs that the caller did not ask
for, and ws_fixed_bytes + ws_per_pair_bytes x pairs holds that many pairs."""
import ctypes
import os

import numpy as np
import pytest

from paper_2509_07021_gb300 import build, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

VIEWS = {"1x1": [(1, 1)], "many_1x1": [(1, 1)] * 128, "tiny": [(128, 128)], "square": [(800, 800)],
         "1080p": [(1920, 1080)], "two_1080p": [(1920, 1080)] * 2, "ring": [(1600, 1066)] * 16,
         "4k": [(3840, 2160)], "uneven": [(3840, 2160)] + [(1, 1)] * 100, "radix": [(5120, 2900)],
         "four_passes": [(80_000, 80_000)]}
CAPS = (0, 1, 65, 1000, 10_000, 100_000, 2**20, 2**20 + 1, 2_000_000, 5_700_000, 12 * 2**20, 12 * 2**20 + 1,
        2**24, 2**24 + 1, 32 * 2**20 + 1, 252_000_000)


def _query(views, n, cap):
    if not os.path.exists(build.library_path()):
        build.build()
    ds = DeviceScene.from_host(synth.make_scene(np.random.default_rng(0), 10, lobes=1), device="cpu")
    s = ds.struct()
    s.n = n   # sizes only: no pointer is read
    cams = sgsplat.camera_array([synth.make_camera(w, h, 100.0) for w, h in views])
    out = sgsplat.sg_sizes()
    assert sgsplat.lib().sg_workspace_query(ctypes.byref(s), cams, len(views), cap, ctypes.byref(out)) == sgsplat.SG_OK
    return out.as_dict()


@pytest.mark.parametrize("name", VIEWS)
@pytest.mark.parametrize("n", [0, 10_000, 1_000_000])
def test_fixed_part_and_per_pair_share_hold_the_pairs(name, n):
    last = 0
    for cap in CAPS:
        q = _query(VIEWS[name], n, cap)
        assert q["ws_bytes"] <= q["ws_fixed_bytes"] + q["ws_per_pair_bytes"] * cap, cap
        assert q["ws_bytes"] >= last, cap   # a larger workspace never holds fewer pairs
        last = q["ws_bytes"]


@pytest.mark.parametrize("name", VIEWS)
@pytest.mark.parametrize("n", [0, 10_000, 1_000_000])
def test_fixed_part_is_what_the_forward_leaves(name, n):
    q = _query(VIEWS[name], n, 0)
    # an entry: 48-byte record, tiles touched, rectangle and clamp bits (61), the depth sort's keys
    # and values twice (16), its look-back flags (4 x 256 words, with the groups', for 3072
    # keys and pass) and the chunk cutter's; a tile: range, place in the order and a share
    # of the scan's words (12.25); the tables, and rounding
    flags = 1024 * (17 / 16) * (5 if len(VIEWS[name]) > 1 else 4) / 3072
    most = (77 + flags + 1 / 32) * q["n_entries"] + 12.25 * q["n_tiles"] + 72 * 1024
    assert q["ws_fixed_bytes"] <= most
