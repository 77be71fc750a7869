"""A blend shape that a caller names is the one that runs, also where it names the
defaults' values; only the defaults themselves follow the tile count."""
import numpy as np
import pytest
import torch

from paper_2509_07021_gb300 import render, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def test_named_default_shape_is_pinned():
    """One tile: with 8 pixels per thread one warp sums an entry's gradient, bit for bit the
    same in every run; with fewer, several warps' sums meet, and round otherwise."""
    rng = np.random.default_rng(4)
    ds = DeviceScene.from_host(synth.make_scene(rng, 400, lobes=1, means="cube", cube_side=1.4, masks="uniform"))
    cam = synth.make_camera(16, 16, 20.0)
    d = torch.randn(1, 3, 16, 16, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def grads():
        out = render.render_forward(ds, [cam])
        g = render.render_backward(ds, [cam], out, d)
        return torch.cat([v.flatten() for v in g.values()])
    old = sgsplat.sg_get_tuning()
    try:
        sgsplat.sg_set_tuning()
        assert sgsplat.sg_get_tuning()["auto_shapes"] == 3
        by_tiles = grads()
        sgsplat.sg_set_tuning(4, 8, 1, 1, fwd_batch=64, bwd_batch=64)
        pinned = grads()
        sgsplat.sg_set_tuning()
        sgsplat.sg_set_tuning(4, 8, 1, 1, fwd_batch=0, bwd_batch=0)
        named = grads()
        assert torch.equal(named, pinned) and not torch.equal(by_tiles, pinned)
        # a look at the tuning and back changes nothing, nor does another field
        sgsplat.sg_set_tuning()
        sgsplat.sg_set_tuning(**sgsplat.sg_get_tuning())
        sgsplat.sg_set_tuning(sort_wait_polls=0)
        assert sgsplat.sg_get_tuning()["auto_shapes"] == 3
        sgsplat.sg_set_tuning(bwd_pixels_per_thread=8)
        assert sgsplat.sg_get_tuning()["auto_shapes"] == 1 and torch.equal(grads(), pinned)
    finally:
        sgsplat.sg_set_tuning(**old)
