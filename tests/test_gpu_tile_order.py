"""The backward's own tile order (by walk length) at the edges of the tile counts
that get one, against the one-block-per-tile form, which has no order: every
tile must be walked exactly once, also by a second backward of one forward and
after the workspace held another forward's order."""
import numpy as np
import pytest
import torch

from paper_2509_07021_gb300 import render, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("views", [
    [(1408, 1024)],               # 5632 tiles: the forward's order
    [(688, 2096)],                # 5633: its own
    [(1393, 1030), (40, 17)],     # two views, ragged edges
    [(2048, 2048)],               # 16384: its own
    [(2320, 1808)],               # 16385: the forward's
], ids=lambda v: "+".join(f"{w}x{h}" for w, h in v))
@pytest.mark.parametrize("fwd_persistent", [1, 0])
def test_every_tile_is_walked_once(views, fwd_persistent):
    rng = np.random.default_rng(77)
    scene = synth.make_scene(rng, 3000, lobes=1, means="cube", cube_side=1.4, masks="uniform")
    cams = [synth.make_camera(w, h, 0.9 * w) for w, h in views]
    ds = DeviceScene.from_host(scene)
    # a positive upstream gradient: the colour sums have no cancellation, so their
    # order changes them by at most (tiles reached) x 2^-24 in relative terms
    def grads(out):
        g = render.render_backward(ds, cams, out, torch.ones_like(out.img))
        return g["c0"].clone()
    old = sgsplat.sg_get_tuning()
    try:
        sgsplat.sg_set_tuning(fwd_persistent=0, bwd_persistent=0)
        ref = render.render_forward(ds, cams)
        want = grads(ref)
        assert float(want.abs().max()) > 0
        sgsplat.sg_set_tuning(fwd_persistent=fwd_persistent, bwd_persistent=1)
        out = render.render_forward(ds, cams)
        assert torch.equal(out.img, ref.img) and torch.equal(out.last, ref.last)
        for _ in range(2):
            torch.testing.assert_close(grads(out), want, rtol=2e-4, atol=1e-6 * float(want.abs().max()))
        # an importance forward files no walk lengths: the backward takes its list order
        scored = render.render_forward(ds, cams, importance=torch.empty(ds.n, device="cuda"))
        torch.testing.assert_close(grads(scored), want, rtol=2e-4, atol=1e-6 * float(want.abs().max()))
        img = torch.empty_like(out.img)
        sgsplat.sg_render_forward(ds, cams, out.ws, img, out.T_final, out.last)
        torch.testing.assert_close(grads(out), want, rtol=2e-4, atol=1e-6 * float(want.abs().max()))
    finally:
        sgsplat.sg_set_tuning(**old)
