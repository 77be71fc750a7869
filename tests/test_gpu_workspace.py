"""Forwards in the smallest workspaces and on the smallest frames. The binning's count
matrix lives in the image until the blend writes it, or, where the frame is too small,
in the workspace."""
import numpy as np
import pytest
import torch

from paper_2509_07021_gb300 import render, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

from test_gpu_parity import run_parity

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n,views", [(1000, [(1920, 1080)]), (20_000, [(800, 800)]), (3000, [(640, 480), (1, 1), (1600, 1066)]),
                                     (3000, [(2048, 1552)])], ids=lambda v: str(v))
def test_a_workspace_of_just_the_pairs(n, views):
    """fixed + per pair x pairs is enough, and the pairs' number is what decides: the
    outputs and gradients are those of a roomy workspace."""
    rng = np.random.default_rng(12)
    ds = DeviceScene.from_host(synth.make_scene(rng, n, lobes=2, means="cube", cube_side=1.4, masks="uniform"))
    cams = [synth.make_camera(w, h, 0.9 * w) for w, h in views]
    ref = render.render_forward(ds, cams)
    d = torch.ones_like(ref.img)
    want = render.render_backward(ds, cams, ref, d)["c0"]
    pairs = ref.sizes["n_pairs"]
    q = sgsplat.sg_workspace_query(ds, cams, pairs)
    for size in (q["ws_bytes"], q["ws_fixed_bytes"] + q["ws_per_pair_bytes"] * pairs):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        img, T, last = torch.empty_like(ref.img), torch.empty_like(ref.T_final), torch.empty_like(ref.last)
        st, sizes = sgsplat.sg_render_forward(ds, cams, ws, img, T, last, raise_on_error=False)
        assert st == sgsplat.SG_OK and sizes["n_pairs"] == pairs <= sizes["pair_capacity"]
        assert torch.equal(img, ref.img) and torch.equal(T, ref.T_final) and torch.equal(last, ref.last)
        got = render.render_backward(ds, cams, render.ForwardOut(img, T, last, ws, sizes), d)["c0"]
        # a positive upstream gradient: no cancellation, only the order of the tiles' sums
        torch.testing.assert_close(got, want, rtol=2e-4, atol=1e-6 * float(want.abs().max()))
    # one pair fewer is refused, and says what is needed
    small = sgsplat.sg_workspace_query(ds, cams, pairs - 256)
    ws = torch.empty(small["ws_bytes"], dtype=torch.uint8, device="cuda")
    st, sizes = sgsplat.sg_render_forward(ds, cams, ws, img, T, last, raise_on_error=False)
    assert st == sgsplat.SG_ERR_CAPACITY and sizes["n_pairs"] == pairs


@pytest.mark.parametrize("views", [[(1, 1)], [(1, 2)], [(2, 2)], [(1, 1)] * 5, [(33, 1)], [(1, 130)],
                                   [(96, 64), (1, 1), (3, 3)]], ids=lambda v: "+".join(f"{w}x{h}" for w, h in v))
def test_smallest_frames(views):
    rng = np.random.default_rng(9)
    scene = synth.make_scene(rng, 700, lobes=1, means="cube", cube_side=1.2, masks="uniform")
    run_parity(scene, [synth.make_camera(w, h, 60.0) for w, h in views], seed=2)


def test_backward_without_room_for_its_tile_order():
    rng = np.random.default_rng(13)
    ds = DeviceScene.from_host(synth.make_scene(rng, 3000, lobes=1, means="cube", cube_side=1.4, masks="uniform"))
    cams = [synth.make_camera(1920, 1080, 1700.0)]
    out = render.render_forward(ds, cams)
    d = torch.ones_like(out.img)
    want = render.render_backward(ds, cams, out, d)["c0"]
    grads = render.alloc_grads(ds)
    bwd = torch.empty(out.sizes["bwd_ws_bytes"] - 4 * out.sizes["n_tiles"], dtype=torch.uint8, device="cuda")
    sgsplat.sg_render_backward(ds, cams, out.ws, out.T_final, out.last, d, bwd, grads)
    torch.testing.assert_close(grads["c0"], want, rtol=2e-4, atol=1e-6 * float(want.abs().max()))
