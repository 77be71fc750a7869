"""The chunked binning at the sizes where it can go wrong: one tile, ragged and
empty views between full ones, more than 12288 tiles (sorted tile ids kept), an
entry that covers a whole frame, views without any pair, and a view past the
chunks' tile limit (radix passes). The lists are compared with the oracle's
decisions and the library's binning rule bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_07021_gb300 import render, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

from parity_util import GpuView, check_decisions

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

AWAY = synth.look_at((0.0, 0.0, -9.0), (0.0, 0.0, -20.0))   # sees nothing

CASES = {
    # name: (Gaussians, views (width, height, fx, viewmat))
    "one_tile": (500, [(16, 16, 20.0, None)]),
    "ragged": (4000, [(129, 97, 110.0, None), (33, 47, 30.0, None), (17, 300, 60.0, None)]),
    "empty_views": (3000, [(64, 48, 60.0, AWAY), (80, 50, 70.0, None), (40, 40, 45.0, AWAY), (48, 80, 60.0, None),
                           (16, 16, 20.0, AWAY)]),
    "all_empty": (300, [(64, 48, 60.0, AWAY), (80, 50, 70.0, AWAY)]),
    "kept_tile_ids": (2500, [(1936, 1104, 1500.0, None), (1040, 800, 900.0, None), (700, 300, 400.0, None)]),
    "past_the_chunk_limit": (400, [(3856, 3856, 3000.0, None), (64, 64, 60.0, None)]),
}


@pytest.mark.parametrize("name", CASES)
def test_lists_match_the_binning_rule(name):
    n, views = CASES[name]
    rng = np.random.default_rng(990)
    scene = synth.make_scene(rng, n, lobes=1, means="cube", cube_side=1.4, masks="uniform")
    scene.scales[:, 0] = 2.0      # covers whole frames
    scene.opac[0] = scene.gmask[0] = 1.0
    cams = [synth.make_camera(w, h, f, viewmat=vm) for w, h, f, vm in views]
    ds = DeviceScene.from_host(scene)
    out = render.render_forward(ds, cams)
    lay = sgsplat.sg_workspace_layout(ds, cams, out.ws.numel())
    assert (lay["pair_tile"] == sgsplat.NO_OFFSET) == (out.sizes["n_tiles"] <= 12288)
    gv = GpuView.plain(ds, cams, out)
    checks = []
    for v, cam in enumerate(cams):
        res, _ = oracle.render(scene, [cam], tile_sel=[np.zeros(cam.n_tiles, bool)])
        checks.append((v, scene, res[0]))
    check_decisions(gv, cams, checks)
    assert gv.K == int(gv.tt.sum()) and (gv.K == 0) == (name == "all_empty")
    # a second forward on the same workspace leaves the same lists
    img, T, last = torch.empty_like(out.img), torch.empty_like(out.T_final), torch.empty_like(out.last)
    st, sizes = sgsplat.sg_render_forward(ds, cams, out.ws, img, T, last, raise_on_error=False)
    assert st == sgsplat.SG_OK and sizes["n_pairs"] == gv.K
    again = GpuView.plain(ds, cams, out)
    assert np.array_equal(again.pair_entry, gv.pair_entry) and np.array_equal(again.ranges, gv.ranges)
    assert torch.equal(img, out.img) and torch.equal(T, out.T_final) and torch.equal(last, out.last)


@pytest.mark.parametrize("n,views", [(1, 1), (2048, 1), (2049, 1), (2048, 2), (2049, 2), (8192, 1), (4096, 2), (8193, 1),
                                     (4097, 2), (60_000, 1), (30_000, 3)])
def test_depth_order_at_the_kernels_edges(n, views):
    """One block sorts up to 8192 entries (2, 4 or 8 keys a thread), the digit
    passes the larger ones; with several views the order is by view first. Every
    tile list must hold its entries by (depth bits, entry), each entry in as
    many lists as it reaches tiles. Equal depths are planted."""
    rng = np.random.default_rng(n + views)
    scene = synth.make_scene(rng, n, lobes=0, means="cube", cube_side=1.4, masks="uniform")
    scene.means[2, n // 3:n // 2] = 4.0
    cams = [synth.make_camera(200 + 16 * v, 120, 150.0) for v in range(views)]
    ds = DeviceScene.from_host(scene)
    out = render.render_forward(ds, cams)
    gv = GpuView.plain(ds, cams, out)
    assert gv.K == int(gv.tt.sum())
    np.testing.assert_array_equal(np.bincount(gv.pair_entry, minlength=n * views), gv.tt)
    depth = gv.rec[gv.pair_entry, 11].view(np.uint32).astype(np.int64)
    key = (gv.pair_tile * 2**32 + depth) * 1.0   # exact below 2^53: tiles here are few
    same = np.diff(gv.pair_tile) == 0
    assert np.all(np.diff(gv.pair_tile) >= 0) and np.all(np.diff(key)[same] >= 0)
    tie = same & (np.diff(depth) == 0)
    assert np.all(np.diff(gv.pair_entry)[tie] > 0)


@pytest.mark.parametrize("w,h", [(640, 640), (1024, 640), (1040, 640), (960, 960), (976, 960), (1408, 1024), (1424, 1024),
                                 (1920, 1024), (1936, 1024)])
def test_default_shape_at_its_tile_counts(w, h):
    """The tile count picks the default blends' pixels per thread; on both sides of
    every line the outputs are those of a pinned shape (bit exact forward, the
    backward's atomics in another order)."""
    rng = np.random.default_rng(5)
    scene = synth.make_scene(rng, 3000, lobes=1, means="cube", cube_side=3.0, masks="uniform")
    cam = synth.make_camera(w, h, 1.2 * w)
    ds = DeviceScene.from_host(scene)
    d = torch.randn(1, 3, h, w, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    out = render.render_forward(ds, [cam])
    g = render.render_backward(ds, [cam], out, d)
    old = sgsplat.sg_get_tuning()
    sgsplat.sg_set_tuning(4, 8, 1, 1, fwd_batch=64, bwd_batch=64)
    try:
        ref = render.render_forward(ds, [cam])
        gr = render.render_backward(ds, [cam], ref, d)
    finally:
        sgsplat.sg_set_tuning(**old)
    assert torch.equal(out.img, ref.img) and torch.equal(out.T_final, ref.T_final) and torch.equal(out.last, ref.last)
    for k in gr:
        assert torch.linalg.norm(g[k] - gr[k]) <= 2e-5 * torch.linalg.norm(gr[k]) + 1e-12, k


@pytest.mark.parametrize("views,line", [([(3856, 2160)], 12 << 20), ([(2560, 2048), (300, 200)], 32 << 20)],
                         ids=["one_chunk_per_sm", "two_chunks_per_sm"])
def test_large_frames_at_the_pairs_where_the_route_changes(views, line):
    """Past so much room for pairs a large frame takes the radix passes: on both sides of
    the line the lists, the images and (a positive upstream gradient) the sums agree."""
    rng = np.random.default_rng(8)
    ds = DeviceScene.from_host(synth.make_scene(rng, 3000, lobes=1, means="cube", cube_side=1.4, masks="uniform"))
    cams = [synth.make_camera(w, h, 0.9 * w) for w, h in views]
    got = []
    for cap in (line, line + 4096):
        q = sgsplat.sg_workspace_query(ds, cams, cap)
        ref = render._alloc_outputs(cams, torch.device("cuda"))
        ws = torch.empty(q["ws_bytes"], dtype=torch.uint8, device="cuda")
        st, sizes = sgsplat.sg_render_forward(ds, cams, ws, *ref, raise_on_error=False)
        assert st == sgsplat.SG_OK and 0 < sizes["n_pairs"] <= cap <= sizes["pair_capacity"]
        out = render.ForwardOut(*ref, ws, sizes)
        gv = GpuView.plain(ds, cams, out)
        c0 = render.render_backward(ds, cams, out, torch.ones_like(out.img))["c0"]
        got.append((gv.pair_entry, gv.ranges, out, c0))
    a, b = got
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert torch.equal(a[2].img, b[2].img) and torch.equal(a[2].last, b[2].last)
    torch.testing.assert_close(a[3], b[3], rtol=2e-4, atol=1e-6 * float(b[3].abs().max()))
