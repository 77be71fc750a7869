"""One batched training step run again on the same inputs: lists, images and positions
repeat bit for bit; gradients may move only by the order in which an entry's sums over
tiles meet, which has to stay inside what a gradient may be off by at all."""
import numpy as np
import pytest
import torch

from paper_2509_07021_gb300 import render, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("views", [
    [(160, 120), (75, 201)],                 # few tiles: one pixel per thread, eight warps a tile
    [(1408, 1040), (640, 480)],              # the backward's 8-pixel form
], ids=lambda v: "+".join(f"{w}x{h}" for w, h in v))
def test_repeated_batched_steps_agree(views):
    rng = np.random.default_rng(2024)
    scenes = [DeviceScene.from_host(synth.make_scene(rng, n, lobes=synth.LOBE_MIX, means="cube", cube_side=1.6,
                                                     masks="uniform")) for n in (5000, 1700)]
    cams = [synth.make_camera(w, h, 0.9 * w) for w, h in views] * 2
    br = render.BatchedRenderer(scenes, cams, [0] * len(views) + [1] * len(views))
    loss = render.l1_loss_grad(br, torch.rand(br.img.numel(), device="cuda"))
    runs = []
    for _ in range(4):
        br.step(loss)
        torch.cuda.synchronize()
        runs.append(([t.clone() for t in (br.img, br.T_final, br.last)],
                     [{k: v.double().clone() for k, v in g.items()} for g in br.grads]))
    for outs, grads in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs, runs[0][0]))
        for g, ref in zip(grads, runs[0][1]):
            for k, v in ref.items():
                # a gradient is held to 1e-3 (relative L2) of the oracle's: two of them to twice that
                assert float((g[k] - v).norm()) <= 2e-3 * float(v.norm()), k
