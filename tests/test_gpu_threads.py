"""Host threads that render frames of different sizes at the same time, each on its own
stream, workspace and outputs: no call may make another's fail or change its result.
(The binning's shared memory follows the frame: 4 bytes per tile of the largest view.)"""
import threading

import numpy as np
import pytest
import torch

from paper_2509_07021_gb300 import sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def test_threads_with_frames_of_different_sizes():
    rng = np.random.default_rng(31)
    ds = DeviceScene.from_host(synth.make_scene(rng, 3000, lobes=1, means="cube", cube_side=1.4, masks="uniform"))
    # rows of 2, 33, 40 and 200 KB; capacities on both sides of the sizes at which the
    # scan's shared memory changes
    frames = [((400, 300), 900_000), ((1920, 1080), 2_000_000), ((1600, 1600), 900_000), ((3584, 3584), 4_000_000)]
    jobs = []
    for (w, h), cap in frames:
        cams = [synth.make_camera(w, h, 0.9 * w)]
        q = sgsplat.sg_workspace_query(ds, cams, cap)
        bufs = [torch.empty(q["ws_bytes"], dtype=torch.uint8, device="cuda"), torch.empty(3, h, w, device="cuda"),
                torch.empty(h, w, device="cuda"), torch.empty(h, w, dtype=torch.int32, device="cuda")]
        sgsplat.sg_render_forward(ds, cams, *bufs)
        torch.cuda.synchronize()
        jobs.append((cams, bufs, bufs[1].clone()))
    wrong = []

    def work(cams, bufs, want):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(150):
                st, _ = sgsplat.sg_render_forward(ds, cams, *bufs, raise_on_error=False)
                if st != sgsplat.SG_OK:
                    wrong.append((cams[0].width, st, sgsplat.sg_last_error()))
                    return
            if not torch.equal(bufs[1], want):
                wrong.append((cams[0].width, "image"))
        stream.synchronize()

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
