"""Workloads of the SG-splatting rasterizer, for timing and for comparing outputs.

Every case is what a program that renders, trains or prunes a scene of Gaussians with
spherical-Gaussian lobes asks of the library, through its public entry points:

* `forward`     one call of render.render_forward (a viewer, an evaluation render)
* `autograd`    render.rasterize and the gradients of every parameter (a training step)
* `pair`        render.render_forward + render.render_backward (a training step that manages
                its own gradients; the SH colour model is trained this way)
* `batched`     render.BatchedRenderer: forward, loss gradient, backward over many scenes x views
* `graph`       the same step captured once and replayed as one CUDA graph
* `importance`  render.render_forward with the per-Gaussian importance score (a pruning pass)
* `admm`        the opacity and sharpness proximal steps and their penalty gradients
* `post`        sgsplat.sg_postprocess (thresholds, colour compensation, compaction)

A case holds plain values: `sizes` lists the scenes' Gaussian counts, `res` the views every
scene is seen from, `means` / `lobes` / `masks` / `storage` / `colour` the distributions and
the storage form. Scenes follow the distributions of the repository's seeded workloads
(paper_2509_07021_gb300/synth.py); they are drawn on the GPU so that making them is quick.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_07021_gb300 import render, sgsplat, synth
from paper_2509_07021_gb300.sgsplat import DeviceScene

LOBE_P = (0.20, 0.30, 0.25, 0.15, 0.10)      # 0..4 lobes per Gaussian
FIELDS = ("means", "scales", "quats", "opac", "gmask", "c0", "axis", "sharp", "amp", "lmask")
HALF = ("means", "scales", "quats", "opac", "axis", "amp", "sharp")   # binary16 in the f16 forms


def _case(name, api, sizes, res="", means="clusters", lobes="mix", masks="uniform", storage="f32",
          colour="sg"):
    return {"name": name, "api": api, "sizes": sizes, "res": res, "means": means, "lobes": lobes,
            "masks": masks, "storage": storage, "colour": colour}


def listed():
    return [
        # the smallest call: a thumbnail of a toy scene, where latency and launches are all there is
        _case("view_tiny", "forward", "1000", "128x128", means="cube", lobes="3", masks="ones"),
        # an early training step of a small object at a ragged image size
        _case("step_small", "autograd", "20011", "401x299"),
        # a training loop over a small scene with the step captured as a CUDA graph
        _case("graph_50k", "graph", "50000", "800x800"),
        # an interactive viewer on a pruned scene kept in binary16 (sharpness in bfloat16)
        _case("view_f16", "forward", "600000", "1600x1066", storage="f16_bf16s", masks="ones"),
        # training steps at full resolution on a mid-sized and on the benchmark's scene
        _case("step_500k", "autograd", "500000", "1920x1080"),
        _case("step_1m", "autograd", "1000000", "1920x1080"),
        # the 3DGS colour (degree-3 SH), which the paper compares against
        _case("sh3_step", "pair", "300000", "1280x720", colour="sh3"),
        # several scenes of uneven size, each seen from four cameras, in one call
        _case("batch_6x4", "batched", "50000,120000,300000,600000,1200000,2000000",
              "800x800,1280x720,1600x1066,1920x1080"),
        # the largest scene: 6M packed Gaussians, most of them pruned, a ring of 16 views
        _case("batch_16v_6m", "batched", "6000000", ",".join(["1600x1066"] * 16), means="packed",
              lobes="4", masks="pruned"),
        # a pruning pass: importance over four views of the benchmark's scene
        _case("importance_1m", "importance", "1000000", ",".join(["1280x720"] * 4)),
        # the ADMM iteration between training steps, and the final compaction
        _case("admm_1m", "admm", "1000003"),
        _case("post_1m", "post", "1000003", masks="admm"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def res():
        w = log(97, 1920)
        return f"{w}x{max(33, int(w * rng.uniform(0.5, 1.05)))}"

    api = rng.choice(["forward", "forward", "autograd", "autograd", "autograd", "pair", "graph", "batched",
                      "batched", "importance", "admm", "post"])
    if api in ("admm", "post"):
        return _drawn(api, str(log(5000, 4_000_000)), masks="admm" if api == "post" else "uniform")
    if api == "batched":
        scenes = rng.randint(1, 5)
        return _drawn(api, ",".join(str(log(2000, 1_500_000)) for _ in range(scenes)),
                      ",".join(res() for _ in range(rng.randint(1, 5))))
    if api == "importance":
        r = res()
        return _drawn(api, str(log(1000, 2_000_000)), ",".join([r] * rng.randint(1, 4)))
    storage = rng.choice(["f32", "f32", "f16", "f16_bf16s"]) if api in ("forward", "autograd") else "f32"
    return _drawn(api, str(log(1000, 2_000_000)), res(), storage=storage,
                  colour=rng.choice(["sg", "sh3"]) if api == "pair" else "sg")


def _drawn(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    return c


def _ints(text):
    return [int(x) for x in text.split(",") if x]


def _views(case):
    return [tuple(int(v) for v in r.split("x")) for r in case["res"].split(",") if r]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _look_at(eye):
    """World->camera [R | t] of a camera at eye looking at the origin (x right, y down, z forward)."""
    eye = np.asarray(eye, np.float64)
    z = -eye / np.linalg.norm(eye)
    y = np.array([0.0, 1.0, 0.0])
    y = y - y.dot(z) * z
    y /= np.linalg.norm(y)
    rot = np.stack([np.cross(y, z), y, z])
    return np.concatenate([rot, (-rot @ eye)[:, None]], 1).astype(np.float32)


def _cameras(case):
    """Cubes are seen from the origin, the other scenes from a ring of radius 8."""
    cams, views = [], _views(case)
    for i, (w, h) in enumerate(views):
        if case["means"] == "cube":
            cams.append(synth.make_camera(w, h, 150.0 * w / 128.0))
            continue
        th = 2.0 * math.pi * i / len(views)
        fx = w * (1250.0 / 1600.0 if case["means"] == "packed" else 1500.0 / 1920.0)
        cams.append(synth.make_camera(w, h, fx, viewmat=_look_at((8.0 * math.sin(th), 0.0, -8.0 * math.cos(th))),
                                      bg=(0.1, 0.0, 0.2) if i % 2 else (0.0, 0.0, 0.0)))
    return cams


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _scene(case, n, gen):
    """One scene's arrays (planar, as DeviceScene holds them), drawn from gen."""
    dev = gen.device

    def rand(*s):
        return torch.rand(*s, generator=gen, device=dev)

    def randn(*s):
        return torch.randn(*s, generator=gen, device=dev)

    def unit(d, k):
        v = randn(d, k)
        return v / v.norm(dim=0, keepdim=True)

    def lobe_counts(k):
        """Lobes of k Gaussians: every count in its share of the mix, in random order (the total
        is the same for every seed)."""
        if sh3 or case["lobes"] != "mix":
            return torch.full((k,), 0 if sh3 else int(case["lobes"]), dtype=torch.int64, device=dev)
        edges = torch.tensor(np.cumsum(LOBE_P)[:-1] * k, dtype=torch.float64, device=dev)
        at = torch.randperm(k, generator=gen, device=dev)
        return torch.bucketize(at.double() + 0.5, edges)

    sh3 = case["colour"] == "sh3"
    off_g = torch.zeros(n, dtype=torch.bool, device=dev)
    if case["masks"] == "admm":           # exactly half of the Gaussians off
        off_g[torch.randperm(n, generator=gen, device=dev)[:n // 2]] = True
        counts = torch.empty(n, dtype=torch.int64, device=dev)
        counts[off_g], counts[~off_g] = lobe_counts(n // 2), lobe_counts(n - n // 2)
    else:
        counts = lobe_counts(n)
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(counts, 0, out=off[1:])
    n_l = int(off[-1])

    if case["means"] == "cube":
        means = rand(3, n) - 0.5
        means[2] += 4.0
    elif case["means"] == "packed":       # most of the scene in a ball at the centre
        inner = unit(3, n) * 1.5 * rand(n).pow(1.0 / 3.0)
        means = torch.where(rand(n) < 0.7, inner, 10.0 * (rand(3, n) - 0.5))
    else:                                 # 32 anisotropic clusters
        centres = 10.0 * (rand(32, 3) - 0.5)
        axes = torch.linalg.qr(randn(32, 3, 3))[0]
        spread = axes * (0.3 + 1.2 * rand(32, 1, 3))
        which = (rand(n) * 32).long().clamp_(max=31)
        means = (centres[which] + torch.einsum("nij,nj->ni", spread[which], randn(n, 3))).t().contiguous()
    out = {"means": means, "scales": torch.exp(-3.5 + 0.5 * randn(3, n)), "quats": unit(4, n),
           "opac": torch.sigmoid(randn(n)), "gmask": torch.ones(n, device=dev),
           "c0": torch.zeros(3, n, device=dev) if sh3 else rand(3, n), "axis": unit(3, n_l),
           "sharp": torch.exp(math.log(50.0) * rand(n_l)), "amp": 0.3 * randn(3, n_l),
           "lmask": torch.ones(n_l, device=dev)}
    if case["masks"] in ("uniform", "pruned"):
        out["gmask"], out["lmask"] = rand(n), rand(n_l)
    if case["masks"] == "admm":
        # after the constrained optimisation: the pruned opacities and sharpnesses are at zero,
        # the others well above the thresholds
        out["opac"] = torch.where(off_g, 1e-3 * rand(n), 0.1 + 0.9 * out["opac"])
        out["sharp"] += 0.5
        kept = torch.nonzero(~torch.repeat_interleave(off_g, counts))[:, 0]
        gone = kept[torch.randperm(kept.numel(), generator=gen, device=dev)[:kept.numel() // 2]]
        out["sharp"][gone] = 0.5 * rand(gone.numel())
    if case["masks"] == "pruned":         # 60 % of the Gaussians and half of the lobes exactly off
        out["gmask"][rand(n) < 0.6] = 0.0
        out["lmask"][rand(n_l) < 0.5] = 0.0
    if case["storage"] != "f32":
        for k in HALF:
            bf = case["storage"] == "f16_bf16s" and k == "sharp"
            out[k] = out[k].to(torch.bfloat16 if bf else torch.float16)
    out["lobe_off"] = off.to(torch.int32)
    if sh3:
        out["sh"] = 0.2 * randn(3, 16, n)
        out["sh"][:, 0] *= 5.0
    return {k: v.contiguous() for k, v in out.items()}


def _inputs(case, seed):
    """(scenes' arrays, cameras, loss target or upstream gradient), from the seed alone."""
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed) * 7919 + 17)
    arrays = [_scene(case, n, gen) for n in _ints(case["sizes"])]
    cams = _cameras(case)
    pix = 3 * len(arrays) * sum(c.n_pixels for c in cams)
    if case["api"] in ("batched", "graph"):
        extra = torch.rand(pix, generator=gen, device=gen.device)             # target images
    elif case["api"] in ("autograd", "pair"):
        extra = 0.01 * torch.randn(pix, generator=gen, device=gen.device)     # upstream gradient
    elif case["api"] == "admm":
        n, n_l = arrays[0]["opac"].numel(), arrays[0]["sharp"].numel()
        extra = {"importance": torch.rand(n, generator=gen, device=gen.device).pow(4),
                 "lam_o": 0.05 * torch.randn(n, generator=gen, device=gen.device),
                 "lam_s": 0.5 * torch.randn(n_l, generator=gen, device=gen.device),
                 "grad_o": torch.randn(n, generator=gen, device=gen.device),
                 "grad_s": torch.randn(n_l, generator=gen, device=gen.device)}
    else:
        extra = None
    return arrays, cams, extra


def _device_scene(case, a):
    dg = sgsplat.SG_F32 if case["storage"] == "f32" else sgsplat.SG_F16
    ds = sgsplat.SG_BF16 if case["storage"] == "f16_bf16s" else dg
    return DeviceScene(**a, dtype_geom=dg, dtype_lobe=dg, dtype_sharp=ds)


def _mse_grad(renderer, target):
    """Loss gradient of the summed per-view mean squared error, written in place."""
    scale = torch.cat([torch.full((3 * n,), 2.0 / (3 * n), device=renderer.device) for n in renderer.npix])

    def fn(img, out):
        torch.sub(img, target, out=out)
        out.mul_(scale)
    return fn


class _State:
    pass


TAU_OPACITY, DELTA = 0.05, 0.01


def prepare(case, seed):
    arrays, cams, extra = _inputs(case, seed)
    st = _State()
    st.api, st.cams, st.extra = case["api"], cams, extra
    scenes = [_device_scene(case, a) for a in arrays]
    st.scene = scenes[0]
    if st.api in ("batched", "graph"):
        view_scene = [s for s in range(len(scenes)) for _ in cams]
        st.renderer = render.BatchedRenderer(scenes, cams * len(scenes), view_scene)
        st.loss = _mse_grad(st.renderer, extra)
        if st.api == "graph":
            st.renderer.capture(st.loss)
    elif st.api == "autograd":
        st.params = [getattr(st.scene, k).requires_grad_(True) for k in FIELDS]
    elif st.api == "importance":
        st.importance = torch.empty(st.scene.n, device=st.scene.means.device)
    elif st.api == "admm":
        st.tilde_o = torch.zeros_like(st.scene.opac)
        st.tilde_s = torch.zeros_like(st.scene.sharp)
        st.ws = torch.empty(max(sgsplat.sg_admm_workspace_bytes(st.scene.n),
                                sgsplat.sg_admm_workspace_bytes(st.scene.n_lobes), 256),
                            dtype=torch.uint8, device=st.scene.opac.device)
    return st


def run(st):
    if st.api == "forward":
        out = render.render_forward(st.scene, st.cams)
        return {"img": out.img, "T_final": out.T_final, "last": out.last}
    if st.api == "autograd":
        img, T, last = render.rasterize(st.scene, st.cams)
        grads = torch.autograd.grad(img, st.params, st.extra.view(img.shape))
        return {"img": img, "T_final": T, "last": last, "grads": dict(zip(FIELDS, grads))}
    if st.api == "pair":
        out = render.render_forward(st.scene, st.cams)
        grads = render.render_backward(st.scene, st.cams, out, st.extra)
        return {"img": out.img, "T_final": out.T_final, "last": out.last, "grads": grads}
    if st.api in ("batched", "graph"):
        r = st.renderer
        if st.api == "graph":
            r.replay()
        else:
            r.step(st.loss)
        return {"img": r.img, "T_final": r.T_final, "last": r.last, "grads": r.grads}
    if st.api == "importance":
        out = render.render_forward(st.scene, st.cams, importance=st.importance)
        return {"img": out.img, "T_final": out.T_final, "last": out.last, "importance": st.importance}
    if st.api == "admm":
        # the step keeps the previous dual variables and gradients (a program that logs the residual)
        sc, e = st.scene, st.extra
        lam_o, lam_s = e["lam_o"].clone(), e["lam_s"].clone()
        g_o, g_s = e["grad_o"].clone(), e["grad_s"].clone()
        sgsplat.sg_admm_opacity_step(sc.opac, lam_o, st.tilde_o, sc.n // 2, importance=e["importance"], ws=st.ws)
        sgsplat.sg_admm_sharpness_step(sc.sharp, sc.amp, lam_s, st.tilde_s, sc.n_lobes // 2, ws=st.ws)
        sgsplat.sg_admm_penalty_grad(sc.opac, st.tilde_o, lam_o, DELTA, g_o)
        sgsplat.sg_admm_penalty_grad(sc.sharp, st.tilde_s, lam_s, DELTA, g_s)
        return {"tilde_o": st.tilde_o, "lam_o": lam_o, "tilde_s": st.tilde_s, "lam_s": lam_s,
                "grad_o": g_o, "grad_s": g_s}
    out = sgsplat.sg_postprocess(st.scene, TAU_OPACITY)
    return {k: getattr(out, k) for k in FIELDS + ("lobe_off",)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: parameters read and results (gradients included) written once. Flops: projection
    and colour per Gaussian and view, and the blend of the pairs that contribute: a pixel blends
    the Gaussians whose alpha >= 1/255 ellipse covers it until it is opaque (about 60 of them at
    these opacities)."""
    sizes, views = _ints(case["sizes"]), _views(case)
    n = sum(sizes)
    per_lobe = 1.65 if case["lobes"] == "mix" else float(case["lobes"])
    n_l = 0.0 if case["colour"] == "sh3" else per_lobe * n
    half = 2 if case["storage"] != "f32" else 4
    if case["api"] == "admm":
        # two steps: (x, score or amplitude, dual) in, (x~, dual) out; two penalty gradients; four copies
        return {"bytes": 4.0 * (n * (3 + 2 + 5 + 4) + n_l * (5 + 2 + 5 + 4)), "flops": 10.0 * n + 30.0 * n_l}
    lobe_bytes = 7 * half + 4
    params = n * (11 * half + 4 * (1 + 3 + 1)) + n_l * lobe_bytes
    if case["colour"] == "sh3":
        params += 4.0 * 45 * n
    if case["api"] == "post":
        return {"bytes": 1.5 * params, "flops": 5.0 * n + 20.0 * n_l}
    grads = case["api"] in ("autograd", "pair", "batched", "graph")
    pix = float(len(sizes) * sum(w * h for w, h in views))
    bytes_ = params + 20.0 * pix
    if grads:
        bytes_ += params + 20.0 * pix
    if case["api"] == "importance":
        bytes_ += 4.0 * n
    pairs = 0.0
    for s in sizes:
        kept = 0.4 if case["masks"] == "pruned" else 0.55 if case["means"] == "clusters" else 0.9
        for w, h in views:
            sigma = 0.03 * (1.17 if case["means"] == "cube" else 0.78) * w / (4.0 if case["means"] == "cube" else 8.0)
            cover = kept * s * math.pi * (2.2 * max(sigma, 0.55)) ** 2 / (w * h)
            pairs += w * h * min(cover, 60.0)
    flops = pairs * (23.0 + (69.0 if grads else 0.0)) + len(views) * (n * 400.0 + n_l * 30.0) * (2.0 if grads else 1.0)
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

EXACT_PIXELS = 4_000_000     # views beyond this many pixels in all, or more than
EXACT_GAUSSIANS = 8_000_000  # this many projected Gaussians, take too long


def exact(case, seed):
    if case["api"] == "admm":
        return _exact_admm(case, seed)
    if case["api"] == "post":
        return _exact_post(case, seed)
    sizes, views = _ints(case["sizes"]), _views(case)
    if (len(sizes) * sum(w * h for w, h in views) > EXACT_PIXELS
            or len(views) * sum(sizes) > EXACT_GAUSSIANS):
        return None
    arrays, cams, extra = _inputs(case, seed)
    want_grads = case["api"] in ("autograd", "pair", "batched", "graph")
    same = len({(c.width, c.height) for c in cams}) == 1 and case["api"] not in ("batched", "graph")
    imgs, Ts, all_grads, at = [], [], [], 0
    importance = None
    for a in arrays:
        names = FIELDS + (("sh",) if "sh" in a else ())
        leaves = {k: a[k].double().requires_grad_(want_grads) for k in names}
        total = {k: torch.zeros_like(v) for k, v in leaves.items()}
        for cam in cams:
            n = cam.n_pixels
            if want_grads:
                given = extra[3 * at:3 * (at + n)].double().view(3, cam.height, cam.width)
                if case["api"] in ("batched", "graph"):
                    upstream = lambda img, t=given, k=n: (img - t) * (2.0 / (3 * k))   # noqa: E731
                else:
                    upstream = lambda img, t=given: t                                 # noqa: E731
            else:
                upstream = None
            img, T, weight, g = _exact_view(leaves, a["lobe_off"].long(), cam, upstream)
            imgs.append(img)
            Ts.append(T)
            if case["api"] == "importance":
                importance = weight if importance is None else importance + weight
            if g is not None:
                for k in total:
                    total[k] += g[k]
            at += n
        all_grads.append(total)
    if same:
        out = {"img": torch.stack(imgs), "T_final": torch.stack(Ts), "last": None}
    else:
        out = {"img": torch.cat([i.reshape(-1) for i in imgs]), "T_final": torch.cat([t.reshape(-1) for t in Ts]),
               "last": None}
    if want_grads:
        out["grads"] = all_grads if case["api"] in ("batched", "graph") else all_grads[0]
    if case["api"] == "importance":
        out["importance"] = importance
    return out


def _sh_basis(x, y, z):
    """Degree-3 real spherical harmonics with the Condon-Shortley phase, index l^2 + l + m."""
    xx, yy, zz = x * x, y * y, z * z
    p = math.pi
    c1, c2, c2z = math.sqrt(3 / (4 * p)), math.sqrt(15 / (4 * p)), math.sqrt(5 / (16 * p))
    c33, c32, c31, c30 = (math.sqrt(35 / (32 * p)), math.sqrt(105 / (4 * p)), math.sqrt(21 / (32 * p)),
                          math.sqrt(7 / (16 * p)))
    return torch.stack([torch.full_like(x, math.sqrt(1 / (4 * p))), -c1 * y, c1 * z, -c1 * x,
                        c2 * x * y, -c2 * y * z, c2z * (2 * zz - xx - yy), -c2 * x * z, c2 / 2 * (xx - yy),
                        -c33 * y * (3 * xx - yy), c32 * x * y * z, -c31 * y * (4 * zz - xx - yy),
                        c30 * z * (2 * zz - 3 * xx - 3 * yy), -c31 * x * (4 * zz - xx - yy),
                        c32 / 2 * z * (xx - yy), -c33 * x * (xx - 3 * yy)])


def _exact_view(p, lobe_off, cam, upstream):
    """(image, T_final, sum of alpha T per Gaussian, gradients of `p` or None) of one view."""
    dev = p["means"].device
    V = torch.tensor(np.asarray(cam.viewmat, np.float64).reshape(3, 4), device=dev)
    R, t = V[:, :3], V[:, 3]
    n = p["means"].shape[1]
    # projection: EWA with the 3DGS dilation, guard band and 3-sigma rectangle
    tv = R @ p["means"] + t[:, None]
    tx, ty, tz = tv
    w, x, y, z = p["quats"] / p["quats"].norm(dim=0, keepdim=True)
    rot = torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)]),
                       torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)]),
                       torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])])
    M = rot * p["scales"][None]
    ux, uy = tx / tz, ty / tz
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    cx, cy = ux.clamp(-lx, lx) * tz, uy.clamp(-ly, ly) * tz
    A0 = (cam.fx / tz)[None] * R[0][:, None] - (cam.fx * cx / tz ** 2)[None] * R[2][:, None]
    A1 = (cam.fy / tz)[None] * R[1][:, None] - (cam.fy * cy / tz ** 2)[None] * R[2][:, None]
    m0, m1 = torch.einsum("in,ijn->jn", A0, M), torch.einsum("in,ijn->jn", A1, M)
    a, b, c = (m0 * m0).sum(0) + 0.3, (m0 * m1).sum(0), (m1 * m1).sum(0) + 0.3
    det = a * c - b * b
    px, py = cam.fx * ux + cam.cx - 0.5, cam.fy * uy + cam.cy - 0.5
    op = p["gmask"] * p["opac"]
    # colour: diffuse + lobes (or SH), seen along the ray from the camera to the Gaussian
    v = p["means"] + (R.t() @ t)[:, None]
    v = v / v.norm(dim=0, keepdim=True)
    if "sh" in p:
        col = 0.5 + (p["sh"] * _sh_basis(*v)[None]).sum(1)
    else:
        owner = torch.repeat_interleave(torch.arange(n, device=dev), lobe_off[1:] - lobe_off[:-1])
        mu = p["axis"] / p["axis"].norm(dim=0, keepdim=True)
        e = p["lmask"] * torch.exp(p["sharp"] * ((mu * v[:, owner]).sum(0) - 1.0))
        col = p["c0"].index_add(1, owner, p["amp"] * e)
    col = col.clamp(min=0.0)
    flat = torch.stack([px, py, c / det, -b / det, a / det, op, col[0], col[1], col[2]], 1)

    with torch.no_grad():
        mid = 0.5 * (a + c)
        rad = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        nx, ny = cam.tiles_x, cam.tiles_y

        def tile(f, k):
            return torch.floor(f / 16.0).clamp(0, k).nan_to_num(0.0).long()
        x0, x1 = tile(px - rad, nx), tile(px + rad + 15.0, nx)
        y0, y1 = tile(py - rad, ny), tile(py + rad + 15.0, ny)
        vis = (tz > cam.near) & (det > 0) & (x1 > x0) & (y1 > y0) & (op >= 1.0 / 255.0)
        ids = torch.nonzero(vis)[:, 0]
        ids = ids[torch.argsort(tz[ids], stable=True)]
        cnt = ((x1 - x0) * (y1 - y0))[ids]
        rep = torch.repeat_interleave(torch.arange(ids.numel(), device=dev), cnt)
        k = torch.arange(rep.numel(), device=dev) - (torch.cumsum(cnt, 0) - cnt)[rep]
        g = ids[rep]
        wd = (x1 - x0)[g]
        tid = (y0[g] + k // wd) * nx + x0[g] + k % wd
        order = torch.argsort(tid, stable=True)
        g = g[order]
        length = torch.bincount(tid, minlength=nx * ny)
        start = torch.cumsum(length, 0) - length
        by_len = torch.argsort(length, descending=True).tolist()
        lens = length.tolist()
        data = torch.cat([flat.detach(), torch.zeros(1, 9, device=dev, dtype=torch.float64)])   # row n: no Gaussian
        data[n, 2] = data[n, 4] = 1.0
        g = torch.cat([g, torch.full((1,), n, device=dev)])
        bg = torch.tensor(np.asarray(cam.bg, np.float64), device=dev)
        pad = torch.zeros(4, ny * 16, nx * 16, device=dev, dtype=torch.float64)
        ly_, lx_ = torch.meshgrid(torch.arange(16, device=dev), torch.arange(16, device=dev), indexing="ij")
        ly_, lx_ = ly_.reshape(-1), lx_.reshape(-1)
        weight = torch.zeros(n + 1, device=dev, dtype=torch.float64)

    def groups():
        i = 0
        while i < len(by_len):
            longest = max(1, lens[by_len[i]])
            m = max(1, min(len(by_len) - i, 8_000_000 // (256 * longest)))
            tiles = torch.tensor(by_len[i:i + m], device=dev)
            at = torch.arange(longest, device=dev)[None]
            idx = torch.where(at < length[tiles][:, None], start[tiles][:, None] + at, g.numel() - 1)
            yield tiles, g[idx]
            i += m

    def blend(q, tiles):
        fx = (tiles % nx)[:, None] * 16.0 + lx_[None]
        fy = (tiles // nx)[:, None] * 16.0 + ly_[None]
        dx, dy = fx[:, :, None] - q[:, None, :, 0], fy[:, :, None] - q[:, None, :, 1]
        power = -0.5 * (q[:, None, :, 2] * dx * dx + q[:, None, :, 4] * dy * dy) - q[:, None, :, 3] * dx * dy
        alpha = (q[:, None, :, 5] * torch.exp(power)).clamp(max=0.99)
        keep = (power.detach() <= 0) & (alpha.detach() >= 1.0 / 255.0)
        alpha = alpha * keep
        keep = keep & (torch.exp(torch.cumsum(torch.log1p(-alpha.detach()), 2)) >= 1e-4)
        alpha = alpha * keep
        lt = torch.cumsum(torch.log1p(-alpha), 2)
        wgt = alpha * torch.exp(lt - torch.log1p(-alpha))
        T = torch.exp(lt[:, :, -1])
        return wgt @ q[:, :, 6:9] + T[:, :, None] * bg, T, wgt

    def scatter(dst, tiles, val):          # val [tiles, 256, channels] -> dst [channels, H, W] (padded)
        yy, xx = (tiles // nx)[:, None] * 16 + ly_[None], (tiles % nx)[:, None] * 16 + lx_[None]
        dst[:, yy, xx] = val.permute(2, 0, 1)

    with torch.no_grad():
        for tiles, who in groups():
            img, T, wgt = blend(data[who], tiles)
            inside = ((tiles % nx)[:, None] * 16 + lx_ < cam.width) & ((tiles // nx)[:, None] * 16 + ly_ < cam.height)
            wgt = wgt * inside[:, :, None]
            scatter(pad, tiles, torch.cat([img, T[:, :, None]], 2))
            weight.index_add_(0, who.reshape(-1), wgt.sum(1).reshape(-1))
    img, T = pad[:3, :cam.height, :cam.width].contiguous(), pad[3, :cam.height, :cam.width].contiguous()
    if upstream is None:
        return img, T, weight[:n], None
    d_pad = torch.zeros(3, ny * 16, nx * 16, device=dev, dtype=torch.float64)
    d_pad[:, :cam.height, :cam.width] = upstream(img)
    d_flat = torch.zeros(n + 1, 9, device=dev, dtype=torch.float64)
    for tiles, who in groups():
        yy, xx = (tiles // nx)[:, None] * 16 + ly_[None], (tiles % nx)[:, None] * 16 + lx_[None]
        q = data[who].requires_grad_(True)
        dq, = torch.autograd.grad(blend(q, tiles)[0], q, d_pad[:, yy, xx].permute(1, 2, 0))
        d_flat.index_add_(0, who.reshape(-1), dq.reshape(-1, 9))
    d_flat = torch.where(vis[:, None], d_flat[:n], torch.zeros_like(d_flat[:n]))
    # a culled Gaussian gets no gradient, whatever its projection did
    got = torch.autograd.grad(torch.where(vis[:, None], flat, torch.zeros_like(flat)), list(p.values()), d_flat,
                              allow_unused=True)
    return img, T, weight[:n], {k: torch.zeros_like(p[k]) if x is None else x.nan_to_num(0.0)
                                for k, x in zip(p, got)}


def _exact_prox(x, lam, score, kappa):
    order = torch.argsort(score, descending=True, stable=True)[:kappa]
    keep = torch.zeros_like(x, dtype=torch.bool)
    keep[order] = True
    z = x + lam
    tilde = torch.where(keep, z, torch.zeros_like(z))
    return tilde, lam + (x - tilde)


def _exact_admm(case, seed):
    (a,), _, e = _inputs(case, seed)
    e = {k: v.double() for k, v in e.items()}
    o, s, amp = a["opac"].double(), a["sharp"].double(), a["amp"].double()
    t_o, l_o = _exact_prox(o, e["lam_o"], e["importance"], o.numel() // 2)
    span = amp.norm(dim=0) * (1.0 - torch.exp(-2.0 * (s + e["lam_s"]))).abs()
    t_s, l_s = _exact_prox(s, e["lam_s"], span, s.numel() // 2)
    return {"tilde_o": t_o, "lam_o": l_o, "tilde_s": t_s, "lam_s": l_s,
            "grad_o": e["grad_o"] + DELTA * (o - t_o + l_o), "grad_s": e["grad_s"] + DELTA * (s - t_s + l_s)}


def _exact_post(case, seed):
    (a,), _, _ = _inputs(case, seed)
    off = a["lobe_off"].long()
    n = off.numel() - 1
    owner = torch.repeat_interleave(torch.arange(n, device=off.device), off[1:] - off[:-1])
    keep_g = a["gmask"] * a["opac"] >= torch.tensor(TAU_OPACITY, device=off.device)   # a binary32 decision
    sharp = a["sharp"].double()
    keep_l = keep_g[owner] & (a["sharp"] >= 1.0)
    gone = keep_g[owner] & ~keep_l
    f = torch.where(sharp.abs() < 1e-9, torch.ones_like(sharp), -torch.expm1(-2.0 * sharp) / (2.0 * sharp))
    add = a["amp"].double() * (a["lmask"].double() * f * gone)
    c0 = a["c0"].double().index_add(1, owner, add)
    per = torch.zeros(n, dtype=torch.int64, device=off.device).index_add_(0, owner, keep_l.long())[keep_g]
    out = {k: a[k][..., keep_g].double() for k in ("means", "scales", "quats", "opac", "gmask")}
    out["c0"] = c0[:, keep_g]
    out |= {k: a[k][..., keep_l].double() for k in ("axis", "sharp", "amp", "lmask")}
    out["lobe_off"] = torch.cat([torch.zeros_like(per[:1]), torch.cumsum(per, 0)]).to(torch.int32)
    return out
