"""What the performance of this framework is measured on: its entry points at the sizes users call them with.

The workloads are the framework's own: training steps of one cell (render, Eq. 1 loss, backward) from a
10k-Gaussian toy cell to the 20M-Gaussian urban cell, several aerial cells trained in one batch, novel views
of the merged city, the appearance loss of Eq. 3, and the steps around the loop: Adam, densification, the
seamless merge, the camera selection and the corrected evaluation.  Scenes follow ``scenes.py``'s recipes, drawn
on the GPU so that inputs of a new seed are quick to make.

``exact`` evaluates the same definitions in 64 bits with plain torch.
"""
import copy
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2402_17427_gb300 import appearance as AP
from paper_2402_17427_gb300 import batch as BT
from paper_2402_17427_gb300 import optim as OP
from paper_2402_17427_gb300 import partition as PT
from paper_2402_17427_gb300 import rasterize as R
from paper_2402_17427_gb300 import scenes
from paper_2402_17427_gb300 import serving as SV

DEV = "cuda"
Y00 = 0.5 / math.sqrt(math.pi)


def listed():
    return [
        # the smallest training step: the 10k-Gaussian toy cell, where launches and host work count
        {"name": "step_10k_128", "kind": "step", "scene": "box", "n": 10_000, "degree": 0, "w": 128, "h": 128,
         "tile": 16, "stats": True},
        # the headline: one training step of a 1M-Gaussian cell at 1080p, with densification statistics
        {"name": "step_1m_1080p", "kind": "step", "scene": "blob", "n": 1_000_000, "degree": 3, "w": 1920, "h": 1080,
         "tile": 16, "stats": True},
        # a training step of the densest cell one GPU holds: 20M Gaussians, gradients of all of them
        {"name": "step_20m_1080p", "kind": "step", "scene": "city", "n": 20_000_000, "degree": 3, "w": 1920, "h": 1080,
         "tile": 16, "stats": False},
        # uneven aerial cells trained together in one call a stage, with two tile sizes as the autotuner picks
        {"name": "batch_6cells", "kind": "batch", "cells": "300000,500000,800000,1200000,1500000,2000000",
         "degree": 3, "w": 1152, "h": 864, "tiles": "8,16"},
        # one request batch of the novel-view server over the merged city: the three resolutions it is asked for
        {"name": "views_720p_1080p_4k", "kind": "views", "cells": 16, "n": 8_000_000, "degree": 3,
         "views": "1280x720,1280x720,1920x1080,3840x2160"},
        # the appearance loss of Eq. 3 with every gradient, at the training resolution
        {"name": "appearance_1080p", "kind": "appearance", "w": 1920, "h": 1080, "grad": True},
        # the same on a small ragged crop, where the low-resolution layers and the launches dominate
        {"name": "appearance_330x200", "kind": "appearance", "w": 330, "h": 200, "grad": True},
        # the optimiser update of a 1M-Gaussian cell: one per training iteration
        {"name": "adam_1m", "kind": "adam", "n": 1_000_000, "degree": 3},
        # clone / split / prune of that cell: every 200 iterations
        {"name": "densify_1m", "kind": "densify", "n": 1_000_000, "degree": 3},
        # the seamless merge of 16 expanded cells into one 20M-input model: once per scene
        {"name": "merge_16x1250k", "kind": "merge", "cells": 16, "n": 1_250_000, "degree": 3},
        # airspace boxes of 16 cells and the selection among 4000 cameras: once per scene
        {"name": "select_16x4000", "kind": "select", "cells": 16, "n": 1_250_000, "cameras": 4000},
        # colour-corrected PSNR / SSIM of one held-out view
        {"name": "evaluate_1080p", "kind": "evaluate", "w": 1920, "h": 1080},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _image(rng, lo, hi):
    """A width drawn over its logarithm, odd or even alike, with an aspect between 1:1 and 2:1."""
    w = _log(rng, lo, hi)
    return w, max(32, min(1080, int(round(w / rng.uniform(1.0, 2.0)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "views", "appearance", "appearance", "adam", "densify",
                       "merge", "select", "evaluate"])
    deg = rng.choice([0, 1, 2, 3, 3])
    if kind == "step":
        w, h = _image(rng, 64, 1920)
        scene = rng.choice(["box", "blob", "city"])
        n = _log(rng, 2_000, {"box": 100_000, "blob": 1_500_000, "city": 8_000_000}[scene])
        return {"kind": "step", "scene": scene, "n": n, "degree": deg, "w": w, "h": h, "tile": rng.choice([8, 16, 16, 16, 32]),
                "stats": rng.random() < 0.5}
    if kind == "batch":
        k = rng.randint(2, 6)
        w, h = _image(rng, 256, 1152)
        return {"kind": "batch", "cells": ",".join(str(_log(rng, 20_000, 1_500_000)) for _ in range(k)), "degree": deg,
                "w": w, "h": h, "tiles": rng.choice(["16", "8,16", "8,16,32"])}
    if kind == "views":
        res = rng.choices(["1280x720", "1920x1080", "3840x2160", "1003x757"], weights=[5, 3, 1, 2], k=rng.randint(1, 4))
        return {"kind": "views", "cells": rng.randint(2, 16), "n": _log(rng, 300_000, 4_000_000), "degree": deg,
                "views": ",".join(res)}
    if kind == "appearance":
        w, h = _image(rng, 64, 1920)
        return {"kind": "appearance", "w": w, "h": h, "grad": rng.random() < 0.75}
    if kind in ("adam", "densify"):
        return {"kind": kind, "n": _log(rng, 5_000, 3_000_000 if kind == "adam" else 1_500_000), "degree": deg}
    if kind == "merge":
        return {"kind": "merge", "cells": rng.randint(2, 16), "n": _log(rng, 10_000, 1_000_000), "degree": deg}
    if kind == "select":
        return {"kind": "select", "cells": rng.randint(1, 40), "n": _log(rng, 10_000, 400_000),
                "cameras": _log(rng, 100, 4000)}
    w, h = _image(rng, 64, 1920)
    return {"kind": "evaluate", "w": w, "h": h}


# ---------------------------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (int(seed) + 1) + salt)
    return g


def _rand(g, *shape):
    return torch.rand(shape, device=DEV, generator=g)


def _randn(g, *shape):
    return torch.randn(shape, device=DEV, generator=g)


def _params(g, means, log_scale, degree):
    """Raw parameters around the given means: log-scales N(log_scale, 0.5), unit quaternions, logits N(0, 1),
    base colours U(0, 1) as DC coefficients and N(0, 0.2) above."""
    n, k = means.shape[0], (degree + 1) ** 2
    sh = 0.2 * _randn(g, n, k, 3)
    sh[:, 0] = (_rand(g, n, 3) - 0.5) / Y00
    q = _randn(g, n, 4)
    return [means.contiguous(), log_scale + 0.5 * _randn(g, n, 3), q / q.norm(dim=1, keepdim=True), _randn(g, n), sh]


def _ground(x, z):
    return 2.0 * torch.sin(x / 57.0) * torch.cos(z / 83.0) + torch.sin((x + z) / 31.0)


def _city_points(g, n, x0, x1, z0, z1, boxes, facade=0.7):
    """Points on building boxes (walls and roofs) and on the ground, in random order."""
    bx, bz = x0 + (x1 - x0) * _rand(g, boxes), z0 + (z1 - z0) * _rand(g, boxes)
    bw, bd, bh = 10 + 30 * _rand(g, boxes), 10 + 30 * _rand(g, boxes), 10 + 50 * _rand(g, boxes)
    area = torch.stack([bw * bh, bw * bh, bd * bh, bd * bh, bw * bd], 1).reshape(-1)
    cum = torch.cumsum(area.double(), 0)
    m = int(n * facade)
    pick = torch.searchsorted(cum, cum[-1] * _rand(g, m).double()).clamp_(max=area.numel() - 1)
    b, face = pick // 5, pick % 5
    s, t = _rand(g, m) - 0.5, _rand(g, m)
    p = torch.stack([bx[b] + s * bw[b], _ground(bx, bz)[b] + t * bh[b], bz[b] + s * bd[b]], 1)
    off = 0.1 * _randn(g, m)
    for f, axis, sign, ext in ((0, 2, -1, bd), (1, 2, 1, bd), (2, 0, -1, bw), (3, 0, 1, bw)):
        centre = (bz if axis == 2 else bx)[b]
        p[:, axis] = torch.where(face == f, centre + sign * (0.5 * ext[b] + off), p[:, axis])
    roof = face == 4
    p[:, 1] = torch.where(roof, (_ground(bx, bz) + bh)[b] + off, p[:, 1])
    p[:, 2] = torch.where(roof, bz[b] + (t - 0.5) * bd[b], p[:, 2])
    gx, gz = x0 + (x1 - x0) * _rand(g, n - m), z0 + (z1 - z0) * _rand(g, n - m)
    ground = torch.stack([gx, _ground(gx, gz) + 0.1 * _randn(g, n - m), gz], 1)
    return torch.cat([p, ground])[torch.randperm(n, device=DEV, generator=g)]


def _aerial_camera(rng, w, h, x0, x1, z0, z1, alt, pitch):
    yaw = rng.uniform(0.0, 2.0 * math.pi)
    eye = (rng.uniform(x0, x1), alt, rng.uniform(z0, z1))
    up = (math.sin(yaw), 0.0, math.cos(yaw)) if pitch < -1.55 else (0.0, 1.0, 0.0)
    return scenes.camera_from_forward(eye, scenes.yaw_pitch_forward(yaw, pitch), w, h, up_hint=up)


def _scene(case, seed):
    """(raw parameters, camera, target) of a single-cell training step."""
    g, rng = _gen(seed), np.random.Generator(np.random.PCG64(seed))
    n, w, h, deg = case["n"], case["w"], case["h"], case["degree"]
    if case["scene"] == "box":
        p = _params(g, 4.0 * _rand(g, n, 3) - 2.0, -3.0, deg)
        cam = scenes.look_at((0.0, 0.0, -6.0), (0.0, 0.0, 0.0), w, h, fx=float(w))
    elif case["scene"] == "blob":
        ext = torch.tensor([100.0, 20.0, 100.0], device=DEV)
        centres, std = ext * _rand(g, 64, 3), 2.0 + 6.0 * _rand(g, 64)
        which = torch.randint(0, 64, (n,), device=DEV, generator=g)
        means = torch.minimum((centres[which] + std[which, None] * _randn(g, n, 3)).clamp_(min=0.0), ext)
        p = _params(g, means, math.log(0.08) + math.log(1e6 / n) / 3.0, deg)
        yaw = rng.uniform(0.0, 2.0 * math.pi)
        cam = scenes.camera_from_forward((50.0 + 30.0 * math.sin(yaw), 30.0, 50.0 + 30.0 * math.cos(yaw)),
                                         scenes.yaw_pitch_forward(yaw + math.pi, -math.pi / 4), w, h)
    else:
        means = _city_points(g, n, 0.0, 500.0, 0.0, 500.0, 150)
        p = _params(g, means, math.log(0.5 * math.sqrt(500.0 * 500.0 / n)), deg)
        cam = _aerial_camera(rng, w, h, 100.0, 400.0, 100.0, 400.0, 80.0, -math.pi / 4)
    return p, cam, _rand(g, 3, h, w)


def _batch_scene(case, seed):
    g, rng = _gen(seed), np.random.Generator(np.random.PCG64(seed))
    cells, cams, targets = [], [], []
    for k, n in enumerate(int(v) for v in case["cells"].split(",")):
        x0, z0 = 250.0 * (k % 4), 500.0 * (k // 4)
        means = _city_points(g, n, x0, x0 + 250.0, z0, z0 + 500.0, 20)
        cells.append(_params(g, means, math.log(0.5 * math.sqrt(250.0 * 500.0 / n)), case["degree"]))
        cams.append(_aerial_camera(rng, case["w"], case["h"], x0 + 35.0, x0 + 215.0, z0 + 25.0, z0 + 475.0, 100.0,
                                   -math.pi / 2))
        targets.append(_rand(g, 3, case["h"], case["w"]))
    return cells, cams, targets


def _settings(tiles, n):
    t = [int(v) for v in tiles.split(",")]
    return [R.RasterSettings(tile_size=t[k % len(t)]) for k in range(n)]


def _views_scene(case, seed):
    """The merged city: cells of uneven size on a 250 m grid, and one camera a requested view."""
    g, rng = _gen(seed), np.random.Generator(np.random.PCG64(seed))
    k = case["cells"]
    share = np.array([1.0 + i / 5.0 for i in range(k)])
    sizes = np.maximum(1, case["n"] * share / share.sum()).astype(int)
    side = math.ceil(math.sqrt(k))
    cells = []
    for slot, n in zip(rng.permutation(k).tolist(), sizes.tolist()):
        x0, z0 = 250.0 * (slot % side), 250.0 * (slot // side)
        means = _city_points(g, n, x0, x0 + 250.0, z0, z0 + 250.0, 10)
        cells.append(_params(g, means, math.log(0.5 * math.sqrt(250.0 * 250.0 / n)), case["degree"]))
    cams = []
    for v in case["views"].split(","):
        w, h = (int(t) for t in v.split("x"))
        cams.append(_aerial_camera(rng, w, h, 0.0, 250.0 * side, 0.0, 250.0 * side, rng.uniform(20.0, 150.0),
                                   math.radians(rng.uniform(-90.0, -30.0))))
    return cells, cams


def _photo(g, w, h):
    """A smooth image with detail and noise, and a rendering of it under another exposure: (rendering, target)."""
    y = F.interpolate(_rand(g, 1, 3, max(2, h // 16), max(2, w // 16)), size=(h, w), mode="bicubic", align_corners=False)[0]
    y = (y + 0.05 * _randn(g, 3, h, w)).clamp_(0.0, 1.0)
    x = (0.9 * y + 0.05 + 0.05 * _randn(g, 3, h, w)).clamp_(0.0, 1.0)
    return x.contiguous(), y.contiguous()


def _raw_like(g, n, degree, scale):
    return [scale * _randn(g, *s) for s in ((n, 3), (n, 3), (n, 4), (n,), (n, (degree + 1) ** 2, 3))]


def _densify_scene(case, seed):
    """Parameters, moments and statistics that prune, keep, clone and split a share each.  What decides is the same
    set for every seed, in another order, so that the number of Gaussians that come out is too."""
    g, one, n = _gen(seed), _gen(0, 7), case["n"]
    order = torch.randperm(n, device=DEV, generator=g)
    p = _raw_like(g, n, case["degree"], 1.0)
    p[1] = (0.8 * _randn(one, n, 3) + math.log(0.05))[order]
    p[3] = (3.0 * _randn(one, n))[order]
    m, v = _raw_like(g, n, case["degree"], 1e-2), [t.square() for t in _raw_like(g, n, case["degree"], 1e-2)]
    accum = torch.empty(n, device=DEV).exponential_(1.0 / 3e-4, generator=one)[order]
    count = torch.randint(0, 4, (n,), device=DEV, generator=one, dtype=torch.int32)[order]
    return p, m, v, accum, count, _randn(g, n, 2, 3)


def _expanded_cells(case, seed, points_only=False):
    """Cells on a 250 m grid holding the Gaussians of their 20 % expanded rectangles.  The ground positions of a merge
    are the same set for every seed, in another order, so that the number of Gaussians kept is too."""
    g, one, k, n = _gen(seed), _gen(0, 11), case["cells"], case["n"]
    side = math.ceil(math.sqrt(k))
    cells, regions = [], []
    for c in range(k):
        x0, z0 = 250.0 * (c % side), 250.0 * (c // side)
        lo, ext = torch.tensor([x0 - 25.0, 0.0, z0 - 25.0], device=DEV), torch.tensor([300.0, 60.0, 300.0], device=DEV)
        means = lo + ext * (_rand(g, n, 3) if points_only else _rand(one, n, 3)[torch.randperm(n, device=DEV, generator=g)])
        cells.append(means if points_only else [means, *_raw_like(g, n, case["degree"], 1.0)[1:]])
        regions.append((x0, x0 + 250.0, z0, z0 + 250.0))
    return cells, regions


def _selection_cameras(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    ext = 250.0 * math.ceil(math.sqrt(case["cells"]))
    return [_aerial_camera(rng, *scenes.RESOLUTIONS[i % 3], 0.0, ext, 0.0, ext, rng.uniform(20.0, 150.0),
                           math.radians(rng.uniform(-88.0, -30.0))) for i in range(case["cameras"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        p, cam, target = _scene(case, seed)
        p = [t.requires_grad_(True) for t in p]
        ras = R.Rasterizer(R.RasterSettings(tile_size=case["tile"]))
        s = {"params": p, "cam": cam, "target": target, "ras": ras, "loss": R.LossL1DSSIM(0.2)}
        if case["stats"]:
            s["stats"] = OP.DensifyStats(case["n"], DEV)
        with torch.no_grad():      # one synchronous render sizes the pair list; training then never waits for the GPU
            ras.forward(*p, case["degree"], cam)
        ras.check = "defer"
    elif kind == "batch":
        cells, cams, targets = _batch_scene(case, seed)
        br = BT.BatchRasterizer(_settings(case["tiles"], len(cells)))
        br.forward(cells, case["degree"], cams)
        br.check = "defer"
        s = {"cells": cells, "cams": cams, "targets": targets, "br": br, "loss": [R.LossL1DSSIM(0.2) for _ in cells]}
    elif kind == "views":
        cells, cams = _views_scene(case, seed)
        host = [scenes.Cell(scenes.Gaussians(*(t.cpu().numpy() for t in c), case["degree"]),
                            torch.cat([c[0].amin(0), c[0].amax(0)]).cpu().numpy()) for c in cells]
        s = {"server": SV.SceneServer(host), "cams": cams}
        s["server"].render(cams)   # allocates the workspace and learns the pairs a megapixel
    elif kind == "appearance":
        x, y = _photo(_gen(seed), case["w"], case["h"])
        s = {"img": x, "target": y, "model": AP.AppearanceModel(4, seed=seed)}
    elif kind == "adam":
        g = _gen(seed)
        p = _raw_like(g, case["n"], case["degree"], 1.0)
        s = {"params": p, "grads": _raw_like(g, case["n"], case["degree"], 1e-4), "adam": OP.Adam(p)}
        s["adam"].m = tuple(_raw_like(g, case["n"], case["degree"], 1e-4))
        s["adam"].v = tuple(1e-9 + t.square() for t in _raw_like(g, case["n"], case["degree"], 1e-4))
        s["adam"].t = 1000
    elif kind == "densify":
        p, m, v, accum, count, normals = _densify_scene(case, seed)
        adam, stats = OP.Adam(p), OP.DensifyStats(case["n"], DEV)
        adam.m, adam.v, stats.accum, stats.count = tuple(m), tuple(v), accum, count
        s = {"params": p, "adam": adam, "stats": stats, "normals": normals}
    elif kind == "merge":
        cells, regions = _expanded_cells(case, seed)
        s = {"cells": cells, "regions": regions}
    elif kind == "select":
        cells, _ = _expanded_cells(case, seed, points_only=True)
        s = {"points": torch.cat(cells), "offsets": [case["n"] * k for k in range(case["cells"] + 1)],
             "cams": PT.camera_table(_selection_cameras(case, seed))}
    else:
        x, y = _photo(_gen(seed), case["w"], case["h"])
        s = {"img": x, "target": y}
    s["case"] = case
    return s


# ---------------------------------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        img = R.rasterize(*s["params"], case["degree"], s["cam"], s["ras"])
        loss = R.l1_dssim_loss(img, s["target"], 0.2, s["loss"])
        out = {"image": img.detach(), "loss": loss.detach(), "grads": torch.autograd.grad(loss, s["params"])}
        if case["stats"]:
            s["stats"].add_view(s["ras"], case["n"], s["cam"])
            out["accum"], out["count"] = s["stats"].accum, s["stats"].count
        return out
    if kind == "batch":
        outs = s["br"].forward(s["cells"], case["degree"], s["cams"])
        lg = [f(o[0], t) for f, o, t in zip(s["loss"], outs, s["targets"])]
        grads = s["br"].backward(s["cells"], case["degree"], s["cams"], outs, [g for _, g in lg])
        return {"outs": outs, "loss": [v for v, _ in lg], "grad_image": [g for _, g in lg], "grads": grads}
    if kind == "views":
        return s["server"].render(s["cams"])[0]
    if kind == "appearance":
        return s["model"].loss(s["img"], s["target"], 1, grad=case["grad"], want_map=not case["grad"])
    if kind == "adam":
        s["adam"].step(s["params"], s["grads"], case["degree"])
        return {"params": s["params"], "m": s["adam"].m, "v": s["adam"].v}
    if kind == "densify":
        adam, stats = copy.copy(s["adam"]), copy.copy(s["stats"])
        new = OP.densify_with(s["params"], adam, stats, case["degree"], OP.DensifySettings(scene_extent=10.0), s["normals"])
        return {"params": new, "m": adam.m, "v": adam.v}
    if kind == "merge":
        return PT.merge_cells(s["cells"], s["regions"], case["degree"])
    if kind == "select":
        boxes = PT.airspace_boxes(s["points"], s["offsets"], 0.0)
        vis, sel = PT.camera_visibility(boxes, s["cams"])
        return {"boxes": boxes, "visibility": vis, "selected": sel}
    return R.color_corrected_metrics(s["img"], s["target"])


def work(case):
    """Bytes: every input read once, every output written once.  Operations: the method's own, about 224 (pixel,
    Gaussian) evaluations of 11 operations a pixel and 56 of them blended (7 operations, 37 in the adjoint), the
    counts of the 1M-Gaussian cell; 3x3 convolutions as multiply-adds; the other paths are copies and sums."""
    kind = case["kind"]
    f = 11 + 3 * (case.get("degree", 0) + 1) ** 2
    px = case["w"] * case["h"] if "w" in case else 0
    evals, step_ops = 224 * 11, 224 * 11 * 2 + 56 * 44
    if kind == "step":
        return {"bytes": 8 * f * case["n"] + 24 * px, "flops": step_ops * px}
    if kind == "batch":
        sizes = [int(v) for v in case["cells"].split(",")]
        return {"bytes": 8 * f * sum(sizes) + 44 * px * len(sizes), "flops": step_ops * px * len(sizes)}
    if kind == "views":
        total = sum(int(v.split("x")[0]) * int(v.split("x")[1]) for v in case["views"].split(","))
        return {"bytes": 4 * f * case["n"] + 20 * total, "flops": (evals + 56 * 7) * total}
    if kind == "appearance":
        h, w, fwd = case["h"] // 32, case["w"] // 32, 0
        for k, (c, o) in enumerate(AP.LAYERS):
            fwd += 2 * 9 * c * o * (px if k > 4 else (h << k) * (w << k))
        return {"bytes": 36 * px + 4 * 255_539 * (2 if case["grad"] else 1),
                "flops": fwd * (3 if case["grad"] else 1)}
    if kind == "adam":
        return {"bytes": 28 * f * case["n"], "flops": 12 * f * case["n"]}
    if kind == "densify":   # about 1.17 Gaussians out for one in, each with two moments
        return {"bytes": int(12 * f * case["n"] * 2.17) + 32 * case["n"], "flops": 0}
    if kind == "merge":     # (250 / 300)^2 of the Gaussians are kept
        return {"bytes": int(case["cells"] * case["n"] * (12 + 8 * f * 0.694)), "flops": 0}
    if kind == "select":
        pairs = case["cells"] * case["cameras"]
        return {"bytes": 12 * case["cells"] * case["n"] + 6 * pairs, "flops": 1000 * pairs}
    return {"bytes": 24 * px, "flops": 600 * px}


# ---------------------------------------------------------------------------------------- 64 bits

def _t64(a):
    return torch.as_tensor(np.asarray(a, np.float64), device=DEV)


def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    c = lambda v: math.sqrt(v / math.pi)  # noqa: E731
    b = [torch.full_like(x, 0.5 * c(1.0))]
    if degree > 0:
        b += [-c(0.75) * y, c(0.75) * z, -c(0.75) * x]
    if degree > 1:
        b += [c(3.75) * x * y, -c(3.75) * y * z, c(0.3125) * (2 * zz - xx - yy), -c(3.75) * x * z, c(0.9375) * (xx - yy)]
    if degree > 2:
        b += [-c(35 / 32) * y * (3 * xx - yy), c(26.25) * x * y * z, -c(21 / 32) * y * (4 * zz - xx - yy),
              c(7 / 16) * z * (2 * zz - 3 * xx - 3 * yy), -c(21 / 32) * x * (4 * zz - xx - yy),
              c(105 / 16) * z * (xx - yy), -c(35 / 32) * x * (xx - 3 * yy)]
    return torch.stack(b, 1)


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _project(p, cam, degree):
    """2D Gaussians of raw parameters in front of the near plane: dict of u, v, conic, opacity, rgb, r, z, det."""
    means, ls, q, logit, sh = p
    W = _t64(cam.R)
    c = means @ W.T + _t64(cam.t)
    z = c[:, 2]
    xz, yz = c[:, 0] / z, c[:, 1] / z
    limx, limy = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    xc, yc = xz.clamp(-limx, limx), yz.clamp(-limy, limy)
    zero = torch.zeros_like(z)
    J = torch.stack([cam.fx / z, zero, -cam.fx * xc / z, zero, cam.fy / z, -cam.fy * yc / z], 1).view(-1, 2, 3)
    M = J @ W @ _rotation(q) * torch.exp(ls)[:, None, :]
    C = M @ M.transpose(1, 2)
    A, B, D = C[:, 0, 0] + 0.3, C[:, 0, 1], C[:, 1, 1] + 0.3
    det = A * D - B * B
    r = 3.0 * torch.sqrt(0.5 * (A + D) + torch.sqrt((0.5 * (A - D)) ** 2 + B * B)).detach()
    d = means - _t64(cam.cam_pos)
    rgb = ((_sh_basis(d / d.norm(dim=1, keepdim=True), degree)[:, :, None] * sh).sum(1) + 0.5).clamp(min=0.0)
    return {"u": cam.fx * xz + cam.cx, "v": cam.fy * yz + cam.cy, "a": D / det, "b": -B / det, "c": A / det,
            "o": torch.sigmoid(logit), "rgb": rgb, "r": r, "z": z.detach()}


def _rect(g, cam, tile):
    """Tile rectangle of each 2D Gaussian and whether it holds a pixel of the image."""
    u, v, r = g["u"].detach(), g["v"].detach(), g["r"]
    lo = [torch.ceil(t - r).clamp(min=0) for t in (u, v)]
    hi = [torch.minimum(torch.floor(t + r), torch.full_like(t, n - 1.0)) for t, n in ((u, cam.width), (v, cam.height))]
    ok = (lo[0] <= hi[0]) & (lo[1] <= hi[1])
    return [(t.clamp(0, 1e5).long() // tile) for t in (lo[0], hi[0], lo[1], hi[1])], ok


class _Exact64:
    """The rasteriser's definition in 64 bits: lists by a stable sort, compositing over padded tile lists."""

    def __init__(self, params, cam, degree, tile):
        self.cam, self.degree, self.tile, self.n = cam, degree, tile, params[0].shape[0]
        self.shapes = [t.shape for t in params]
        front = []
        for k in range(0, self.n, 1 << 20):
            m = params[0][k:k + (1 << 20)].detach().double()
            c = m @ _t64(cam.R).T + _t64(cam.t)
            front.append((c[:, 2] > cam.near).nonzero()[:, 0] + k)
        ids = torch.cat(front)
        keep = []
        for k in range(0, ids.numel(), 1 << 20):
            part = ids[k:k + (1 << 20)]
            with torch.no_grad():
                g = _project([t.detach()[part].double() for t in params], cam, degree)
                keep.append(part[_rect(g, cam, tile)[1]])
        self.ids = torch.cat(keep)
        self.leaf = [t.detach()[self.ids].double().requires_grad_(True) for t in params]
        self.g = _project(self.leaf, cam, degree)
        rect, _ = _rect(self.g, cam, tile)
        self.tx, self.ty = -(-cam.width // tile), -(-cam.height // tile)
        order = torch.argsort(self.g["z"], stable=True)
        x0, x1, y0, y1 = (t[order] for t in rect)
        nx = x1 - x0 + 1
        count = nx * (y1 - y0 + 1)
        own = torch.repeat_interleave(torch.arange(order.numel(), device=DEV), count)
        at = torch.arange(own.numel(), device=DEV) - (torch.cumsum(count, 0) - count)[own]
        tiles = (y0[own] + at // nx[own]) * self.tx + x0[own] + at % nx[own]
        tiles, by = torch.sort(tiles, stable=True)
        self.lists = order[own[by]]
        edges = torch.searchsorted(tiles, torch.arange(self.tx * self.ty + 1, device=DEV))
        self.first, self.count = edges[:-1], edges[1:] - edges[:-1]
        self.flat = {k: self.g[k].detach().requires_grad_(True) for k in ("u", "v", "a", "b", "c", "o", "rgb")}

    def _batches(self):
        t2 = self.tile * self.tile
        order = torch.argsort(self.count, descending=True)
        lens = self.count[order].cpu().tolist()
        k = 0
        while k < len(lens) and lens[k] > 0:
            m = max(1, (24 << 20) // (lens[k] * t2))
            yield order[k:k + m], lens[k]
            k += m

    def _compose(self, tiles, longest):
        at = torch.arange(longest, device=DEV)
        live = at[None] < self.count[tiles][:, None]
        gid = self.lists[torch.where(live, self.first[tiles][:, None] + at[None], 0)]
        f = {k: t[gid] for k, t in self.flat.items()}
        px = torch.arange(self.tile * self.tile, device=DEV)
        X = (tiles % self.tx * self.tile)[:, None] + px % self.tile
        Y = (tiles // self.tx * self.tile)[:, None] + px // self.tile
        dx, dy = X[:, None] - f["u"][..., None], Y[:, None] - f["v"][..., None]
        power = -0.5 * (f["a"][..., None] * dx * dx + f["c"][..., None] * dy * dy) - f["b"][..., None] * dx * dy
        alpha = (f["o"][..., None] * torch.exp(power.clamp(max=0.0))).clamp(max=0.99)
        alpha = torch.where(live[..., None] & (power <= 0) & (alpha >= 1.0 / 255.0), alpha, torch.zeros((), device=DEV, dtype=torch.float64))
        T = torch.cumprod(1.0 - alpha, 1)
        on = T.detach() >= 1e-4
        before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        w = torch.where(on, alpha * before, torch.zeros((), device=DEV, dtype=torch.float64))
        rgb = torch.einsum("blp,blc->bcp", w, f["rgb"])
        Tf = torch.where(on, T, torch.ones((), device=DEV, dtype=torch.float64)).amin(1)
        inside = (X < self.cam.width) & (Y < self.cam.height)
        return rgb, Tf, X, Y, inside

    def forward(self):
        H, W = self.cam.height, self.cam.width
        img = torch.zeros(3, H, W, dtype=torch.float64, device=DEV)
        T = torch.ones(H, W, dtype=torch.float64, device=DEV)
        with torch.no_grad():
            for tiles, longest in self._batches():
                rgb, Tf, X, Y, ok = self._compose(tiles, longest)
                T[Y[ok], X[ok]] = Tf[ok]
                img[:, Y[ok], X[ok]] = rgb.permute(1, 0, 2)[:, ok]
        return img, T

    def backward(self, dimg):
        """Dense gradients of the raw parameters, and those of (u, v) of the visible Gaussians."""
        for tiles, longest in self._batches():
            rgb, _, X, Y, ok = self._compose(tiles, longest)
            g = torch.zeros_like(rgb)
            g.permute(1, 0, 2)[:, ok] = dimg[:, Y[ok], X[ok]]
            rgb.backward(g)
        zero = lambda t: torch.zeros_like(t) if t.grad is None else t.grad  # noqa: E731
        names = list(self.flat)
        grads = torch.autograd.grad([self.g[k] for k in names], self.leaf, [zero(self.flat[k]) for k in names], allow_unused=True)
        dense = []
        for s, g in zip(self.shapes, grads):
            t = torch.zeros(tuple(s), dtype=torch.float64, device=DEV)
            t[self.ids] = g
            dense.append(t)
        return tuple(dense), zero(self.flat["u"]), zero(self.flat["v"])


def _ssim64(x, y):
    """Per-pixel SSIM, 11 x 11 Gaussian window (sigma 1.5), zero padding."""
    k = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / 4.5)
    k = k / k.sum()
    H, W = x.shape[-2:]

    def blur(t):
        t = F.pad(t, (5, 5, 0, 0))
        t = sum(k[i] * t[..., i:i + W] for i in range(11))
        t = F.pad(t, (0, 0, 5, 5))
        return sum(k[i] * t[..., i:i + H, :] for i in range(11))

    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 1e-4, 9e-4
    return (2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))


def _eq1(img, target, lam=0.2):
    return (1 - lam) * (img - target).abs().mean() + lam * (1 - _ssim64(img, target).mean())


def _step64(params, cam, target, degree, tile):
    e = _Exact64(params, cam, degree, tile)
    img, T = e.forward()
    leaf = img.clone().requires_grad_(True)
    loss = _eq1(leaf, target.double())
    dimg, = torch.autograd.grad(loss, leaf)
    return e, img, T, loss.detach(), dimg, e.backward(dimg)


def _visibility64(boxes, cams):
    """Share of the image covered by each box in each camera.  The box faces turned away from the camera tile its
    silhouette whether or not the near plane cuts it, so the area is the sum over those faces of the face
    clipped by the near plane, projected and clipped by the image rectangle."""
    n_cams, n = len(cams), boxes.shape[0]
    get = lambda f: _t64([f(c) for c in cams])  # noqa: E731
    w2c = get(lambda c: list(c.world_to_cam)).view(-1, 3, 4)
    fx, fy, cx, cy, near = (get(lambda c, k=k: getattr(c, k)) for k in ("fx", "fy", "cx", "cy", "near_plane"))
    W, H = get(lambda c: c.width), get(lambda c: c.height)
    b = boxes.double()
    bit = torch.tensor([[k & 1, (k >> 1) & 1, k >> 2] for k in range(8)], device=DEV)
    corner = torch.where(bit[None].bool(), b[:, None, 3:], b[:, None, :3])
    c = torch.einsum("irk,nck->incr", w2c[:, :, :3], corner) + w2c[:, None, None, :, 3]
    quad = torch.tensor([[0, 2, 6, 4], [1, 3, 7, 5], [0, 1, 5, 4], [2, 3, 7, 6], [0, 1, 3, 2], [4, 5, 7, 6]], device=DEV)
    face = c[:, :, quad]                                            # [cams, cells, 6, 4, 3]
    normal = torch.linalg.cross(face[..., 1, :] - face[..., 0, :], face[..., 3, :] - face[..., 0, :])
    centre = c.mean(2)[:, :, None]
    outward = torch.sign((normal * (face.mean(3) - centre)).sum(-1, keepdim=True)) * normal
    away = (outward * face.mean(3)).sum(-1) > 0
    poly, ok = face.reshape(-1, 4, 3), torch.ones(n_cams * n * 6, 4, dtype=torch.bool, device=DEV)

    def clip(poly, ok, dist):
        """Sutherland-Hodgman by dist >= 0; empty slots repeat a vertex, which adds no area."""
        k = poly.shape[1]
        nxt, dn = poly.roll(-1, 1), dist.roll(-1, 1)
        cross = (dist >= 0) != (dn >= 0)
        t = torch.where(cross, dist / torch.where(cross, dist - dn, torch.ones_like(dist)), torch.zeros_like(dist))
        pts = torch.stack([poly, poly + t[..., None] * (nxt - poly)], 2).reshape(-1, 2 * k, poly.shape[2])
        use = torch.stack([dist >= 0, cross], 2).reshape(-1, 2 * k)
        order = torch.argsort((~use).to(torch.int8), dim=1, stable=True)[:, :k + 1]
        pts = torch.gather(pts, 1, order[..., None].expand(-1, -1, pts.shape[2]))
        use = torch.gather(use, 1, order)
        last = (use.sum(1, keepdim=True) - 1).clamp(min=0)
        fill = torch.gather(pts, 1, last[..., None].expand(-1, 1, pts.shape[2]))
        return torch.where(use[..., None], pts, fill), ok[:, :1].expand(-1, k + 1) & use.any(1, keepdim=True)

    per = lambda t: t[:, None, None].expand(n_cams, n, 6).reshape(-1)  # noqa: E731
    poly, ok = clip(poly, ok, poly[..., 2] - per(near)[:, None])
    z = torch.where(ok, poly[..., 2], torch.ones_like(poly[..., 2])).clamp(min=1e-6)
    p = torch.stack([per(fx)[:, None] * poly[..., 0] / z + per(cx)[:, None], per(fy)[:, None] * poly[..., 1] / z + per(cy)[:, None]], 2)
    for axis, bound, sign in ((0, per(W) * 0 - 0.5, 1), (0, per(W) - 0.5, -1), (1, per(H) * 0 - 0.5, 1), (1, per(H) - 0.5, -1)):
        p, ok = clip(p, ok, sign * (p[..., axis] - bound[:, None]))
    q = p.roll(-1, 1)
    area = 0.5 * (p[..., 0] * q[..., 1] - p[..., 1] * q[..., 0]).sum(1).abs() * ok[:, 0]
    area = (area.view(n_cams, n, 6) * away).sum(2)
    return area / (W * H)[:, None]


def _appearance64(img, target, emb, params, grad, lam=0.2):
    leaves = [t.double().requires_grad_(grad) for t in (img, emb, params)]
    x, e, flat = leaves
    layers, off = [], 0
    for c, o in AP.LAYERS:
        layers.append((flat[off:off + 9 * c * o].view(o, c, 3, 3), flat[off + 9 * c * o:off + 9 * c * o + o]))
        off += 9 * c * o + o
    H, W = x.shape[1:]
    h, w = H // 32, W // 32
    low = F.avg_pool2d(x[None, :, :32 * h, :32 * w], 32)
    t = F.conv2d(torch.cat([low, e.view(1, 64, 1, 1).expand(1, 64, h, w)], 1), *layers[0], padding=1)
    for k in range(1, 5):
        t = torch.relu(F.conv2d(F.pixel_shuffle(t, 2), *layers[k], padding=1))
    t = F.interpolate(t, size=(H, W), mode="bilinear", align_corners=False)
    M = F.conv2d(torch.relu(F.conv2d(t, *layers[5], padding=1)), *layers[6], padding=1)[0]
    y = target.double()
    loss = (1 - lam) * (x * M - y).abs().mean() + lam * (1 - _ssim64(x, y).mean())
    return loss.detach().view(1), M.detach(), torch.autograd.grad(loss, leaves) if grad else None


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        p, cam, target = _scene(case, seed)
        e, img, _, loss, _, (grads, du, dv) = _step64(p, cam, target, case["degree"], case["tile"])
        out = {"image": img, "loss": loss, "grads": grads}
        if case["stats"]:
            out["accum"] = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
            out["accum"][e.ids] = torch.sqrt((0.5 * case["w"] * du) ** 2 + (0.5 * case["h"] * dv) ** 2)
            out["count"] = None
        return out
    if kind == "batch":
        outs, losses, dimgs, grads = [], [], [], []
        cells, cams, targets = _batch_scene(case, seed)
        tiles = [st.tile_size for st in _settings(case["tiles"], len(cells))]
        for p, cam, target, tile in zip(cells, cams, targets, tiles):
            _, img, T, loss, dimg, (g, _, _) = _step64(p, cam, target, case["degree"], tile)
            outs.append((img, T, None))
            losses.append(loss)
            dimgs.append(dimg)
            grads.append(g)
        return {"outs": outs, "loss": losses, "grad_image": dimgs, "grads": grads}
    if kind == "views":
        cells, cams = _views_scene(case, seed)
        whole = [torch.cat(t) for t in zip(*cells)]
        return [(*_Exact64(whole, cam, case["degree"], 16).forward(), None) for cam in cams]
    if kind == "appearance":
        s = prepare(case, seed)
        loss, M, g = _appearance64(s["img"], s["target"], s["model"].embeddings[1], s["model"].params, case["grad"])
        return {"loss": loss, "grad_img": g[0], "grad_embedding": g[1], "grad_params": g[2]} if case["grad"] else {"loss": loss, "map": M}
    if kind == "adam":
        s = prepare(case, seed)
        a = s["adam"].s
        f32 = lambda v: float(np.float32(v))  # noqa: E731
        b1, b2, t = f32(a.beta1), f32(a.beta2), s["adam"].t + 1
        lr = [torch.tensor(f32(v), dtype=torch.float64, device=DEV) for v in (a.lr_means, a.lr_log_scales, a.lr_quats, a.lr_opacity)]
        rest = torch.full(((case["degree"] + 1) ** 2, 1), f32(a.lr_sh_rest), dtype=torch.float64, device=DEV)
        rest[0] = f32(a.lr_sh_dc)
        out = {"params": [], "m": [], "v": []}
        for p, g, m, v, step in zip(s["params"], s["grads"], s["adam"].m, s["adam"].v, [*lr, rest]):
            g = g.double()
            m, v = b1 * m.double() + (1 - b1) * g, b2 * v.double() + (1 - b2) * g * g
            out["params"].append(p.double() - step * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + f32(a.eps)))
            out["m"].append(m)
            out["v"].append(v)
        out["m"], out["v"] = tuple(out["m"]), tuple(out["v"])
        return out
    if kind == "densify":
        p, m, v, accum, count, normals = _densify_scene(case, seed)
        d = OP.DensifySettings(scene_extent=10.0)
        f32 = lambda t: torch.tensor(t, dtype=torch.float32, device=DEV)  # noqa: E731
        ln16 = f32(math.log(1.6))
        grad = torch.where(count > 0, accum / count.clamp(min=1), torch.zeros_like(accum))
        act = torch.where(grad >= f32(d.grad_threshold),
                          torch.where(p[1].amax(1) > f32(math.log(d.percent_dense * d.scene_extent)), 3, 2), 1)
        act = torch.where(p[3] < f32(math.log(d.min_opacity / (1 - d.min_opacity))), torch.zeros_like(act), act)
        biggest = f32(math.log(d.max_world_scale_frac * d.scene_extent))
        fits = torch.where(act == 3, (p[1] - ln16).amax(1), p[1].amax(1)) <= biggest
        emit = torch.where(fits, torch.tensor([0, 1, 2, 2], device=DEV)[act], 0)
        src = torch.repeat_interleave(torch.arange(case["n"], device=DEV), emit)
        nth = torch.arange(src.numel(), device=DEV) - (torch.cumsum(emit, 0) - emit)[src]
        split, fresh = act[src] == 3, (act[src] == 3) | (nth == 1)
        new = [t[src].double() for t in p]
        shift = torch.einsum("nij,nj->ni", _rotation(new[2]), torch.exp(new[1]) * normals[src, nth].double())
        new[0] = torch.where(split[:, None], new[0] + shift, new[0])
        new[1] = torch.where(split[:, None], (p[1][src] - ln16).double(), new[1])
        zero = lambda t: torch.where(fresh.view(-1, *[1] * (t.dim() - 1)), torch.zeros((), device=DEV), t[src]).double()  # noqa: E731
        return {"params": tuple(new), "m": tuple(zero(t) for t in m), "v": tuple(zero(t) for t in v)}
    if kind == "merge":
        cells, regions = _expanded_cells(case, seed)
        keep = [(c[0][:, 0] >= x0) & (c[0][:, 0] < x1) & (c[0][:, 2] >= z0) & (c[0][:, 2] < z1)
                for c, (x0, x1, z0, z1) in zip(cells, regions)]
        return tuple(torch.cat([c[j][k] for c, k in zip(cells, keep)]).double() for j in range(5))
    if kind == "select":
        cells, _ = _expanded_cells(case, seed, points_only=True)
        boxes = torch.stack([torch.cat([c.amin(0), c.amax(0)]) for c in cells]).double()
        boxes[:, 1] = 0.0
        return {"boxes": boxes, "visibility": _visibility64(boxes, PT.camera_table(_selection_cameras(case, seed))), "selected": None}
    s = prepare(case, seed)
    x, y = s["img"].double().view(3, -1), s["target"].double().view(3, -1)
    mx, my = x.mean(1, keepdim=True), y.mean(1, keepdim=True)
    A = torch.linalg.solve((x - mx) @ (x - mx).T, (x - mx) @ (y - my).T).T
    b = (my - A @ mx)[:, 0]
    fit = (A @ x + b[:, None]).clamp(0.0, 1.0)
    shape = (3, case["h"], case["w"])
    ssim = _ssim64(fit.view(shape), y.view(shape)).mean()
    return torch.cat([-10.0 * torch.log10((fit - y).square().mean()).view(1), ssim.view(1), A.reshape(-1), b])
