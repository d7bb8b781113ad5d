"""Boxes of which nothing is in the image have visibility exactly 0 and are not selected at threshold 0, as in the FP64
oracle's clipping: beside, above and below the image, cut by the near plane or not, and boxes without an area (points,
lines, a plane seen edge on)."""
import math

import numpy as np
import pytest
import torch

from oracle import partition as OP
from paper_2402_17427_gb300 import partition as PT
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


def _visibility(boxes, cams):
    vis, sel = PT.camera_visibility(torch.from_numpy(boxes).cuda(), cams, 0.0)
    return vis.cpu().numpy(), sel.cpu().numpy()


@pytest.mark.parametrize("near", [0.2, 20.0])
def test_nothing_of_the_box_in_the_image(near):
    rng = np.random.default_rng(int(near))
    lo = rng.uniform([-300, -20, -300], [300, 60, 300], (64, 3))
    boxes = np.concatenate([lo, lo + rng.uniform(0.5, 150, lo.shape)], 1).astype(np.float32)
    cams = []
    for i in range(60):
        eye = rng.uniform([-400, 5, -400], [400, 200, 400])
        c = scenes.camera_from_forward(eye, scenes.yaw_pitch_forward(rng.uniform(0, 2 * math.pi), rng.uniform(-1.5, 0.3)),
                                       *((64, 48), (1920, 1080), (333, 777))[i % 3])
        c.near = near
        cams.append(c)
    vis, sel = _visibility(boxes, cams)
    ref = OP.visibility_matrix(boxes.astype(np.float64), cams)
    outside = ref == 0.0
    assert outside.mean() > 0.3 and (~outside).sum() > 100
    assert not vis[outside].any() and not sel[outside].any()
    assert np.abs(vis - ref).max() <= 1e-6 and sel[ref > 1e-9].all()


def test_beside_the_image_in_front_of_the_camera():
    # camera coordinates = world coordinates; the image spans |x| <= z / 2, |y| <= z / 2 and half a pixel
    cam = scenes.Camera(64, 64, 64.0, 64.0, 31.5, 31.5, np.eye(3, dtype=np.float32), np.zeros(3, np.float32),
                        np.zeros(3, np.float32), 0.2)
    rng = np.random.default_rng(1)
    boxes = []
    for sx, sy in ((1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (1, -1), (-1, 1), (-1, -1)):
        for _ in range(100):
            z0 = rng.uniform(0.5, 50)
            z1 = z0 + rng.uniform(0.1, 50)
            # its lower or upper side along each chosen axis beyond the image everywhere; the other axis anywhere
            c = [rng.uniform(-60, 60), rng.uniform(-60, 60)]
            e = [rng.uniform(0.1, 80), rng.uniform(0.1, 80)]
            for a, s in enumerate((sx, sy)):
                if s:
                    c[a] = s * (0.51 * z1 + rng.uniform(0.01, 5) + e[a] / 2)
            boxes.append([c[0] - e[0] / 2, c[1] - e[1] / 2, z0, c[0] + e[0] / 2, c[1] + e[1] / 2, z1])
    vis, sel = _visibility(np.array(boxes, np.float32), [cam])
    assert not vis.any() and not sel.any()


def test_boxes_without_an_area():
    cam = scenes.Camera(64, 64, 64.0, 64.0, 31.5, 31.5, np.eye(3, dtype=np.float32), np.zeros(3, np.float32),
                        np.zeros(3, np.float32), 0.2)
    rng = np.random.default_rng(2)
    boxes = []
    for k in range(300):
        lo = rng.uniform([-3, -3, 1], [3, 3, 9])
        ext = rng.uniform(0.1, 4, 3)
        if k % 4 == 0:
            ext[:] = 0                          # a point
        elif k % 4 == 1:
            ext[[k % 3, (k + 1) % 3]] = 0       # a line
        else:
            lo[k % 2], ext[k % 2] = 0, 0        # a plane through the camera
        boxes.append(np.concatenate([lo, lo + ext]))
    vis, sel = _visibility(np.array(boxes, np.float32), [cam])
    ref = OP.visibility_matrix(np.array(boxes, np.float32).astype(np.float64), [cam])
    assert np.abs(vis).max() <= 1e-12 and np.array_equal(sel, ref > 0.0)
