"""Camera visibility over boxes that take the silhouette path (in front of the near plane) and the general one
(cut by it, flat, behind, around the camera), mixed within a block; and airspace boxes at cell sizes and offsets
around the 16-byte loads and the blocks' share of 4,096 points.  Against the FP64 oracle."""
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


@pytest.mark.parametrize("n_cells,n_cams", [(1, 1), (7, 37), (16, 40), (130, 3)])
def test_visibility_of_any_box(n_cells, n_cams):
    rng = np.random.default_rng(n_cells)
    lo = rng.uniform([-300, -20, -300], [300, 60, 300], (n_cells, 3))
    ext = rng.uniform(0.5, 120, (n_cells, 3))
    for k in range(n_cells):          # some flat along an axis, one a point
        if k % 5 == 3:
            ext[k, k % 3] = 0.0
    boxes = np.concatenate([lo, lo + ext], 1).astype(np.float32)
    cams = []
    for i in range(n_cams):
        W, H = ((64, 48), (1920, 1080), (333, 777))[i % 3]
        eye = rng.uniform([-400, 5, -400], [400, 200, 400]) if i % 4 else lo[i % n_cells] + 0.5 * ext[i % n_cells]
        cams.append(scenes.camera_from_forward(eye, scenes.yaw_pitch_forward(rng.uniform(0, 2 * math.pi),
                                                                             rng.uniform(-1.5, 0.3)), W, H))
    vis, sel = PT.camera_visibility(torch.from_numpy(boxes).cuda(), cams, 0.25)
    ref = OP.visibility_matrix(boxes.astype(np.float64), cams)
    assert sel.dtype == torch.bool and vis.shape == sel.shape == (n_cams, n_cells)
    assert np.abs(vis.cpu().numpy() - ref).max() <= 1e-6
    settled = np.abs(ref - 0.25) > 1e-9
    assert np.array_equal(sel.cpu().numpy()[settled], OP.select(ref, 0.25)[settled])


@pytest.mark.parametrize("sizes", [(1,), (2, 3, 5, 6), (4095, 4096, 4097), (8193, 1, 12289)])
def test_airspace_boxes_at_block_edges(sizes):
    rng = np.random.default_rng(sum(sizes))
    pts = rng.normal(0, 100, (sum(sizes), 3)).astype(np.float32)
    offs = np.concatenate([[0], np.cumsum(sizes)]).tolist()
    out = PT.airspace_boxes(torch.from_numpy(pts).cuda(), offs, ground_y=1.5).cpu().numpy()
    for k in range(len(sizes)):
        assert np.array_equal(out[k], OP.airspace_box(pts[offs[k]:offs[k + 1]], 1.5).astype(np.float32)), k
