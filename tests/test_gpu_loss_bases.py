"""The values that the SSIM moments are taken relative to: even images at any level lose no digits to the level, and a
highlight among the pixels that a base is chosen from costs nobody else any.

Bounds (u = 2^-24).  Where an image is even, every difference from a base is 0, so variances and covariance are exactly 0
and S errs by the rounding of the means alone: 8 u.  Windows that hold the zero padding or a highlight have variances of
the values' own size, and S errs by a few times 148 u: 4e-5; 15 times that if the four pixels a base is chosen from
are all bright and have only 0.15 of the window's weight."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_17427_gb300 import rasterize as R
from test_gpu_loss_outliers import U, H, W, _check, _noisy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    oracle.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("h,w", [(96, 96), (75, 100), (33, 41), (8, 11), (3, 5), (1, 1)])
@pytest.mark.parametrize("a,b", [(0.9, 0.6), (3.0, 2.0), (0.3, 0.7), (-0.5, -0.6), (30.0, 0.1)])
def test_even_images(h, w, a, b):
    x, y = np.full((3, h, w), a, np.float32), np.full((3, h, w), b, np.float32)
    loss, _ = R.LossL1DSSIM(1.0)(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    want, _ = oracle.loss_l1_dssim(x.astype(np.float64), y.astype(np.float64), 1.0)
    border = 1.0 - max(0, h - 10) * max(0, w - 10) / (h * w)
    assert abs(float(loss) - want) <= 8 * U + 4e-5 * border


@pytest.mark.parametrize("size,loud", [(1, 4e-5), (3, 4e-5), (4, 6e-4)])
@pytest.mark.parametrize("row,col", [(2, 2), (3, 13), (18, 29), (26, 5)])
def test_highlights_among_the_bases(row, col, size, loud):
    """Windows are based on columns and rows 2 .. 5 of every eight: from one bright pixel of them to all."""
    x, y = _noisy(0.02, 8 * row + col)
    odd = np.zeros((H, W), bool)
    for r in range(row, H, 32):
        for c in range(col, W, 32):
            odd[r:r + size, c:c + size] = True
    x[:, odd] = 10.0
    y[:, odd] = 7.0
    _check(x, y, odd, 1.1 * 0.02, loud)
