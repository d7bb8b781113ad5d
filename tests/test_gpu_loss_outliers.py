"""Loss, its gradient and the evaluation's SSIM on images with values unlike their surroundings: single bright pixels
(the renderer's colours have no upper bound) at the middles of the 32 x 32 tiles, and an image half dark, half bright.
Away from them nothing may lose digits to them.

Bounds (u = 2^-24).  A window sum of squares takes 22 additions, a product and the weights' rounding, so with every
value at most m it errs by 25 u m^2, a squared mean by 49 u m^2; the denominator's variances by 148 u m^2 together,
relative to C2 = 9e-4 at least: rho = 148 u m^2 / C2.  S then errs by 2 rho, and the SSIM part of dL/dx, formed of three
terms of size 2 m k / C2 (k = 1 / (3 H W)) with at most 10 rho between them, by 20 m k rho / C2.  Windows that hold an
outlier v have variances of v^2's size, so their S errs by a few times 148 u: 4e-5.  Bright values of 10 % noise have
variances of v^2 / 300 in each image: 2 x 148 u x 1.1^2 x 150 = 3.2e-3."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_17427_gb300 import rasterize as R

pytestmark = pytest.mark.gpu

H, W = 75, 100
U = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    oracle.build()
    assert torch.cuda.is_available()


def _near(mask, r):
    """Pixels within r (Chebyshev) of a set one."""
    out = np.zeros_like(mask)
    for y, x in zip(*np.nonzero(mask)):
        out[max(0, y - r):y + r + 1, max(0, x - r):x + r + 1] = True
    return out


def _middles():
    m = np.zeros((H, W), bool)
    for oy in range(0, H, 32):
        for ox in range(0, W, 32):
            m[min(oy + 16, H - 1), min(ox + 16, W - 1)] = True
    return m


def _noisy(level, seed):
    rng = np.random.default_rng(seed)
    return [(level * (1.0 + 0.1 * rng.uniform(-1, 1, (3, H, W)))).astype(np.float32) for _ in range(2)]


def _check(x, y, odd, m, loud):
    loss, grad = R.LossL1DSSIM(1.0)(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    want, g = oracle.loss_l1_dssim(x.astype(np.float64), y.astype(np.float64), 1.0)
    rho, k = 148 * U * m * m / 9e-4, 1.0 / (3 * H * W)
    quiet = ~_near(odd, 10)                   # no window of a window holds one of them
    assert quiet.sum() > 500
    err = np.abs(grad.cpu().numpy() - g)[:, quiet].max()
    assert err <= 20 * m * k * rho / 9e-4, err / k
    assert abs(float(loss) - want) <= 2 * rho + loud * _near(odd, 5).mean() + 4 * U


@pytest.mark.parametrize("level", [0.02, 0.2])
@pytest.mark.parametrize("middle", [1.0, 3.0, 10.0, 100.0, 1000.0])
def test_bright_pixels_at_tile_middles(level, middle):
    x, y = _noisy(level, int(middle))
    odd = _middles()
    x[:, odd] = middle
    _check(x, y, odd, 1.1 * level, 4e-5)


@pytest.mark.parametrize("dark,bright", [(0.02, 1.0), (0.2, 10.0)])
def test_half_bright_image(dark, bright):
    x, y = _noisy(dark, 5)
    for a in (x, y):
        a[:, :, 60:] *= bright / dark         # the tile of columns 32 .. 63 is bright on its right
        a[:, :, :10] *= bright / dark
    odd = np.zeros((H, W), bool)
    odd[:, 60:] = odd[:, :10] = True
    _check(x, y, odd, 1.1 * dark, 3.2e-3)


def test_l1_of_the_values_as_they_came():
    """lambda = 0: |x - y| is exact in FP32 for neighbours; the sums are FP32 within a warp (32 x 8 values: 13 roundings)."""
    x, _ = _noisy(0.2, 9)
    x[:, _middles()] = 1000.0
    y = np.nextafter(x, np.float32(2000.0))
    loss, _ = R.LossL1DSSIM(0.0)(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    want = np.abs(x.astype(np.float64) - y).mean()
    assert abs(float(loss) - want) <= 16 * U * want


def test_evaluation_with_highlights():
    x, y = _noisy(0.02, 3)
    odd = _middles()
    x[:, odd] = y[:, odd] = 1.0
    out = R.color_corrected_metrics(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()).cpu().numpy().astype(np.float64)
    A, b = out[2:11].reshape(3, 3), out[11:14]
    c = np.clip(np.einsum("ij,jhw->ihw", A, x.astype(np.float64)) + b[:, None, None], 0.0, 1.0)
    m = 0.05                                  # of the corrected image away from the highlights
    assert c[:, ~odd].max() <= m
    # the corrected image itself is rounded: 4 u of 1 against a deviation of at least C2
    rho = 148 * U * m * m / 9e-4
    assert abs(out[1] - oracle.ssim(c, y.astype(np.float64))) <= 2 * rho + 4e-5 * _near(odd, 5).mean() + 8 * U
