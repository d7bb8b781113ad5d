"""Visibility of needles: a Gaussian is drawn if the determinant of its 2D covariance is positive in FP32, the product
A C entering unrounded (fused).  The camera's first two rows are equal, so that A = B + dilation = C, and the dilation
is lost in A >= 2^24: the determinant is the rounding error of A^2, known exactly."""
import numpy as np
import pytest

from _gpu import read_state, run_forward
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    import torch
    assert torch.cuda.is_available()


@pytest.mark.parametrize("degree", [0, 3])
def test_visible_by_the_fused_determinant(degree):
    n, f = 2000, np.float32(5000.0)
    rng = np.random.default_rng(degree)
    z = rng.uniform(0.25, 1.0, n).astype(np.float32)
    means = np.stack([0 * z, 0 * z, z], 1)
    ls = np.tile(np.array([0.0, -20.0, -20.0], np.float32), (n, 1))       # one unit axis: exp(0) = 1
    quats = np.tile(np.array([1.0, 0.0, 0.0, 0.0], np.float32), (n, 1))
    sh = rng.standard_normal((n, (degree + 1) ** 2, 3)).astype(np.float32)
    g = scenes.Gaussians(means, ls, quats, np.full(n, -1.0, np.float32), sh, degree)
    R = np.array([[1, 0, 0], [1, 0, 0], [0, 0, 1]], np.float32)
    cam = scenes.Camera(64, 48, float(f), float(f), 31.5, 23.5, R, np.zeros(3, np.float32), np.zeros(3, np.float32), 0.2)
    t = f * (np.float32(1.0) / z)
    A = t * t
    assert A.min() >= 2 ** 24 and np.array_equal(A + np.float32(0.3), A)
    det = A.astype(np.float64) ** 2 - (A * A).astype(np.float64)          # exact: 48 bits
    ras, _, out = run_forward(g, cam)
    state = read_state(ras, g, cam)
    assert 0.3 * n < (det > 0).sum() < 0.7 * n
    assert np.array_equal(state["touched"] > 0, det > 0)
    assert np.array_equal(state["proj"][:, 2] != 0, det > 0)              # a record for each, and for no other
    assert np.isfinite(out["image"]).all()
