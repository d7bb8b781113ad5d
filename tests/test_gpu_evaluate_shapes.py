"""The corrected evaluation at image sizes and addresses that leave its 16-byte loads (pixel counts that are no
multiple of 4, images off a 16-byte boundary) and at sizes around one block's share, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import evaluate as OE
from paper_2402_17427_gb300 import rasterize as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    import oracle
    oracle.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("H,W,offset", [(5, 7, 0), (32, 32, 0), (32, 32, 1), (33, 31, 0), (17, 61, 3), (128, 904, 2),
                                        (601, 777, 0)])
def test_metrics_at_any_size_and_alignment(H, W, offset):
    rng = np.random.default_rng(H * W + offset)
    y = rng.uniform(0, 1, (3, H, W)).astype(np.float32)
    x = np.clip(0.8 * y[[1, 0, 2]] + 0.1 + 0.05 * rng.standard_normal(y.shape), 0, 1).astype(np.float32)

    def put(a):
        buf = torch.empty(a.size + 4, dtype=torch.float32, device="cuda")
        t = buf[offset:offset + a.size].view(a.shape)
        t.copy_(torch.from_numpy(a))
        return t
    out = R.color_corrected_metrics(put(x), put(y)).cpu().numpy().astype(np.float64)
    c, A, b = OE.color_correct(x, y)
    import oracle
    assert abs(out[0] - OE.psnr(c, y)) <= 1e-3
    assert abs(out[1] - oracle.ssim(c, y)) <= 2e-5
    assert np.allclose(out[2:11].reshape(3, 3), A, rtol=1e-4, atol=1e-5)
    assert np.allclose(out[11:14], b, rtol=1e-4, atol=1e-5)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3e18])
def test_infinite_and_huge_targets(value):
    """One target pixel that is infinite, NaN or so large that the sums pass FP32's range: what plain FP64 sums of the
    same fit give (a NaN fit is clipped to 0, and the squared error follows)."""
    x = torch.rand(3, 65, 260, device="cuda")
    y = torch.rand(3, 65, 260, device="cuda")
    y[1] = y[1] if not np.isfinite(value) else value * (0.5 + 0.5 * y[1])
    if not np.isfinite(value):
        y[1, 7, 9] = value
    out = R.color_corrected_metrics(x, y).cpu().numpy().astype(np.float64)
    if np.isnan(value):
        assert out[0] == np.inf and np.isnan(out[12])     # a squared error that is no positive number
    elif np.isinf(value):
        assert np.isnan(out[12]) and out[0] == -np.inf
    else:
        d = y[1].double() - 1.0           # the fit is far above 1 everywhere, so it is clipped to 1
        rest = sum(float((y[c].double() - y[c].double().mean()).square().sum()) for c in (0, 2))
        mse = (float(d.square().sum()) + rest) / y.numel()
        assert abs(out[0] + 10.0 * np.log10(mse)) <= 1e-3
        assert np.isfinite(out).all()
