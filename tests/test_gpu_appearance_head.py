"""The head of the appearance network at the edges of its tiles (8 rows x 30 columns of outputs), and the order in
which its forward convolutions add up their taps.

Conv5's sums gate the gradient by their sign and conv6's set the sign of the L1 term, so a sum within rounding of
zero must come out the same whatever the layout of the pass: taps in row-major order, the channels of a tap in
eights.  The weights below make the order visible: 2^-60 at tap (0, 0) is lost in the 1 that channel 0 of tap (1, 1)
adds, which channel 8 takes away again (exactly 0), while 2^-60 at tap (2, 2) comes after them and stays."""
import numpy as np
import pytest
import torch

from paper_2402_17427_gb300 import appearance as AP
from test_gpu_appearance import _compare

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -60


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    import oracle
    oracle.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("W,H,seed", [(61, 33, 11), (91, 129, 12), (60, 64, 13)])
def test_tile_edges_match_oracle(W, H, seed):
    # a last tile of one column and one row, the same with several tiles, whole tiles only
    _compare(W, H, seed)


def _cancelling(layer):
    """Output 0: 2^-60 before the pair that cancels; output 1: after it."""
    layer[0, 0, 0, 0] = TINY
    layer[1, 0, 2, 2] = TINY
    layer[:2, 0, 1, 1] = 1.0
    layer[:2, 8, 1, 1] = -1.0


SIZES = [(32, 32), (61, 33), (91, 129), (60, 64)]


@pytest.mark.parametrize("W,H", SIZES)
def test_conv6_adds_taps_in_order(W, H):
    model = AP.AppearanceModel(1)
    model.params.zero_()
    layers = AP.layer_views(model.params)
    layers[5][1].fill_(1.0)                     # conv5: 1 everywhere
    _cancelling(layers[6][0])
    img = torch.full((3, H, W), 0.5, device="cuda")
    M = model.loss(img, torch.zeros_like(img), 0, 0.2, grad=False, want_map=True)["map"].cpu().numpy()
    assert not M[0].any() and not M[2].any()
    want = np.zeros((H, W), np.float32)
    want[:-1, :-1] = TINY
    assert np.array_equal(M[1], want)


@pytest.mark.parametrize("W,H", SIZES)
def test_conv5_units_keep_their_sign(W, H):
    model = AP.AppearanceModel(1)
    model.params.zero_()
    layers = AP.layer_views(model.params)
    layers[4][1].fill_(1.0)                     # the features that are up-sampled: 1 everywhere
    _cancelling(layers[5][0])
    layers[6][0][:, :2, 1, 1] = 1.0
    layers[6][1].fill_(1.0)                     # M = 1
    img = torch.full((3, H, W), 0.5, device="cuda")
    out = model.loss(img, torch.zeros_like(img), 0, 0.2)
    dw, db = [t.cpu().numpy() for t in AP.layer_views(out["grad_params"])[5]]
    assert db[0] == 0.0 and not dw[0].any()     # a unit at exactly 0 is off
    # unit 1 is on but at the last row and column: dL/dunit = 3 x 0.5 x (1 - lambda) / (3 H W)
    assert db[1] == pytest.approx(0.8 * 0.5 * (W - 1) * (H - 1) / (H * W), rel=1e-5)
