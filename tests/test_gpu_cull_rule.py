"""The cull on means and log-scales alone against the projection of every Gaussian (which a render that records its
decision inputs takes): the same tile lists, whatever the sizes, the segments' alignment and the values."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2402_17427_gb300 import batch as BT
from paper_2402_17427_gb300 import rasterize as R
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


def _cell(n, seed, spread=40.0):
    """A cloud around and behind the camera, with scales from 1e-4 to e^4, and a few values no scene has."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    means, ls = spread * rnd(n, 3), -3.0 + 2.0 * rnd(n, 3)
    odd = torch.randint(0, n, (max(1, n // 50), 6), device="cuda", generator=g)
    for k, v in enumerate((float("nan"), float("inf"), -float("inf"), 1e20, 1e-30, 0.0)):
        means[odd[:, k], k % 3] = v
    for k, v in enumerate((float("nan"), float("inf"), -float("inf"), 88.0, -200.0, 5.0)):
        ls[odd[:, 5 - k], k % 3] = v
    return [means, ls, rnd(n, 4), rnd(n), rnd(n, 1, 3)]


def _lists(br, cells, cams, keys):
    outs = br.forward(cells, 0, cams, key_inputs=keys)
    ranges, ids = br.read_state(cells, 0, cams)
    return ranges, ids[:int(ranges[:, 1].max(initial=0))], [o[0].clone() for o in outs]


@pytest.mark.parametrize("sizes,cx", [((1,), None), ((511,), None), ((512,), None), ((513,), None), ((4097,), 1e4),
                                      ((4097,), -700.25), ((300, 1, 513, 777), None), ((1_300_003,), None),
                                      ((700_001, 650_002), None)])
def test_lists_do_not_depend_on_the_cull(sizes, cx):
    cells = [_cell(n, 31 * n + k) for k, n in enumerate(sizes)]
    cam = scenes.look_at((0.0, 0.0, -6.0), (0.0, 0.0, 0.0), 176, 112, fx=150.0)
    if cx is not None:
        cam = dataclasses.replace(cam, cx=cx)
    cams = [cam] * len(cells)
    total = sum(sizes)
    keys = torch.empty(total, 4, device="cuda")
    br = BT.BatchRasterizer([R.RasterSettings() for _ in cells], pair_capacity=1 << 25)
    a, b = _lists(br, cells, cams, keys), _lists(br, cells, cams, None)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for x, y in zip(a[2], b[2]):
        assert torch.equal(torch.nan_to_num(x), torch.nan_to_num(y))
