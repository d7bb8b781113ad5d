"""Dense gradients: every row of a culled Gaussian is zero, every row of a visible one is what the adjoint writes, and
nothing beside the arrays is touched, at run edges, odd sizes, addresses off a 16-byte boundary and several tile sizes."""
import pytest
import torch

from paper_2402_17427_gb300 import batch as BT
from paper_2402_17427_gb300 import rasterize as R
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu
GUARD = 12


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


def _cell(n, degree, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    return [8.0 * rnd(n, 3), -2.5 + 0.5 * rnd(n, 3), rnd(n, 4), rnd(n), 0.3 * rnd(n, (degree + 1) ** 2, 3)]


def _arrays(cell, degree, shift):
    """NaN-filled gradient arrays inside NaN-filled buffers; those without 16-byte rows start `shift` floats off."""
    bufs, views = [], []
    for k, t in enumerate(cell):
        o = 4 + (shift if k in (0, 1, 3) or (k == 4 and degree in (0, 2)) else 0)
        b = torch.full((t.numel() + 2 * GUARD,), float("nan"), device="cuda")
        bufs.append((b, o))
        views.append(b[o:o + t.numel()].view(t.shape))
    return bufs, tuple(views)


@pytest.mark.parametrize("tiles", [(16,), (32,), (8, 16), (16, 8, 32)])
@pytest.mark.parametrize("n,degree,shift", [(1, 0, 1), (3, 1, 3), (511, 2, 1), (513, 3, 2), (5001, 0, 3), (70_001, 3, 1)])
def test_rows(tiles, n, degree, shift):
    cells = [_cell(n + 7 * k, degree, n + k) for k in range(len(tiles))]
    cam = scenes.look_at((0.0, 0.0, -9.0), (0.0, 0.0, 0.0), 150, 90, fx=120.0)
    cams = [cam] * len(tiles)
    br = BT.BatchRasterizer([R.RasterSettings(tile_size=t) for t in tiles])
    keys = torch.empty(sum(c[0].shape[0] for c in cells), 4, device="cuda")
    br.forward(cells, degree, cams, key_inputs=keys)
    outs = br.forward(cells, degree, cams)
    dLs = [torch.randn_like(o[0]) for o in outs]
    made = [_arrays(c, degree, shift) for c in cells]
    br.backward(cells, degree, cams, outs, dLs, grads=[v for _, v in made])
    _, ids = br.read_state(cells, degree, cams)
    ranges, _ = br.read_state(cells, degree, cams)
    seen = torch.zeros(keys.shape[0], dtype=torch.bool, device="cuda")
    seen[torch.from_numpy(ids[:int(ranges[:, 1].max())].astype("int64")).cuda()] = True
    at = 0
    for c, (bufs, views) in zip(cells, made):
        mine = seen[at:at + c[0].shape[0]]
        at += c[0].shape[0]
        for (b, o), v in zip(bufs, views):
            assert torch.isfinite(v).all()
            assert (v[~mine] == 0).all()
            assert torch.isnan(b[:o]).all() and torch.isnan(b[o + v.numel():]).all()
        if n > 500:
            assert (views[0][mine] != 0).any()
