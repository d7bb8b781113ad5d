"""Several renders through one Rasterizer before their backward passes: each gradient is that of its own render,
whatever the later ones left in the workspace (another scene, size, Gaussian count or layout)."""
import pytest
import torch

from paper_2402_17427_gb300 import rasterize as R
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


class Mine(R.Rasterizer):      # takes the node written in Python
    pass


def _scene(n, w, h, degree, seed):
    g, cam, _ = scenes.tiny_scene(n=n, width=w, height=h, degree=degree, seed=seed)
    weight = torch.rand(3, h, w, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
    return [p.requires_grad_(True) for p in R.to_device(g)], g.sh_degree, cam, weight


def _close(a, b):      # sums of FP32 atomics in another order
    for x, y in zip(a, b):
        assert torch.allclose(x, y, rtol=1e-4, atol=1e-5 * float(y.abs().max()) + 1e-12)


@pytest.mark.parametrize("kind", [R.Rasterizer, Mine])
@pytest.mark.parametrize("second", [(150, 48, 40, 2), (700, 96, 80, 3), (40, 33, 17, 0)])
def test_backward_after_another_forward(kind, second):
    a, b = _scene(150, 48, 40, 2, 9), _scene(*second, 10)
    want = [torch.autograd.grad((R.rasterize(*p, d, cam, kind()) * w).sum(), p) for p, d, cam, w in (a, b)]
    ras = kind()
    with torch.no_grad():      # a workspace large enough for all: the renders below share the buffer
        big, d, cam, _ = _scene(2000, 160, 120, 3, 1)
        ras.forward(*big, d, cam)
    buf = ras.ws.buf
    x, y = [(R.rasterize(*p, d, cam, ras) * w).sum() for p, d, cam, w in (a, b)]
    assert ras.ws.buf is buf
    got = torch.autograd.grad(x, a[0], retain_graph=True)
    _close(got, want[0])
    _close(torch.autograd.grad(y, b[0]), want[1])     # the later render's state still stands, or is made again
    _close(torch.autograd.grad(x, a[0]), want[0])


def test_sum_over_views_and_a_copied_rasterizer():
    import copy
    p, d, cam, w = _scene(150, 48, 40, 2, 9)
    turned = copy.copy(cam)
    turned.cx, turned.cy = cam.cx + 5.0, cam.cy - 3.0
    want = [torch.autograd.grad((R.rasterize(*p, d, c) * w).sum(), p) for c in (cam, turned)]
    ras = R.Rasterizer()
    total = sum((R.rasterize(*p, d, c, ras) * w).sum() for c in (cam, turned))
    _close(torch.autograd.grad(total, p), [u + v for u, v in zip(*want)])
    img = R.rasterize(*p, d, cam, ras)
    other = copy.deepcopy(ras)
    R.rasterize(*p, d, turned, other)          # a buffer and a count of its own
    assert other.ws.uses.value == ras.ws.uses.value + 1
    _close(torch.autograd.grad((img * w).sum(), p), want[0])
