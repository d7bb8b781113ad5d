"""Where the C++ autograd nodes were not built (no torch headers), rasterize() and l1_dssim_loss() take the nodes
written in Python: the same gradients and the same refusal of an overwritten loss workspace."""
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


def test_without_the_extension_the_python_nodes_serve(monkeypatch):
    g, cam, target = scenes.tiny_scene(n=150, width=48, height=40, degree=2, seed=9)
    p, target = [t.requires_grad_(True) for t in R.to_device(g)], torch.from_numpy(target).cuda()
    ref = torch.autograd.grad(R.l1_dssim_loss(R.rasterize(*p, 2, cam), target, 0.2), p)
    monkeypatch.setattr(R, "_front", lambda: None)
    f = R.LossL1DSSIM(0.2)
    got = torch.autograd.grad(R.l1_dssim_loss(R.rasterize(*p, 2, cam), target, 0.2, f), p)
    for x, y in zip(got, ref):             # sums of FP32 atomics in another order
        assert torch.allclose(x, y, rtol=1e-4, atol=1e-5 * float(y.abs().max()) + 1e-12)
    assert f.calls == 1 and f.uses is None
    x = torch.rand_like(target, requires_grad=True)
    loss = R.l1_dssim_loss(x, target, 0.2, f)
    f.value(x.detach(), target)
    with pytest.raises(RuntimeError):      # the workspace was used again
        loss.backward()
