"""The autograd nodes of the torch front end: the same gradients as the direct calls, saved-tensor hooks, a second
backward, in-place changes, subclasses, other streams and errors behave as with nodes written in Python."""
import pytest
import torch

from paper_2402_17427_gb300 import binding as B
from paper_2402_17427_gb300 import rasterize as R
from paper_2402_17427_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


def _scene(degree=2):
    g, cam, target = scenes.tiny_scene(n=150, width=48, height=40, degree=degree, seed=9)
    return [p.requires_grad_(True) for p in R.to_device(g)], g.sh_degree, cam, torch.from_numpy(target).cuda()


def _close(a, b):      # sums of a few dozen FP32 atomics in another order
    for x, y in zip(a, b):
        assert torch.allclose(x, y, rtol=1e-4, atol=1e-5 * float(y.abs().max()) + 1e-12)


def test_gradients_equal_the_direct_calls():
    p, deg, cam, target = _scene()
    img = R.rasterize(*p, deg, cam)
    loss = R.l1_dssim_loss(img, target, 0.2)
    assert img.requires_grad and loss.requires_grad and loss.shape == ()
    got = torch.autograd.grad(3.0 * loss, p)
    ras, f = R.Rasterizer(), R.LossL1DSSIM(0.2)
    d = [t.detach() for t in p]
    rgb, T, last = ras.forward(*d, deg, cam)
    value, dL = f(rgb, target)
    assert torch.equal(rgb, img.detach()) and torch.equal(value, loss.detach())
    _close(got, ras.backward(*d, deg, cam, T, last, 3.0 * dL))


def test_non_contiguous_image_and_partial_requirements():
    p, deg, cam, target = _scene()
    for t in p[1:]:
        t.requires_grad_(False)
    img = R.rasterize(*p, deg, cam)
    flipped = img.transpose(1, 2)
    loss = R.l1_dssim_loss(flipped, target.transpose(1, 2).contiguous(), 0.2)
    g, = torch.autograd.grad(loss, p[:1])
    ref, = torch.autograd.grad(R.l1_dssim_loss(R.rasterize(*p, deg, cam), target, 0.2), p[:1])
    _close([g], [ref])
    with torch.no_grad():
        assert not R.rasterize(*p, deg, cam).requires_grad
    assert not R.rasterize(*[t.detach() for t in p], deg, cam).requires_grad


def test_saved_tensors_go_through_hooks_and_are_versioned():
    p, deg, cam, target = _scene()
    seen = []

    def pack(t):
        seen.append(t.shape)
        return t.cpu()
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda t: t.cuda()):
        loss = R.l1_dssim_loss(R.rasterize(*p, deg, cam), target, 0.2)
    got = torch.autograd.grad(loss, p)
    assert len(seen) == 7 + 2
    _close(got, torch.autograd.grad(R.l1_dssim_loss(R.rasterize(*p, deg, cam), target, 0.2), p))
    img = R.rasterize(*p, deg, cam)
    with torch.no_grad():
        p[0].add_(0.0)
    with pytest.raises(RuntimeError):
        img.sum().backward()


def test_second_backward_and_retained_graph():
    p, deg, cam, _ = _scene()
    img = R.rasterize(*p, deg, cam)
    a = torch.autograd.grad(img.sum(), p, retain_graph=True)
    _close(a, torch.autograd.grad(img.sum(), p))
    with pytest.raises(RuntimeError):
        torch.autograd.grad(img.sum(), p)


def test_subclass_methods_are_called():
    calls = []

    class Mine(R.Rasterizer):
        def backward(self, *a, **k):
            calls.append("backward")
            return super().backward(*a, **k)
    p, deg, cam, _ = _scene()
    a = torch.autograd.grad(R.rasterize(*p, deg, cam, Mine()).sum(), p)
    assert calls == ["backward"]
    _close(a, torch.autograd.grad(R.rasterize(*p, deg, cam).sum(), p))


def test_other_stream_and_thread_of_the_engine():
    p, deg, cam, target = _scene()
    ref = torch.autograd.grad(R.l1_dssim_loss(R.rasterize(*p, deg, cam), target, 0.2), p)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        loss = R.l1_dssim_loss(R.rasterize(*p, deg, cam), target, 0.2)
        got = torch.autograd.grad(loss, p)
    s.synchronize()
    _close(got, ref)


def test_backward_error_is_the_bindings():
    p, deg, cam, _ = _scene()
    ras = R.Rasterizer()
    rgb, T, last = ras.forward(*[t.detach() for t in p], deg, cam)
    small = torch.empty(4096, dtype=torch.uint8, device="cuda")      # refused on the host before any launch
    img = R._front().attach_render(*p, rgb, T, last, small, ras.ws.capacity, deg, bytes(R.camera_c(cam)),
                                   bytes(ras.settings.c()))
    with pytest.raises(B.VGError) as e:
        img.sum().backward()
    assert e.value.status == B.VG_ERR_CAPACITY


@pytest.mark.parametrize("unpack", [lambda t: t, lambda t: t.cuda().half(), lambda t: torch.stack([t.cuda()] * 2, -1)[..., 0]],
                         ids=["cpu", "half", "strided"])
def test_what_hooks_hand_back_is_checked(unpack):
    """Saved tensors that come back off the device, in another type or strided are refused on the host."""
    p, deg, cam, target = _scene()
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.cpu(), unpack):
        img = R.rasterize(*p, deg, cam)
    with pytest.raises(ValueError):
        torch.autograd.grad(img.sum(), p)
    x = torch.rand(3, 20, 24, device="cuda", requires_grad=True)
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.cpu(), lambda t: t):
        loss = R.l1_dssim_loss(x, torch.rand(3, 20, 24, device="cuda"))
    with pytest.raises(ValueError):
        loss.backward()


def test_target_that_requires_a_gradient_gets_none():
    x, y = (torch.rand(3, 20, 24, device="cuda") for _ in range(2))
    y.requires_grad_(True)
    loss = R.l1_dssim_loss(x, y)
    assert loss.requires_grad
    loss.backward()
    assert y.grad is None


def test_loss_objects_copy():
    import copy
    f = R.LossL1DSSIM(0.2)
    x, y = torch.rand(3, 20, 24, device="cuda", requires_grad=True), torch.rand(3, 20, 24, device="cuda")
    loss = R.l1_dssim_loss(x, y, 0.2, f)
    other = copy.deepcopy(f)
    assert other.calls == 1
    R.l1_dssim_loss(x, y, 0.2, other)          # another workspace and count: the first one's state stands
    assert (f.calls, other.calls) == (1, 2)
    loss.backward()
    assert torch.isfinite(x.grad).all()
