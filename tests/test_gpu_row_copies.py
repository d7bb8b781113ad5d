"""GPU parity of the cooperative row copies of the merge and of the densification at the edges of a block's share
(1,024 and 512 Gaussians), for every SH degree (16-byte and scalar rows), against the oracles."""
import numpy as np
import pytest
import torch

from oracle import optim as OO
from oracle import partition as OPT
from paper_2402_17427_gb300 import optim as OP
from paper_2402_17427_gb300 import partition as PT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2402_17427_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()


def _rows(rng, n, degree):
    k = (degree + 1) ** 2
    return [rng.normal(0, 1, s).astype(np.float32) for s in ((n, 3), (n, 3), (n, 4), (n,), (n, k, 3))]


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("sizes", [(1,), (1023, 0, 1), (1024, 1025), (3, 5, 2040, 7), (4097,)])
def test_merge_rows_are_exact(degree, sizes):
    rng = np.random.default_rng(sum(sizes) + degree)
    cells = [_rows(rng, n, degree) for n in sizes]
    regions = [(-0.5, 1.0, -1.0, 0.5)] * len(sizes)
    got = PT.merge_cells([[torch.from_numpy(a).cuda() for a in c] for c in cells], regions, degree)
    keep = OPT.merge([c[0] for c in cells], regions)
    assert int(got[0].shape[0]) == len(keep)
    for j, t in enumerate(got):
        ref = np.stack([cells[k][j][i] for k, i in keep]) if keep else np.zeros((0,) + cells[0][j].shape[1:], np.float32)
        assert np.array_equal(t.cpu().numpy(), ref), j


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 511, 512, 513, 1500])
def test_densified_rows_are_exact(degree, n):
    rng = np.random.default_rng(n + degree)
    P = _rows(rng, n, degree)
    P[1] = rng.normal(np.log(0.05), 0.8, (n, 3)).astype(np.float32)
    P[3] = rng.normal(1, 3, n).astype(np.float32)
    acc, cnt = rng.exponential(3e-4, n).astype(np.float32), rng.integers(0, 4, n).astype(np.int32)
    z = rng.standard_normal((n, 2, 3)).astype(np.float32)
    ds = OP.DensifySettings(scene_extent=10.0)
    params = [torch.from_numpy(a).cuda() for a in P]
    adam, stats = OP.Adam(params), OP.DensifyStats(n, "cuda")
    mom = [rng.random(a.shape).astype(np.float32) for a in P]
    adam.m = tuple(torch.from_numpy(a).cuda() for a in mom)
    adam.v = tuple(torch.from_numpy(2 * a).cuda() for a in mom)
    stats.accum.copy_(torch.from_numpy(acc))
    stats.count.copy_(torch.from_numpy(cnt))
    f = np.float32
    th = OO.thresholds(f(ds.grad_threshold), float(f(ds.percent_dense)), float(f(ds.scene_extent)),
                       float(f(ds.min_opacity)), float(f(ds.max_world_scale_frac * ds.scene_extent)))
    new = OP.densify_with(params, adam, stats, degree, ds, torch.from_numpy(z).cuda())
    ref, refm, act = OO.densify(dict(zip(OP.PARAM_NAMES, P)), {k: (mom[i], 2 * mom[i]) for i, k in enumerate(OP.PARAM_NAMES)},
                                acc, cnt, z.astype(np.float64), th)
    assert int(new[0].shape[0]) == len(ref["means"])
    for i, k in enumerate(OP.PARAM_NAMES):
        got = new[i].cpu().numpy().astype(np.float64)
        if len(ref[k]) == 0:
            continue
        if k == "means":     # a split child's mean is computed in FP32
            assert np.allclose(got, ref[k], rtol=1e-5, atol=1e-6)
        else:
            assert np.array_equal(got, ref[k]), k
        assert np.array_equal(adam.m[i].cpu().numpy().astype(np.float64), refm[k][0]), k
        assert np.array_equal(adam.v[i].cpu().numpy().astype(np.float64), refm[k][1]), k
