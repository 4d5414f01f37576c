"""The reverse sweep in one launch (a cluster of blocks per lattice) where it can go
wrong: one to eight blocks per lattice, bands of 1, 2 and 4 rows, idle lane groups,
segments that do not divide the steps, two and three steps in all, schedules, and
groups that sweep beside groups that do not.

Two references: the stored recompute (another kernel and schedule; the two agree to
1e-4 of the gradient from the ordered start, as the existing schedule tests hold
them), and the same lattice inside a batch too large for clusters (the same kernel
launched step by step; the states are the same bits and only the grouping of the
FP32 sums differs, 1e-5 of the largest component covers it)."""
import numpy as np
import pytest
import torch

from paper_2409_06412_gb300 import (XY_ADJOINT_BACKWARD, XY_ADJOINT_RECOMPUTE, XY_INIT_ORDERED, Config, Lattice, build)

pytestmark = pytest.mark.gpu
FIELD = ((0, 30), (1.0, 0.6))
COUPL = ((0, 40), (1.0, 0.8), (1.0, 1.5))


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _grads(shapes, n, K, mode, extra=0, **kw):
    cfgs = [Config(Lx=a, Ly=b, n_replicas=r, seed=9, init_mode=XY_INIT_ORDERED, knots=((0, 60), (1.9, 1.2)),
                   params=dict(staggered_M=i & 1), **kw) for i, (a, b, r) in enumerate(shapes)]
    if extra:
        a, b, _ = shapes[0]
        cfgs.append(Config(Lx=a, Ly=b, n_replicas=extra, seed=9, init_mode=XY_INIT_ORDERED))
    lat = Lattice(cfgs)
    lat.set_autotune(False)
    lat.set_adjoint_mode(mode)
    out = []
    for _ in range(2):  # the second call goes on from the state and memory of the first
        obj, g = lat.adjoint(n, K, 0.8, 0.6)
        out.append(g[:len(shapes)] * lat.n_lattices * n)
    torch.cuda.synchronize()
    return np.stack(out), lat.theta[:sum(a * b * r for a, b, r in shapes)].clone()


@pytest.mark.parametrize("shapes", [
    [(64, 64, 2)], [(128, 128, 1)], [(32, 32, 3)], [(16, 34, 1)], [(8, 2, 2)], [(256, 8, 1)], [(256, 32, 2)],
    [(1024, 16, 1)], [(64, 64, 1), (256, 256, 1), (32, 96, 2)]], ids=lambda s: "+".join("%dx%d" % x[:2] for x in s))
@pytest.mark.parametrize("n,K", [(2, 5), (3, 2), (17, 5), (40, 40)])
def test_sweep_matches_the_stored_recompute(shapes, n, K):
    g, th = _grads(shapes, n, K, XY_ADJOINT_BACKWARD)
    r, th_r = _grads(shapes, n, K, XY_ADJOINT_RECOMPUTE)
    assert torch.equal(th, th_r)
    for c in range(len(shapes)):
        assert np.all(np.abs(g[:, c] - r[:, c]) <= 1e-4 * np.abs(r[:, c]).max(axis=1, keepdims=True)), (c, g[:, c], r[:, c])


@pytest.mark.parametrize("kw", [{}, dict(field=FIELD, couplings=COUPL)], ids=["plain", "schedules"])
@pytest.mark.parametrize("shape,extra", [((64, 64, 1), 600), ((128, 64, 2), 400), ((256, 16, 1), 900)])
def test_sweep_equals_single_launches(shape, extra, kw):
    g, th = _grads([shape], 25, 7, XY_ADJOINT_BACKWARD, **kw)
    r, th_r = _grads([shape], 25, 7, XY_ADJOINT_BACKWARD, extra=extra, **kw)
    assert torch.equal(th, th_r)
    assert np.all(np.abs(g - r) <= 1e-5 * np.abs(r).max()), (g, r)
