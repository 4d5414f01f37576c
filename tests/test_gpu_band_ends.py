"""Runs that end inside a captured chunk while others of the chunk go on.

Each configuration is a slice of its own (one lattice each, four slices per
shape), so past its last step a slice's launches hold nothing but blocks whose
run has ended, and its last real launch, which writes the state and commits a
record, is ordered before the end of the chunk only through them.  The last
step of each run is a recorded one.  States are compared bit for bit with the
plain stepper; records are sums of the same FP32 site terms in another order: a
lane adds at most 4 * 64 terms and a warp butterfly 5 more levels, so each side is
within 261 * 2^-24 of the mean absolute term (at most 1 for M, at most 25 for the
site energies relative to their reference at these temperatures)."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu
TOL_M = 2 * 261 * 2.0 ** -24
TOL_E = 25 * TOL_M


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape", [(256, 64), (200, 48), (100, 64), (1100, 24)], ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("totals", [(4, 37, 41, 200), (9, 9, 9, 130)], ids=str)
def test_slices_that_end_inside_a_chunk(shape, totals):
    cfgs = [Config(Lx=shape[0], Ly=shape[1], seed=5, init_mode=0, knots=((0, 40), (2.5, 0.5)), n_total=t,
                   params=dict(staggered_M=i & 1)) for i, t in enumerate(totals)]
    ref, band = Lattice(cfgs), Lattice(cfgs)
    ref.set_path(XY_PATH_PLAIN)
    for _ in range(2):  # the second call starts from runs that have all but one ended
        r0, r1 = ref.step(150, 4), band.step(150, 4)
        torch.cuda.synchronize()
        assert torch.equal(ref.theta, band.theta) and torch.equal(ref.omega, band.omega)
        assert torch.equal(torch.isnan(r0), torch.isnan(r1))
        d = (torch.nan_to_num(r0) - torch.nan_to_num(r1)).abs().amax(dim=(0, 1))
        assert d[0] <= TOL_M and d[1] <= TOL_E, d
    assert list(band.observe()[1]) == [min(t, 300) for t in totals]
