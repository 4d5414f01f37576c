"""Calls whose length is no multiple of the record interval begin at another step of it
each time: states bit for bit, and the steps that record, as with the plain stepper,
over more calls than the library keeps captured chunks."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("n,every", [(27, 20), (47, 40), (127, 50), (90, 64), (77, 16), (70, 65)])
def test_calls_at_every_phase_of_the_interval(n, every):
    # the second configuration ends early, the third is resident and goes on longest
    cfgs = [Config(Lx=100, Ly=8, seed=2, init_mode=0, n_total=60 * n), Config(Lx=256, Ly=4, seed=2, init_mode=0, n_total=9 * n + 5),
            Config(Lx=16, Ly=16, seed=2, init_mode=0)]
    ref, lat = Lattice(cfgs), Lattice(cfgs)
    ref.set_path(XY_PATH_PLAIN)
    for i in range(66):
        r0, r1 = ref.step(n, every), lat.step(n, every)
        torch.cuda.synchronize()
        assert torch.equal(ref.theta, lat.theta) and torch.equal(ref.omega, lat.omega), i
        assert torch.equal(torch.isnan(r0), torch.isnan(r1)), i
        d = (torch.nan_to_num(r0) - torch.nan_to_num(r1)).abs().amax(dim=(0, 1))
        assert d[0] < 1e-6 and d[1] < 3e-5, (i, d)  # FP32 sums of the same terms in another order
