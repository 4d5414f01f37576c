"""Objects of several groups (noise seeds, shapes): fewer and more of them than the
library has branch streams.  States are those of the plain stepper, bit for bit, through
calls with and without records, on the current stream and on one of its own."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _compare(shapes, seeds, calls=((1, 0), (2, 1), (70, 9), (130, 0))):
    cfgs = [Config(Lx=a, Ly=b, n_replicas=r, seed=s, init_mode=0, knots=((0, 40), (2.5, 0.5)))
            for s in range(seeds) for a, b, r in shapes]
    ref, lat = Lattice(cfgs), Lattice(cfgs)
    ref.set_path(XY_PATH_PLAIN)
    side = torch.cuda.Stream()
    own = Lattice(cfgs, stream=side)
    for n, every in calls:
        r0, r1 = ref.step(n, every), lat.step(n, every)
        with torch.cuda.stream(side):
            r2 = own.step(n, every)
        torch.cuda.synchronize()
        assert torch.equal(ref.theta, lat.theta) and torch.equal(ref.omega, lat.omega), (n, every)
        assert torch.equal(ref.theta, own.theta) and torch.equal(ref.omega, own.omega), (n, every)
        if every:
            assert torch.equal(torch.nan_to_num(r1), torch.nan_to_num(r2))
            d = (torch.nan_to_num(r0) - torch.nan_to_num(r1)).abs().amax(dim=(0, 1))
            assert d[0] < 1e-6 and d[1] < 3e-5, d  # FP32 sums of the same terms in another order


@pytest.mark.parametrize("shapes,seeds", [([(64, 64, 1)], 2), ([(64, 64, 3)], 12), ([(32, 32, 2), (128, 128, 1)], 3),
                                          ([(128, 64, 40), (16, 16, 5)], 2)], ids=str)
def test_resident_groups(shapes, seeds):
    _compare(shapes, seeds)


@pytest.mark.parametrize("shapes,seeds", [([(256, 24, 2)], 12), ([(96, 40, 3), (64, 64, 1)], 7),
                                          ([(100, 12, 1), (2176, 4, 1), (2052, 3, 1)], 4)], ids=str)
def test_more_groups_than_streams(shapes, seeds):
    _compare(shapes, seeds)
