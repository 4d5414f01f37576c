"""Records of either step of a pair under schedules, and of runs that end between the
two steps of a launch.

Both sides sum the same FP32 site terms.  The plain stepper rounds the sum of 128 sites
in FP32 (three additions in a quad, five butterfly levels), the band stepper the
three additions in a quad, so they agree within 11 * 2^-24 of the mean absolute term:
at most 1 for M; at most 30 for the site energies relative to their reference (twice
the couplings and twice the field at their largest here, and the kinetic energy)."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu
TOL_M = 11 * 2.0 ** -24
TOL_E = 30 * TOL_M
SCHED = dict(field=((0, 60), (0.4, 2.2)), couplings=((0, 60), (1.0, 0.4), (0.5, 2.5)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _compare(shapes, calls, totals=None, **kw):
    cfgs = [Config(Lx=a, Ly=b, n_replicas=r, seed=8, init_mode=0, knots=((0, 40), (2.5, 0.5)),
                   n_total=totals[i] if totals else 10 ** 9, params=dict(staggered_M=i & 1), **kw)
            for i, (a, b, r) in enumerate(shapes)]
    lats = [Lattice(cfgs) for _ in range(3)]
    lats[0].set_path(XY_PATH_PLAIN)
    lats[1].set_temporal_blocking(2)
    lats[2].set_temporal_blocking(1)
    for n, every in calls:
        r0, r2, r1 = (lat.step(n, every) for lat in lats)
        torch.cuda.synchronize()
        for lat in lats[1:]:
            assert torch.equal(lats[0].theta, lat.theta) and torch.equal(lats[0].omega, lat.omega), (n, every)
        assert torch.equal(torch.nan_to_num(r2, nan=9.0), torch.nan_to_num(r1, nan=9.0)), (n, every)
        assert torch.equal(torch.isnan(r0), torch.isnan(r2)), (n, every)
        d = (torch.nan_to_num(r0) - torch.nan_to_num(r2)).abs().amax(dim=(0, 1))
        assert d[0] <= TOL_M and d[1] <= TOL_E, (n, every, d)


@pytest.mark.parametrize("shapes", [[(200, 33, 2), (60, 20, 1)], [(1100, 12, 1), (256, 8, 2)], [(2048, 3, 1)]], ids=str)
def test_records_under_schedules(shapes):
    _compare(shapes, ((75, 1), (50, 7), (9, 3)), **SCHED)


@pytest.mark.parametrize("every", [1, 3])
def test_records_of_runs_that_end_inside_a_pair(every):
    _compare([(256, 16, 2), (256, 16, 1), (100, 20, 1), (100, 20, 1), (1100, 8, 1)],
             ((30, every), (80, every), (9, every)), totals=[37, 64, 1, 91, 52])
