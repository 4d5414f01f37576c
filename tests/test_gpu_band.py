"""The band stepper on the shapes where it can go wrong: rows that fill no whole
warp, one to sixteen warps side by side, lane groups with lanes left over, last
bands shorter than the others, lattices lower than a band's halo, runs that end
between the two steps of a launch, records on either side of a pair.

States are compared bit for bit with the plain stepper (one thread per quad,
neighbours from global memory), which the oracle tests cover.  Records are sums
of the same FP32 site terms in another order: a lane adds at most 4 * 64 terms
and a warp butterfly 5 more levels, so each side is within 261 * 2^-24 of the
mean absolute term (at most 1 for M; at most 25 for the site energies relative
to their reference at these temperatures)."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu
TOL_M = 2 * 261 * 2.0 ** -24
TOL_E = 25 * TOL_M

SHAPES = [
    [(132, 9, 2)],                       # two warps of 17 and 16 lanes
    [(2044, 10, 1), (1028, 33, 1)],      # sixteen warps, nine warps
    [(2048, 8, 1), (500, 75, 2)],
    [(100, 60, 3), (60, 48, 2)],         # one lane group of 25, two of 15
    [(20, 17, 5), (12, 10, 1)],          # six groups of 5, ten of 3
    [(200, 1, 2), (256, 2, 1), (36, 3, 2)],  # fewer rows than the halo
    [(2052, 6, 1), (384, 7, 1)],         # wider than the kernel takes
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _lattices(shapes, totals=None, **kw):
    cfgs = [Config(Lx=a, Ly=b, n_replicas=r, seed=3, init_mode=0, knots=((0, 40), (2.5, 0.5)),
                   n_total=totals[i] if totals else 10 ** 9, params=dict(staggered_M=i & 1), **kw)
            for i, (a, b, r) in enumerate(shapes)]
    out = []
    for kt in (None, 2, 1):
        lat = Lattice(cfgs)
        if kt is None:
            lat.set_path(XY_PATH_PLAIN)
        else:
            lat.set_temporal_blocking(kt)
        out.append(lat)
    return out


def _same(ref, others):
    torch.cuda.synchronize()
    return all(torch.equal(ref.theta, o.theta) and torch.equal(ref.omega, o.omega) for o in others)


@pytest.mark.parametrize("shapes", SHAPES, ids=lambda s: "+".join("%dx%d" % x[:2] for x in s))
def test_band_stepper_equals_the_plain_stepper(shapes):
    ref, two, one = _lattices(shapes)
    for n, every in ((5, 0), (66, 7), (130, 50), (3, 1)):
        recs = [lat.step(n, every) for lat in (ref, two, one)]
        assert _same(ref, (two, one)), (n, every)
        if every:
            r0, r2, r1 = (torch.nan_to_num(r, nan=9.0) for r in recs)
            assert torch.equal(r2, r1)
            d = (r2 - r0).abs().amax(dim=(0, 1))
            assert d[0] <= TOL_M and d[1] <= TOL_E, d


def test_runs_that_end_inside_a_pair():
    shapes = [(256, 16, 2), (256, 16, 1), (100, 20, 1), (100, 20, 1)]
    ref, two, one = _lattices(shapes, totals=[37, 64, 1, 91])
    for n, every in ((30, 0), (80, 10), (9, 0)):
        for lat in (ref, two, one):
            lat.step(n, every)
        assert _same(ref, (two, one)), (n, every)


def test_band_stepper_with_schedules():
    ref, two, one = _lattices([(200, 33, 2), (60, 20, 1)], field=((0, 60), (0.4, 2.2)),
                              couplings=((0, 60), (1.0, 0.4), (0.5, 2.5)))
    for lat in (ref, two, one):
        lat.step(75, 10)
    assert _same(ref, (two, one))
