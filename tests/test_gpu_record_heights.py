"""Records do not depend on the height of the bands or strips that sum them.

The lanes and warps of a band or strip add their quads' FP32 sums of four terms as pairs of
FP32 values.  A lane adds at most 64 of them here and a warp 5 levels more; each
addition leaves at most 2^-24 of the absolute sum to the rest, and the rest's own 69
additions round it by at most 69 * 2^-24 of itself, so a record is within 69^2 *
2^-48 of the mean absolute term (1 for M, 25 for the site energies relative to their
reference) of the sum of the quads', on each side."""
import pytest
import torch

from paper_2409_06412_gb300 import Config, Lattice, build

pytestmark = pytest.mark.gpu
TOL_M = 2 * 69 ** 2 * 2.0 ** -48
TOL_E = 25 * TOL_M


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape,many", [((256, 256), 256), ((100, 192), 300), ((1100, 128), 100),
                                        ((2176, 128), 40)], ids=str)
@pytest.mark.parametrize("mode", [0, 1])
def test_records_of_one_lattice_alone_and_in_a_large_batch(shape, many, mode):
    """Without the tuner one lattice takes bands of a row or two (strips of 8 where it is
    wider than 2048), the batch bands of up to 64 rows (strips of 32)."""
    recs = []
    for n in (1, many):
        lat = Lattice([Config(Lx=shape[0], Ly=shape[1], n_replicas=n, seed=6, init_mode=mode, knots=((0,), (1.0,)))])
        lat.set_autotune(False)
        recs.append(lat.step(7, 1)[0].clone())
        lat.close()
    d = (recs[0][:7] - recs[1][:7]).abs().amax(dim=0)
    assert d[0] <= TOL_M and d[1] <= TOL_E, d
