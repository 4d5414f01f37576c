"""Calls of a few steps end in the caller's buffers without copies: whatever the
number of steps (past one), the launches of a group are even in number.  States are
those of the plain stepper, bit for bit."""
import pytest
import torch

from paper_2409_06412_gb300 import XY_PATH_PLAIN, Config, Lattice, build

pytestmark = pytest.mark.gpu
STRIP, STRIP2 = 1, 6  # timing classes of launches of one step and of two


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape", [(256, 16), (100, 20), (1100, 8)], ids=str)
def test_short_calls_launch_an_even_number(shape):
    cfgs = [Config(Lx=shape[0], Ly=shape[1], n_replicas=2, seed=7, init_mode=0)]
    ref, lat = Lattice(cfgs), Lattice(cfgs)
    ref.set_path(XY_PATH_PLAIN)
    for timing in (True, False):  # launched directly, and captured
        lat.set_kernel_timing(timing)
        seen = 0
        for n in (2, 3, 4, 5, 6, 7, 10, 66, 97):
            lat.step(n, 3 if n == 7 else 0)
            ref.step(n, 3 if n == 7 else 0)
            torch.cuda.synchronize()
            assert torch.equal(ref.theta, lat.theta) and torch.equal(ref.omega, lat.omega), n
            if timing:
                launches = lat.kernel_timing()[1]
                now = int(launches[STRIP] + launches[STRIP2])
                assert (now - seen) % 2 == 0 and now - seen <= n // 2 + 2, (n, now - seen)
                seen = now
