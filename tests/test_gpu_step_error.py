"""A stepper whose bounded wait ran out leaves a state that is not valid: every call
that uses it says so until a snapshot replaces it.  The wait cannot run out in a
sound launch, so the error word is set from the host, as the kernel would set it."""
import numpy as np
import pytest
import torch

from paper_2409_06412_gb300 import Config, Lattice, XYError, _lib, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def test_a_failed_step_stays_reported_until_the_state_is_replaced():
    lat = Lattice([Config(Lx=1152, Ly=32, seed=4), Config(Lx=64, Ly=64, seed=4)])
    lat.step(4)
    blob = lat.save()
    lat.step(2)
    want = lat.theta.clone()
    _lib.call("xy_debug_set_step_error", lat._h, _lib.XY_ETIMEOUT)
    host_rec = np.zeros((2, 3, 2))
    for _ in range(2):  # no report clears it
        for use in (lambda: lat.label_domains(0, 1), lambda: lat.observe(), lambda: lat.step(2),
                    lambda: lat.step(2, 1, rec=host_rec), lambda: lat.structure_factor(0, 1, K=4),
                    lambda: lat.adjoint(2, 2), lambda: lat.omega_full(), lambda: lat.save(),
                    lambda: lat.synchronize()):
            with pytest.raises(XYError) as e:
                use()
            assert e.value.code == _lib.XY_ETIMEOUT
    lat.load(blob)
    lat.step(2)
    lat.label_domains(0, 1)
    lat.observe()
    torch.cuda.synchronize()
    assert torch.equal(lat.theta, want)
