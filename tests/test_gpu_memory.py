"""Device memory of an object beside its second state: the partial sums of records take
32 bytes per 1024 sites (two steps of a launch, one partial of 16 bytes per 256 quads),
less where a lattice's blocks are larger; tables and counters take little."""
import pytest
import torch

from paper_2409_06412_gb300 import Config, Lattice, build

pytestmark = pytest.mark.gpu


def test_record_partials_of_a_large_batch():
    build.build()
    shape, n = (256, 256), 4096
    sites = shape[0] * shape[1] * n
    theta = torch.zeros(sites, device="cuda")
    omega = torch.zeros(sites, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    lat = Lattice([Config(Lx=shape[0], Ly=shape[1], n_replicas=n)], theta=theta, omega=omega)
    torch.cuda.synchronize()
    extra = free - torch.cuda.mem_get_info()[0] - 8 * sites
    lat.close()
    # allocations come in pieces of 2 MiB: the two states, the partials, the small ones
    assert extra <= 32 * sites // 1024 + 4 * 2 ** 21, extra
