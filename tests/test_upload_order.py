"""Uploads of tables keep the order of the object's stream."""
import os
import re

import pytest
import torch

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_06412_gb300", "csrc")


def test_every_upload_is_on_a_stream():
    """A plain cudaMemcpy from pageable memory neither waits for the data to land
    nor orders a non-blocking stream."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        plain = re.findall(r"cudaMemcpy\((?:[^()]|\([^()]*\))*cudaMemcpyHostToDevice", text)
        assert not plain, (name, plain)


@pytest.mark.gpu
def test_first_calls_on_a_stream_of_its_own():
    """First steps and structure factors of an object on a non-blocking stream that
    is still busy: the same as on the current stream."""
    from paper_2409_06412_gb300 import Config, Lattice, build
    build.build()
    cfgs = [Config(Lx=a, Ly=b, n_replicas=r, seed=2, init_mode=0) for a, b, r in
            ((256, 64, 2), (100, 30, 3), (64, 64, 2), (2176, 32, 1))]
    ref = Lattice(cfgs)
    ref.step(20)
    S0 = ref.structure_factor(0, 7, K=8)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    a = torch.randn(4096, 4096, device="cuda")
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        lat = Lattice(cfgs, stream=side)
        for _ in range(4):
            a = (a @ a).tanh()
        lat.step(20)
        S1 = lat.structure_factor(0, 7, K=8)
    side.synchronize()
    assert torch.equal(ref.theta, lat.theta) and torch.equal(ref.omega, lat.omega)
    assert torch.equal(S0[0], S1[0]) and torch.equal(S0[1], S1[1])
