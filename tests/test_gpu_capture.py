"""Structure factors in a caller's CUDA graph: captured as the first call of an object or
a later one, replayed on new states and after calls that need more working memory."""
import pytest
import torch

from paper_2409_06412_gb300 import Config, Lattice, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [True, False])
def test_captured_structure_factors(first):
    build.build()
    side = torch.cuda.Stream()
    cfgs = [Config(Lx=64, Ly=48, n_replicas=3, seed=1, init_mode=0), Config(Lx=100, Ly=30, n_replicas=2, seed=1, init_mode=0)]
    lat, ref = Lattice(cfgs, stream=side), Lattice(cfgs)
    torch.cuda.synchronize()
    if not first:
        with torch.cuda.stream(side):
            lat.structure_factor(0, 5, K=4)
        side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        S = lat.structure_factor(1, 4, K=8)
    for k in range(3):
        ref.step(5)
        torch.cuda.synchronize()
        lat.theta.copy_(ref.theta)
        torch.cuda.synchronize()
        if k == 1:  # more than the captured call has
            with torch.cuda.stream(side):
                lat.structure_factor(0, 5, K=30)
            side.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        want = ref.structure_factor(1, 4, K=8)
        torch.cuda.synchronize()
        assert torch.equal(S[0], want[0]) and torch.equal(S[1], want[1]), k
