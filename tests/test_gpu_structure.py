"""Structure factors over every split of the line length (multiples of 16, 8, 4
and 2, and odd lengths), lines shorter than a block's share, more wavenumbers than
one pass forms, and lattices of different shapes in one call, against the 64-bit
transform.

Tolerance: a line sum of N = R A terms of modulus at most 1 per component is off by
at most gamma N with gamma = (A + 12) 2^-24 (A terms in order, at most 5 levels and
3 products of the R-point transform, 3 of the reduction, one rounding of the rotor),
so with L lines of the lattice, Cauchy-Schwarz bounds the error of
S = sum |X|^2 / (N L) by (2 gamma N sqrt(4 L S N L) + 4 L (gamma N)^2) / (N L)."""
import math

import pytest
import torch

from paper_2409_06412_gb300 import XY_INIT_USER, Config, Lattice, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _reference(th, axis, K, r):
    S = sum((torch.fft.fft(f(r * th), dim=axis).abs() ** 2).sum(dim=1 - axis) for f in (torch.cos, torch.sin))
    return S[:K] / th.numel()


def _bound(S, N, lines):
    R = next(r for r in (16, 8, 4, 2, 1) if N % r == 0)
    g = (N // R + 12) * 2.0 ** -24
    return (2 * g * N * torch.sqrt(4 * lines * S * N * lines) + 4 * lines * (g * N) ** 2) / (N * lines)


@pytest.mark.parametrize("shapes,K", [
    ([(64, 48, 2)], 16), ([(136, 40, 2)], 24), ([(100, 60, 1), (20, 33, 2)], 17), ([(12, 7, 3)], 7), ([(4, 1, 2)], 1),
    ([(1000, 333, 1), (2048, 62, 1)], 33), ([(1024, 1024, 1)], 16)], ids=lambda v: str(v).replace(" ", ""))
def test_structure_factor_against_64_bits(shapes, K):
    gen = torch.Generator(device="cuda").manual_seed(5)
    n = sum(a * b * r for a, b, r in shapes)
    th = (torch.rand(n, generator=gen, device="cuda") ** 3 - 0.3) * 2.0
    lat = Lattice([Config(Lx=a, Ly=b, n_replicas=r, init_mode=XY_INIT_USER) for a, b, r in shapes], theta=th,
                  omega=torch.zeros_like(th))
    for rotor in (1.0, 2.0):
        S_par, S_perp = lat.structure_factor(K=K, rotor=rotor)
        # a part of the batch gives the same bits
        b0 = lat.n_lattices // 2
        P, _ = lat.structure_factor(b0, 1, K=K, rotor=rotor)
        assert torch.equal(P[0], S_par[b0])
        for b in range(lat.n_lattices):
            t = lat.lattice_view(lat.theta, b).double()
            Ly, Lx = t.shape
            for got, axis, N, lines in ((S_par[b], 1, Lx, Ly), (S_perp[b], 0, Ly, Lx)):
                ref = _reference(t, axis, K, rotor)
                assert torch.all((got - ref).abs() <= _bound(ref, N, lines)), (Lx, Ly, axis, rotor)
        assert math.isfinite(float(S_par.sum()))
