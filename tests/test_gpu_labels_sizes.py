"""Labels and size histograms where the passes can go wrong: tiles that are not
full, runs that join pieces late (combs, spirals, checkerboards), lattices with so
many distinct sizes that the compaction's word list overflows, widths that are and
are not powers of two.  Labels and counts are whole numbers: they equal the
oracle's flood fill exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_06412_gb300 import XY_INIT_USER, Config, Lattice, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _patterns(Lx, Ly, rng):
    y, x = np.mgrid[0:Ly, 0:Lx]
    yield np.ones((Ly, Lx), bool)
    yield (x + y) % 2 == 0
    yield (x % 2 == 0) | (y == Ly - 1)            # comb: teeth join in the last row
    yield (x % 2 == 0) | (y == 0)
    yield (y % 4 < 2) ^ ((x % 32 == 31) & (y % 8 < 4))
    d = np.maximum(abs(x - Lx // 2), abs(y - Ly // 2))
    yield (d % 2 == 0) | ((x > Lx // 2) & (y == Ly // 2) & (d % 4 == 1))  # rings joined by a few bridges
    yield rng.random((Ly, Lx)) < 0.5
    yield rng.random((Ly, Lx)) < 0.41
    yield rng.random((Ly, Lx)) < 0.03


@pytest.mark.parametrize("Lx,Ly", [(4, 1), (32, 32), (36, 33), (64, 31), (100, 65), (128, 96), (260, 70)])
def test_patterns_match_the_flood_fill(Lx, Ly):
    rng = np.random.default_rng(Lx * 1000 + Ly)
    pats = list(_patterns(Lx, Ly, rng))
    th = np.where(np.stack(pats), 0.9, -0.9).astype(np.float32)
    lat = Lattice([Config(Lx=Lx, Ly=Ly, n_replicas=len(pats), init_mode=XY_INIT_USER)],
                  theta=torch.from_numpy(th.reshape(-1)).cuda(), omega=torch.zeros(th.size, device="cuda"))
    for _ in range(2):  # the second call finds the working memory as the first left it
        labels, hist, n_sizes = (t.cpu().numpy() for t in lat.label_domains(hist_cap=4096))
        for b in range(len(pats)):
            lab, h = oracle.ccl(Lx, Ly, th[b].ravel())
            assert np.array_equal(labels[b], lab), (Lx, Ly, b)
            h = np.asarray(h).reshape(-1, 2)
            assert n_sizes[b] == len(h) and np.array_equal(hist[b, :len(h)], h) and not hist[b, len(h):].any(), b


def test_more_size_words_than_the_compaction_lists():
    """Bars of lengths 64, 96, 128, ... each in a word of its own: 1400 words hold a
    size (the shared list takes 1024), plus single sites."""
    lengths = 64 + 32 * np.arange(1400)
    Lx = 4096
    rows, row, used = [], np.zeros(Lx, bool), 0
    placed = []
    for n in lengths[::-1]:
        n = int(n)
        h = -(-n // 2000)                       # a block of h rows, 2000 wide at most
        placed.append((n, h))
    # each domain on rows of its own: full rows of 2000 columns and a rest
    Ly = sum(h + 1 for _, h in placed)
    g = np.zeros((Ly, Lx), bool)
    y = 0
    for n, h in placed:
        flat = np.zeros(h * 2000, bool)
        flat[:n] = True
        g[y:y + h, 1:2001] = flat.reshape(h, 2000)
        y += h + 1
    th = torch.from_numpy(np.where(g, 0.5, -0.5).astype(np.float32).reshape(-1)).cuda()
    lat = Lattice([Config(Lx=Lx, Ly=Ly, n_replicas=1, init_mode=XY_INIT_USER)], theta=th, omega=torch.zeros_like(th))
    want = sorted([int(n) for n in lengths] + [g.size - int(lengths.sum())])
    for _ in range(2):
        _, hist, n_sizes = lat.label_domains(hist_cap=2048)
        assert int(n_sizes[0]) == len(want)
        assert hist[0, :len(want), 0].tolist() == want
        assert (hist[0, :len(want), 1] == 1).all() and not hist[0, len(want):].any()
