"""Autocorrelation times where the work is split differently: one block or a
cluster of up to eight per series, windows that end in the first batch of 256
lags, on its edge or in later ones, the literal half window, series whose
deviations do not fit shared memory.  Against 64-bit sums by FFT: the lag sums
multiply FP32 deviations (relative 2^-24 each) in FP32 runs of at most 256 terms,
so each C(m) / C(0) is within 260 * 2^-24 (the sum of |d_s d_{s+m}| is at most
n C(0)) and a sum of M of them within M times that."""
import numpy as np
import pytest
import torch

from paper_2409_06412_gb300 import build, sampling
from tests.inputs import ar1_series

pytestmark = pytest.mark.gpu
PER_LAG = 260 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _reference(x, c):
    n = x.size
    d = x - x.mean()
    sp = np.fft.rfft(d, 2 * n)
    C = np.fft.irfft(np.abs(sp) ** 2, 2 * n)[:n // 2 + 1] / (n - np.arange(n // 2 + 1))
    tau = 0.5 + np.cumsum(C[1:]) / C[0]
    m = np.arange(1, n // 2 + 1)
    stop = np.nonzero(m >= c * tau)[0] if c > 0 else []
    at = stop[0] if len(stop) else n // 2 - 1
    return x.mean(), C[0], tau, at


@pytest.mark.parametrize("n_series,n,phi,c", [
    (3, 2, 0.5, 6.0), (2, 5, 0.5, 0.0), (700, 515, 0.9, 6.0), (40, 2100, 0.97, 6.0), (5, 4099, 0.99, 6.0),
    (2, 16390, 0.995, 6.0), (2, 49153, 0.98, 6.0), (1, 60001, 0.999, 4.0), (3, 1537, 0.4, 0.0)])
def test_split_sums_match_64_bits(n_series, n, phi, c):
    x = ar1_series(n, phi, seed=n, n_series=min(n_series, 7))
    x = np.stack([x[b % x.shape[0]] for b in range(n_series)]) * 0.2 - 0.4
    rec = np.zeros((n_series, n, 2))
    rec[:, :, 1] = x
    out = sampling.autocorr_time(torch.from_numpy(rec).cuda(), "E", "f", 0, n, c).cpu().numpy()
    for b in range(min(n_series, 7)):
        mean, C0, tau, at = _reference(x[b], c)
        np.testing.assert_allclose(out[b, :2], [mean, C0], rtol=1e-12, atol=1e-14)
        # the stopping lag may move by one where c tau(M) meets M within the tolerance
        near = [abs(out[b, 2] - tau[i]) <= PER_LAG * (i + 2) for i in (at - 1, at, at + 1) if 0 <= i < tau.size]
        assert any(near), (out[b, 2], tau[at], at)
    # equal series give equal bits wherever they sit in the batch
    for b in range(7, n_series):
        assert np.array_equal(out[b], out[b % 7])
