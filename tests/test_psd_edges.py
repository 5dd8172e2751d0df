"""Edges of the Welch kernel and of the resonance fit (GPU) against the oracle.

Welch (per bin, bound of tests/test_psd_parity.py): series that start at an
odd float (4-byte copies), every segment length with one segment, with fewer
and with more segments than the GPU transforms at a time, an infinite sample.
Resonance fit: bands of 8 bins (the fewest), of a few bins beyond a multiple
of the 256 that a row of the fit holds, and longer than the rows whose
logarithm is kept.  The fit stops when chi^2 changes by 1e-12 of itself, which
leaves the parameters within sqrt(1e-12 n) standard errors of the optimum:
two FP64 fits agree within 1e-5 of a standard error for n <= 100 bins and
within 1e-9 relative where the standard errors are small.
"""
import numpy as np
import pytest

from oracle import psd as opsd
from tests.test_psd_parity import psd_tol

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

FS = 1e6


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("M,segments,stride,offset", [
    (4096, 1, 1, 1), (4096, 1217, 1, 0), (4096, 2500, 3, 1), (8192, 609, 1, 1), (8192, 3, 5, 0),
    (16384, 305, 1, 0), (16384, 2, 2, 1), (32768, 1, 1, 1), (32768, 153, 1, 0), (32768, 160, 1, 1),
])
def test_welch_segments_strides_and_offsets(dev, M, segments, stride, offset):
    n = M + (segments - 1) * (M // 2) + M // 2 - 1        # one sample short of another segment
    rng = np.random.default_rng(M + segments)
    x = (1e6 * rng.standard_normal(n) + 2e6 * np.sin(np.arange(n) * 0.1) + 3e5).astype(np.float32)
    buf = torch.full((offset + n * stride,), 5.0, dtype=torch.float32, device=dev)
    buf[offset::stride][:n] = torch.from_numpy(x).to(dev)
    with cg.Psd(M) as p:
        S, K = p.welch(buf[offset:], FS, stride=stride, n=n)
        S = S.cpu().numpy()
    _, So, Ko = opsd.welch(x.astype(np.float64), FS, M)
    assert K == Ko == segments
    assert np.all(np.abs(S - So) <= psd_tol(So, M))


@pytest.mark.parametrize("M", [4096, 32768])
def test_welch_infinite_sample(dev, M):
    x = torch.ones(4 * M, dtype=torch.float32, device=dev)
    x[M // 3] = float("inf")
    with cg.Psd(M) as p:
        S, _ = p.welch(x, FS)
    assert torch.isnan(S).all()


@pytest.mark.parametrize("f0,Q,df,k_lo,k_hi,n_bins", [
    (1000.0, 5.0, 60.0, 14, 21, 2049),          # 8 bins
    (23.7e3, 120.0, 30.0, 700, 955, 16385),     # 256
    (23.7e3, 120.0, 30.0, 640, 902, 16385),     # 263
    (23.7e3, 40.0, 4.0, 1, 16384, 16385),       # every bin: 64 rows of 256
    (23.7e3, 40.0, 2.0, 1, 20000, 20001),       # longer than the kept logarithms
])
def test_resonance_bands(dev, f0, Q, df, k_lo, k_hi, n_bins):
    f = df * np.arange(n_bins)
    S = 3.0 * f0 ** 4 / ((f0 ** 2 - f ** 2) ** 2 + (f * f0 / Q) ** 2) + 2.0
    S *= np.random.default_rng(n_bins).gamma(400.0, 1.0 / 400.0, n_bins)
    lo, hi = (k_lo - 0.5) * df, (k_hi + 0.5) * df
    out = cg.Psd.resonance(torch.from_numpy(S).to(dev), df, lo, hi)
    fb, Sb = opsd.band(f, S, lo, hi)
    r = opsd.fit(fb, Sb)
    assert int(out[11]) == fb.size == k_hi - k_lo + 1
    assert int(out[10]) == r["status"] == 0
    tol = 1e-5 * max(1.0, np.sqrt(fb.size / 100.0)) * np.asarray(r["sigma"]) + 1e-9 * np.abs(r["params"])
    assert np.all(np.abs(out[:4] - r["params"]) <= tol)
    assert np.allclose(out[4:8], r["sigma"], rtol=1e-5)
    assert np.isclose(out[8], r["rss"], rtol=1e-9)
