"""The resonance fit (GPU) gives the recorded values.

The fit ends when chi^2 has settled and takes its last step only if chi^2 did
not rise, which at the optimum its last bit decides: a fit whose FP64
operations differ in rounding ends up to 1e-5 (mostly 1e-8) away.  The values
in golden/resonance_fit.json are those of the plain form of the fit: one block,
divisions, square roots and logarithms as CUDA rounds them, sums of points t,
t + 256, ... added over the lanes of a warp (distances 16 to 1) and over the
warps in order.  The densities are made by exact or correctly rounded
operations alone, so every machine makes the same.
"""
import json
import os

import numpy as np
import pytest

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "resonance_fit.json")

# segment length, segments averaged, f0, Q, floor / A, band
BANDS = [
    (32768, 36620, 23686.0, 100.0, 1e-2, 18e3, 30e3),
    (32768, 3000, 23686.0, 120.0, 1.0, 18e3, 30e3),
    (32768, 60, 23700.0, 115.0, 10.0, 21e3, 26.5e3),
    (16384, 7000, 23686.0, 60.0, 1.0, 18e3, 30e3),
    (8192, 20000, 23686.0, 30.0, 0.1, 18e3, 30e3),
    (4096, 50000, 23686.0, 12.0, 0.1, 18e3, 30e3),
    (32768, 36620, 80e3, 8.0, 2.0, 20.0, 499e3),
]
SEEDS = range(6)


def density(M, K, f0, Q, floor, seed):
    """A density with K averages' scatter: products, quotients and sums only."""
    f = np.arange(M // 2 + 1) * (1e6 / M)
    d = f0 * f0 - f * f
    w = f * f0 / Q
    S = f0 * f0 * f0 * f0 / (d * d + w * w) + floor
    u = np.random.default_rng(seed).integers(-(2 ** 20), 2 ** 20, f.size) / 2.0 ** 20
    return S * (1.0 + u * np.sqrt(3.0 / K)) * 0.37


def cases():
    """name, density, bin width, band, most steps, tolerance"""
    for b, (M, K, f0, Q, floor, lo, hi) in enumerate(BANDS):
        for seed in SEEDS:
            yield f"{b}/{seed}", density(M, K, f0, Q, floor, 100 * b + seed), 1e6 / M, lo, hi, 200, 1e-12
    df, band = 1e6 / 32768, (18e3, 30e3)
    S = density(32768, 300, 23686.0, 100.0, 1.0, 7)
    for steps in (0, 1, 3):
        yield f"steps {steps}", S, df, *band, steps, 1e-12
    yield "tolerance 0", S, df, *band, 40, 0.0
    yield "8 bins", S, df, 23.6e3, 23.6e3 + 8 * df, 200, 1e-12
    for name, v in (("zero", 0.0), ("negative", -1.0), ("infinite", np.inf), ("undefined", np.nan)):
        T = S.copy()
        T[700] = v
        yield name, T, df, *band, 200, 1e-12
    yield "flat", np.full(S.size, 2.0), df, *band, 200, 1e-12
    yield "falling", 1.0 / np.arange(1.0, S.size + 1.0), df, *band, 200, 1e-12


@pytest.mark.gpu
def test_recorded_values():
    torch = pytest.importorskip("torch")
    cg = pytest.importorskip("paper_2307_12988_gb300")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    want = json.load(open(GOLDEN))
    for name, S, df, lo, hi, steps, tol in cases():
        out = cg.Psd.resonance(torch.from_numpy(S).cuda(), df, lo, hi, steps, tol)
        assert [float(v).hex() for v in out] == want[name], name
