"""The Welch sums (GPU) are FP64 sums in a fixed order, bit for bit.

|X_k|^2 of a segment is an FP32 value, which the density of that segment alone
gives back exactly.  Row r of R = min(K, SMs x rows per SM) adds up segments
r, r + R, ... one after another and the rows are added in order, all in FP64:
numpy does the same additions.  The sums reach as far as FP64: finite powers
whose FP32 sum overflows, and powers of FP32's smallest normal values.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

ROWS = {4096: 2, 8192: 1, 16384: 1, 32768: 1}   # rows of sums per SM


def _scale(M, K, fs):
    w = np.array([np.float32(0.5 - 0.5 * math.cos(2.0 * math.pi * n / M)) for n in range(M)], dtype=np.float64)
    sum_w2 = 0.0
    for v in w * w:
        sum_w2 += float(v)
    return 1.0 / (float(K) * fs * sum_w2)


def _powers(p, x, M, fs):
    """|X_k|^2 of every segment [K, M / 2 + 1], from the densities of single segments."""
    K = (x.numel() - M) // (M // 2) + 1
    one = torch.stack([p.welch(x[s * (M // 2):s * (M // 2) + M], fs)[0] for s in range(K)]).cpu().numpy()
    c = np.full(M // 2 + 1, 2.0)
    c[0] = c[-1] = 1.0
    return (one / (_scale(M, 1, fs) * c)).astype(np.float32).astype(np.float64), c


@pytest.mark.parametrize("M,segments", [(4096, 1), (4096, 300), (4096, 1400), (8192, 3), (8192, 470), (16384, 461),
                                        (32768, 60), (32768, 310)])
@pytest.mark.parametrize("amplitude", [1e6, 1.2e16, 3e-23])
def test_sums_are_fp64_in_order(M, segments, amplitude):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = M + (segments - 1) * (M // 2)
    t = torch.arange(n, device="cuda", dtype=torch.float64)
    x = torch.randn(n, device="cuda", dtype=torch.float64, generator=torch.Generator("cuda").manual_seed(M + segments))
    # a line on the middle of a bin: its power is the largest of a segment
    line = 1.0e3 if amplitude > 1e10 else 2.0
    x = ((line * torch.cos(2 * math.pi * (M // 8) / M * t) + 0.3 * x) * (amplitude / line * 4096 / M)).float()
    fs = 1e6
    with cg.Psd(M) as p:
        P, c = _powers(p, x, M, fs)
        S, K = p.welch(x, fs)
    assert K == segments
    assert np.isfinite(P).all()
    R = min(K, ROWS[M] * torch.cuda.get_device_properties(0).multi_processor_count)
    total = np.zeros(M // 2 + 1)
    for r in range(R):
        row = np.zeros(M // 2 + 1)
        for s in range(r, K, R):
            row += P[s]
        total += row
    np.testing.assert_array_equal(S.cpu().numpy(), total * _scale(M, K, fs) * c)
    if amplitude > 1e10 and segments >= 60:
        assert total.max() > np.finfo(np.float32).max
