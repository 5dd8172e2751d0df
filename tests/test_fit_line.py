"""The standalone fit (GPU) on both sides of its rule on the number of spectra.

Up to what fit_kernel holds at once (96 spectra an SM up to 221 teeth) a call
goes to it, beyond that to fit8_kernel: the same sums in the same order, so a
large call equals calls on its parts bit for bit, for every remainder of the
tooth count modulo 8, rows at any float, given starting points, an iteration
cap of zero, magnitudes instead of spectra, flat and undefined spectra.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("params", "rss", "iters", "status")


def _equal(a, b):
    return all(torch.equal(torch.nan_to_num(a[k].float(), nan=-7.0), torch.nan_to_num(b[k].float(), nan=-7.0)) for k in KEYS)


def _parts(call, n):
    out = [call(a, min(a + 4000, n)) for a in range(0, n, 4000)]
    return {k: torch.cat([o[k] for o in out]) for k in KEYS}


@pytest.mark.parametrize("T", [5, 16, 21, 50, 92, 99, 200, 201, 222, 223])
def test_large_calls_equal_their_parts(T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = 96 * sms
    n = line + 1501
    x = 10e6 * (np.arange(T) - T // 2)
    g = torch.Generator("cuda").manual_seed(T)
    span = float(x[-1] - x[0])
    c = (torch.rand(n, 1, generator=g, device="cuda") - 0.5) * 0.6 * span
    w = (0.03 + 0.1 * torch.rand(n, 1, generator=g, device="cuda")) * span + 5e6
    u = torch.tensor(x, dtype=torch.float32, device="cuda")
    y = 1 - 0.7 * w ** 2 / ((u - c) ** 2 + w ** 2) + 0.02 * torch.randn(n, T, generator=g, device="cuda")
    y[3], y[n - 2] = 1.0, float("nan")
    y[n // 2, T // 2], y[n // 3, 0] = float("inf"), float("nan")
    bins = np.arange(2, T + 2)
    for opts in ({}, {"max_iter": 0}):
        with cg.Plan(1.0e9, 1000, bins * 1.0e6, x, np.ones(T), **opts) as p:
            want = _parts(lambda a, b: p.fit(y[a:b]), n)
            for m in (line - 1, line, line + 1, n):
                assert _equal(p.fit(y[:m]), {k: want[k][:m] for k in KEYS}), m
            p0 = want["params"].clone()
            again = _parts(lambda a, b: p.fit(y[a:b], p0[a:b]), n)
            assert _equal(p.fit(y, p0), again)
            for off in (1, 2, 3):
                buf = torch.empty(off + n * T, device="cuda")
                buf[off:] = y.reshape(-1)
                assert _equal(p.fit(buf[off:].view(n, T)), want), off
            cg.cg_check_device(p.handle)


def test_magnitudes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.TINY
    n = 96 * torch.cuda.get_device_properties(0).multi_processor_count + 77
    s = synth.make_stream(g, synth.BASE_SEED + 93)
    frames = synth.frames(s, n, snr_db=30.0, center_amp_hz=5e6, device=torch.device("cuda:0"))["frames"]
    ref = np.full(g.n_teeth, 512.0 * np.sqrt(2.0 / g.n_teeth) * g.frame_len / 2.0) * s.envelope
    with cg.Plan(g.sample_rate, g.frame_len, g.tooth_freqs, g.tooth_x, ref, path=cg.PATH_SPLIT) as p:
        want = _parts(lambda a, b: p.process(frames[a:b], want_y=False), n)
        assert _equal(p.process(frames, want_y=False), want)
        assert _equal(p.process(frames), want)
