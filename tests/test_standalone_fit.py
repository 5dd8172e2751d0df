"""The standalone fit (GPU): tooth counts, batches, alignments and odd spectra.

``Plan.fit`` (eight lanes a frame, two frames a lane group) against the fused
kernel's fit on the same spectra bit for bit (the same sums in the same
order), for tooth counts with every remainder modulo 8, one frame and ragged
batches, spectra that start at any float, flat and undefined spectra, given
starting points and an iteration cap of zero.  The fused kernel (CG_PATH_FUSED)
writes the spectra it fits, so its y is the input of the standalone fit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("params", "rss", "iters", "status")


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _instrument(T, seed, **opts):
    rng = np.random.default_rng(seed)
    N = 480
    bins = rng.choice(np.arange(2, N // 2 - 1), size=T, replace=False)
    x = np.cumsum(rng.uniform(0.6, 1.4, T)) * 10e6
    x -= x.mean()
    amp = 512 * np.sqrt(2.0 / T) * rng.uniform(0.9, 1.1, T)
    args = (1.0e9, N, bins * (1.0e9 / N), x, amp * N / 2.0)
    return N, bins, x, amp, args


def _frames(dev, N, bins, x, amp, n, seed):
    rng = np.random.default_rng(seed)
    span = x[-1] - x[0]
    c = rng.uniform(-0.2, 0.2, (n, 1)) * span
    g = rng.uniform(2.0, 5.0, (n, 1)) * span / (x.size - 1)
    L = 1 - 0.7 * g ** 2 / ((x - c) ** 2 + g ** 2)
    basis = np.cos(2 * np.pi * np.outer(bins, np.arange(N)) / N + rng.uniform(0, 2 * np.pi, x.size)[:, None])
    f = (L * amp) @ basis + rng.normal(0, 20.0, (n, N))
    return torch.from_numpy(np.clip(np.rint(f), -2048, 2047).astype(np.int16)).to(dev)


def _same(a, b, rows=slice(None)):
    for k in KEYS:
        x, y = a[k][rows], b[k][rows]
        assert torch.equal(torch.nan_to_num(x.float(), nan=-7.0), torch.nan_to_num(y.float(), nan=-7.0)), k


@pytest.mark.parametrize("T", [5, 8, 16, 21, 33, 50, 63, 92, 99, 200, 221])
def test_equals_the_fused_fit(dev, T):
    N, bins, x, amp, args = _instrument(T, T)
    n = 1003
    frames = _frames(dev, N, bins, x, amp, n, T)
    with cg.Plan(*args, path=cg.PATH_FUSED) as fused, cg.Plan(*args, path=cg.PATH_SPLIT) as split:
        want = fused.process(frames)
        y = want["y"]
        _same(split.fit(y), want)
        _same(split.process(frames, want_y=False), want)           # magnitudes and 1 / ref
        for m in (1, 7, 8, 9, 33):
            _same(split.fit(y[:m]), {k: want[k][:m] for k in KEYS})
        for off in (1, 2, 3):                                      # rows at any float
            buf = torch.zeros(off + y.numel(), device=dev)
            buf[off:] = y.reshape(-1)
            _same(split.fit(buf[off:].view(n, T)), want)


def test_flat_and_undefined_spectra(dev):
    T = 99
    N, bins, x, amp, args = _instrument(T, 7)
    frames = _frames(dev, N, bins, x, amp, 64, 7)
    with cg.Plan(*args) as plan:
        y = plan.readout(frames)[1]
        good = plan.fit(y)
        bad = y.clone()
        bad[3] = 1.0                        # flat
        bad[4] = 0.0
        bad[10, 50] = float("nan")          # inside
        bad[11, 0] = float("nan")           # among the outer teeth
        bad[12] = float("nan")
        bad[20, 98] = float("inf")
        out = plan.fit(bad)
        odd = [3, 4, 10, 11, 12, 20]
        keep = [i for i in range(64) if i not in odd]
        _same(out, good, keep)              # neighbours are not touched
        st = out["status"].cpu().numpy()
        assert all(st[i] & cg.FIT_INIT_FLAT for i in (3, 4))
        assert all((st[i] & 3) == cg.FIT_NONFINITE for i in (10, 11, 12, 20))


@pytest.mark.parametrize("max_iter", [0, 1, 20])
def test_given_starting_points_and_caps(dev, max_iter):
    T = 50
    N, bins, x, amp, args = _instrument(T, 9)
    frames = _frames(dev, N, bins, x, amp, 500, 9)
    with cg.Plan(*args, max_iter=max_iter) as plan:
        y = plan.readout(frames)[1]
        out = plan.fit(y)
        if max_iter == 0:
            assert (out["iters"] == 0).all() and ((out["status"] & 3) == cg.FIT_MAX_ITER).all()
        p0 = out["params"].clone()
        again = plan.fit(y, p0)
        alone = plan.fit(y[17:18], p0[17:18])
        _same(alone, {k: again[k][17:18] for k in KEYS})
        if max_iter == 20:
            ok = ((out["status"] & 3) == 0) & ((again["status"] & 3) == 0)
            assert ok.float().mean() >= 0.98
            fwhm = 2 * out["params"][ok, 1]
            assert ((again["params"][ok, 0] - out["params"][ok, 0]).abs() <= 2e-3 * fwhm).all()
