"""The general transform's readout (GPU) against FP64 transforms.

Frame lengths cover every radix (2, 3, 5, 7, 11, 13), every pair of radices
taken in one pass, an even last radix (padded buffer), the real, coset and
odd-length forms, short and long frames; batches of one frame,
ragged batches and frames at an odd sample (2-byte aligned).  Full-range int16
samples: |d amps| <= 1e-5 of the frame's rms magnitude (the parity bar of the
readouts; the FP32 transform's rounding is about 1e-7 of it).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _check(dev, N, bins, n, offset=0, **opts):
    rng = np.random.default_rng(N + n)
    x = rng.integers(-32768, 32768, (n, N)).astype(np.int16)
    buf = torch.zeros(offset + n * N, dtype=torch.int16, device=dev)
    buf[offset:] = torch.from_numpy(x.reshape(-1)).to(dev)
    frames = buf[offset:].view(n, N)
    fs = 1.0e9
    ref = rng.uniform(0.5, 2.0, len(bins))
    with cg.Plan(fs, N, np.asarray(bins) * (fs / N), np.arange(len(bins), dtype=float), ref, **opts) as p:
        np.testing.assert_array_equal(p.bins, bins)
        amps, y = p.readout(frames)
        cg.cg_check_device(p.handle)
        kind = p.info["fft_kind"], p.info["coset_modulus"]
    want = np.abs(np.fft.rfft(x.astype(np.float64), axis=1))[:, bins]
    rms = np.sqrt(np.mean(want ** 2))
    assert np.max(np.abs(amps.cpu().numpy() - want)) <= 1e-5 * rms
    assert np.max(np.abs(y.cpu().numpy() - want / ref)) <= 1e-5 * rms / ref.min()
    return kind


# L = N / 2: radices 8, 4, 2, 5, 3, 7, 11, 13 in this order
@pytest.mark.parametrize("N", [12, 16, 20, 28, 26, 30, 32, 36, 42, 48, 64, 90, 98, 154, 242, 338, 512, 1024, 1200,
                               1440, 2310, 2640, 4290, 4400, 12288])
@pytest.mark.parametrize("n,offset", [(1, 0), (701, 1)])
def test_real_transform(dev, N, n, offset):
    rng = np.random.default_rng(N)
    T = min(N // 2 - 1, 60)
    bins = rng.choice(np.arange(0, N // 2 + 1), size=T, replace=False) if N > 12 else np.arange(6)
    bins = np.unique(np.concatenate([[0, 1, N // 2], bins]))[:max(5, T)]
    kind = _check(dev, N, bins, min(n, 4_000_000 // N), offset, fft=cg.FFT_FULL)
    assert kind == (cg.FFT_FULL, 2)


@pytest.mark.parametrize("N", [15, 105, 1155, 3003])
def test_odd_length(dev, N):
    bins = np.unique(np.random.default_rng(N).integers(0, N // 2 + 1, 40))
    assert _check(dev, N, bins, 333, 1)[1] == 1


@pytest.mark.parametrize("N,M,r", [(1000, 10, 1), (2000, 10, 3), (720, 6, 1), (4096, 16, 5), (9000, 50, 7), (13000, 4, 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_coset_transform(dev, N, M, r, offset):
    bins = np.arange(r, N // 2, M)[:100]
    kind = _check(dev, N, bins, 257, offset, path=cg.PATH_SPLIT)      # (not the comb kernels)
    assert kind[0] == cg.FFT_COSET
