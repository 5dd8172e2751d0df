"""The comb readout kernels (GPU) against FP64 transforms.

Every instantiated length (N = 1000, 1100, 2200, 2500), odd and even residues
(the fold's two signs), full-range samples, batches around a block's frames
and around a round of the grid, starts at every alignment the entry points
take.  |d amps| <= 1e-5 of the rms magnitude, the parity bar of the readouts
(the FP32 transform's rounding is about 1e-7 of it), and a frame's values do
not depend on the batch it comes in.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

MOST = 12_345   # frames: more than one round of every grid


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("N,r,bits", [(1000, 1, 16), (1000, 2, 16), (1100, 3, 16), (1100, 4, 16), (2200, 1, 16),
                                      (2200, 4, 16), (2500, 1, 16), (2500, 2, 16), (2200, 1, 8), (2200, 2, 8)])
def test_against_fp64(dev, N, r, bits):
    rng = np.random.default_rng(N + r + bits)
    dtype = np.int16 if bits == 16 else np.int8
    lim = 1 << (bits - 1)
    bins = np.sort(np.concatenate([np.arange(r, N // 2, 10), np.arange(10 - r, N // 2, 10)]))[:221]
    T = len(bins)
    ref = rng.uniform(0.5, 2.0, T)
    x = rng.integers(-lim, lim, (MOST, N)).astype(dtype)
    x[0], x[1], x[2] = -lim, lim - 1, np.where(np.arange(N) % 2, -lim, lim - 1)
    host = torch.from_numpy(x)
    sub = rng.choice(MOST, 400, replace=False)
    sub[:3] = 0, 1, 2
    want = np.abs(np.fft.rfft(x[sub].astype(np.float64), axis=1))[:, bins]
    rms = np.sqrt(np.mean(want ** 2))
    with cg.Plan(1.0e9, N, bins * (1.0e9 / N), np.arange(T, dtype=float), ref) as p:
        np.testing.assert_array_equal(p.bins, bins)
        assert (p.info["fft_kind"], p.info["coset_modulus"]) == (cg.FFT_COSET, 10)
        amps, y = p.readout(host.to(dev))
        cg.cg_check_device(p.handle)
        assert np.max(np.abs(amps.cpu().numpy()[sub] - want)) <= 1e-5 * rms
        assert np.max(np.abs(y.cpu().numpy()[sub] - want / ref)) <= 1e-5 * rms / ref.min()
        # starts: 4-byte steps for int16, single samples for int8
        for n, offset in [(1, 0), (1, 2), (4, 6), (5, 1), (6, 3), (11, 2), (12, 0), (13, 5), (257, 7), (2000, 2), (9973, 1)]:
            off = offset if bits == 8 else 2 * offset
            buf = torch.zeros(off + n * N, dtype=host.dtype, device=dev)
            buf[off:] = host[:n].reshape(-1).to(dev)
            an, yn = p.readout(buf[off:].view(n, N))
            cg.cg_check_device(p.handle)
            assert torch.equal(an, amps[:n]) and torch.equal(yn, y[:n]), (n, off)
