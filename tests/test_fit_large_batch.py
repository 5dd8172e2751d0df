"""The standalone fit (GPU) of many spectra: a frame's result is the same in
any batch.

Beyond the frames that the GPU holds at two per lane group the fit takes four
per group (not at 221 teeth, whose rows do not fit): the same sums in the same
order, so every output of the large batch equals those of its parts fit alone,
bit for bit, for tooth counts with several remainders modulo 8, spectra and
magnitudes, starts at any float, flat and undefined spectra.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("params", "rss", "iters", "status")


@pytest.mark.parametrize("T", [5, 16, 21, 50, 99, 110, 221])
def test_batches_agree(T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 45_003
    x = 10e6 * (np.arange(T) - T // 2)
    g = torch.Generator("cuda").manual_seed(T)
    span = float(x[-1] - x[0])
    c = (torch.rand(n, 1, generator=g, device="cuda") - 0.5) * 0.6 * span
    w = (0.03 + 0.1 * torch.rand(n, 1, generator=g, device="cuda")) * span + 5e6
    u = torch.tensor(x, dtype=torch.float32, device="cuda")
    buf = torch.empty(n * T + 3, device="cuda")
    y = buf[3:].view(n, T)
    y.copy_(1 - 0.7 * w ** 2 / ((u - c) ** 2 + w ** 2) + 0.02 * torch.randn(n, T, generator=g, device="cuda"))
    y[7] = 1.0
    y[-1] = float("nan")
    y[n // 2, T // 2] = float("inf")
    bins = np.arange(2, T + 2)
    same = lambda a, b: torch.equal(torch.nan_to_num(a.float(), nan=-7.0), torch.nan_to_num(b.float(), nan=-7.0))
    with cg.Plan(1.0e9, 1000, bins * 1.0e6, x, np.ones(T)) as p:
        want = p.fit(y)
        again = p.fit(y)
        cg.cg_check_device(p.handle)
        for k in KEYS:
            assert same(again[k], want[k]), k
        for a, b in [(0, 1), (0, 9_001), (9_001, 20_000), (20_000, 20_003), (28_000, n)]:
            part = p.fit(y[a:b])
            for k in KEYS:
                assert same(part[k], want[k][a:b]), (k, a, b)
