"""Sign of the moment guess (GPU): the first of the largest deviations decides.

Spectra of exact binary values, one tooth above and one below the baseline by
the same amount, in both orders, or one side larger; an iteration cap of zero
returns the guess.  Its amplitude is exact and its centre the abscissa of the
deciding tooth to float32 rounding (relative to the span).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [5, 21, 99, 201, 221])
def test_first_of_the_largest_decides(T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = 10e6 * (np.arange(T) - T // 2)
    rows, want_A, want_c = [], [], []
    for up, down, hi, lo in [(1, 2, 0.5, 0.5), (2, 1, 0.5, 0.5), (1, 2, 0.5, 0.75), (2, 1, 0.5, 0.25), (2, 3, 0.25, 0.25)]:
        y = np.ones(T)
        y[T // 2 - 2 + up] += hi
        y[T // 2 - 2 + down] -= lo
        first_up = hi > lo or (hi == lo and up < down)
        rows.append(y)
        want_A.append(hi if first_up else -lo)
        want_c.append(x[T // 2 - 2 + (up if first_up else down)])
    rows.append(np.ones(T))   # flat
    want_A.append(0.0)
    want_c.append(0.0)
    n = 41                    # more than a warp's rows, ragged
    idx = np.arange(n) % len(rows)
    y = torch.from_numpy(np.asarray(rows, np.float32)[idx]).cuda()
    bins = np.arange(2, T + 2)
    with cg.Plan(1.0e9, 1000, bins * 1.0e6, x, np.ones(T), max_iter=0) as p:
        out = p.fit(y)
        cg.cg_check_device(p.handle)
    got = out["params"].cpu().numpy()
    np.testing.assert_array_equal(got[:, 2], np.asarray(want_A, np.float32)[idx])
    np.testing.assert_array_equal(got[:, 3], 1.0)
    assert np.max(np.abs(got[:, 0] - np.asarray(want_c)[idx])) <= 1e-6 * (x[-1] - x[0])
