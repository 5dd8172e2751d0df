"""The training step on operand images (GPU): edges of its tiles and batches.

``train_epoch`` equals ``backward`` + ``adam`` on the same gathered rows bit
for bit (the products and sums have one order); a batch gives the same
gradient whatever ran before it (padding stays zero); entries of the
permutation outside the set are zero rows; batches beyond the step's limit
take the generic products, within the same bounds of the FP64 oracle as the
others (loss 1e-5, gradient blocks 1e-4 of their largest entry).
"""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _set(dev, n, n_in, n_out, seed=0):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return (torch.randn((n, n_in), generator=g, device=dev), torch.randn((n, n_out), generator=g, device=dev))


@pytest.mark.parametrize("shape", [(221, 256, 4), (33, 48, 1), (31, 257, 16), (5, 16, 3)])
@pytest.mark.parametrize("batch", [1, 33, 128, 200])
def test_epoch_equals_single_steps(dev, shape, batch):
    n_in, H, n_out = shape
    n = 2 * batch + (batch + 1) // 2
    x, t = _set(dev, n, n_in, n_out)
    perm = torch.from_numpy(np.random.default_rng(1).permutation(n).astype(np.int32)).to(dev)
    one, two = (cg.Mlp(n_in, H, n_out, max_batch=batch, seed=5) for _ in range(2))
    losses = one.train_epoch(x, t, perm, batch, 1e-3)
    want = []
    for r in range(0, n, batch):
        rows = perm[r:r + batch].long()
        want.append(two.backward(x[rows].contiguous(), t[rows].contiguous())[0])
        two.adam(1e-3)
    assert torch.equal(losses, torch.cat(want))
    np.testing.assert_array_equal(one.params(), two.params())


def test_batch_after_larger_batch(dev):
    x, t = _set(dev, 700, 99, 4)
    net, fresh = (cg.Mlp(99, 256, 4, max_batch=700, seed=2) for _ in range(2))
    net.backward(x, t)
    for n in (513, 129, 128, 31, 1):
        l1, g1 = net.backward(x[:n], t[:n])
        l2, g2 = fresh.backward(x[:n], t[:n]) if n == 513 else cg.Mlp(99, 256, 4, max_batch=n, seed=2).backward(x[:n], t[:n])
        assert torch.equal(l1, l2) and torch.equal(g1, g2), n


def test_permutation_entries_outside_the_set(dev):
    x, t = _set(dev, 64, 21, 4)
    perm = torch.arange(64, dtype=torch.int32, device=dev)
    perm[5], perm[40] = -1, 64
    zx, zt = x.clone(), t.clone()
    zx[5], zx[40], zt[5], zt[40] = 0, 0, 0, 0
    one, two = (cg.Mlp(21, 64, 4, max_batch=64, seed=9) for _ in range(2))
    l1 = one.train_epoch(x, t, perm, 64, 1e-3)
    l2 = two.train_epoch(zx, zt, torch.arange(64, dtype=torch.int32, device=dev), 64, 1e-3)
    assert torch.equal(l1, l2)
    np.testing.assert_array_equal(one.params(), two.params())


@pytest.mark.parametrize("n", [16384, 16385])
def test_batches_around_the_limit(dev, n):
    n_in, H, n_out = 24, 40, 4
    x, t = _set(dev, n, n_in, n_out, seed=3)
    net = cg.Mlp(n_in, H, n_out, max_batch=n, seed=4)
    theta = net.params().astype(np.float64)
    loss, grad = net.backward(x, t)
    L, g = omlp.loss_and_grad(theta, x.cpu().numpy().astype(np.float64), t.cpu().numpy().astype(np.float64), n_in, H,
                              n_out)
    assert abs(loss.item() - L) <= 1e-5 * L
    grad = grad.cpu().numpy().astype(np.float64)
    at = np.cumsum([0, H * n_in, H, H * H, H, n_out * H, n_out])
    for a, b in zip(at[:-1], at[1:]):
        assert np.max(np.abs(grad[a:b] - g[a:b])) <= 1e-4 * np.max(np.abs(g[a:b]))
    net.adam(1e-3)                                   # and the images of the weights follow
    l2, _ = net.backward(x[:100], t[:100])
    L2, _ = omlp.loss_and_grad(net.params().astype(np.float64), x[:100].cpu().numpy().astype(np.float64),
                               t[:100].cpu().numpy().astype(np.float64), n_in, H, n_out)
    assert abs(l2.item() - L2) <= 1e-5 * L2
