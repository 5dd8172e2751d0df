"""Device memory of the training object, and its first step (GPU).

An object that runs forward only, or only batches beyond the step on operand
images, holds its FP32 buffers and the weights' images; the batch images come
with the first step that uses them.  A first step under capture takes the
generic products and gives the same bits, and the weights' images follow the
parameters that a replay leaves.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

SLACK = 64 << 20   # allocation granularity and the module's own first use


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with cg_net(8, 16, 4, 128) as net:   # (loads the library's kernels)
        net.train_epoch(*_set(128, 8, 4), 128, 1e-3)
    torch.cuda.synchronize()
    return torch.device("cuda:0")


class cg_net:
    def __init__(self, *a, **k):
        self.net = cg.Mlp(a[0], a[1], a[2], max_batch=a[3], **k)

    def __enter__(self):
        return self.net

    def __exit__(self, *_):
        self.net.close()


def _set(n, n_in, n_out, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn((n, n_in), generator=g, device="cuda"), torch.randn((n, n_out), generator=g, device="cuda"),
            torch.randperm(n, generator=g, device="cuda").to(torch.int32))


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("shape,max_batch,step", [((1024, 1024, 4), 16384, 0), ((221, 256, 4), 16384, 0),
                                                  ((221, 256, 4), 40000, 20000)])
def test_forward_and_large_batches_need_no_images(dev, shape, max_batch, step):
    n_in, H, n_out = shape
    x, t, _ = _set(max(step, 300), n_in, n_out)
    params = H * n_in + H + H * H + H + n_out * H + n_out
    rows = 6 * H + n_in + 3 * n_out
    images = 2 * (H + 128) * (n_in + 3 * H + 192)          # weights, padded to 128 rows and 32 columns
    want = 4 * (4 * params + max_batch * rows + 8 * H * max(H, n_in) + images)
    before = _free()
    with cg_net(n_in, H, n_out, max_batch) as net:
        net.forward(x[:300])
        if step:
            net.backward(x, t)
        assert before - _free() <= want + SLACK
        net.backward(x[:300], t[:300])
        assert before - _free() > want                      # (the images are what the bound leaves out)
    assert _free() >= before - SLACK


def test_first_step_under_capture(dev):
    n_in, H, n_out, n = 33, 80, 4, 300
    x, t, perm = _set(n, n_in, n_out, seed=5)
    with cg_net(n_in, H, n_out, 128, seed=3) as live, cg_net(n_in, H, n_out, 128, seed=3) as replayed:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            losses = replayed.train_epoch(x, t, perm, 128, 1e-3)
        graph.replay()
        want = live.train_epoch(x, t, perm, 128, 1e-3)
        assert torch.equal(losses, want)
        np.testing.assert_array_equal(replayed.params(), live.params())
        # the next step runs on the images
        (l1, g1), (l2, g2) = replayed.backward(x[:100], t[:100]), live.backward(x[:100], t[:100])
        assert torch.equal(l1, l2) and torch.equal(g1, g2)
        # and a replay after it is followed by them too
        graph.replay()
        theta = replayed.params()
        l1, g1 = replayed.backward(x[:100], t[:100])
    with cg_net(n_in, H, n_out, 128) as fresh:
        fresh.set_params(theta)
        l2, g2 = fresh.backward(x[:100], t[:100])
        assert torch.equal(l1, l2) and torch.equal(g1, g2)
