"""The Welch kernel's three ways of reading a series (GPU) give the same bits.

16-byte aligned series come by bulk copies, 8-byte aligned ones by 8-byte and
the others and strided ones by 4-byte asynchronous copies; the arithmetic after
that is the same, so the density of the same samples is the same.
"""
import pytest

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,segments", [(4096, 2), (4096, 2500), (8192, 1300), (16384, 611), (32768, 1), (32768, 310)])
def test_alignments_agree(M, segments):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = M + (segments - 1) * (M // 2)
    x = torch.randn(n, device="cuda", generator=torch.Generator("cuda").manual_seed(M + segments)) * 1e6 + 3e5
    with cg.Psd(M) as p:
        def run(offset, stride):
            buf = torch.zeros(offset + n * stride, device="cuda")
            assert buf.data_ptr() % 16 == 0
            buf[offset::stride][:n] = x
            S, K = p.welch(buf[offset:], 1e6, stride=stride, n=n)
            assert K == segments
            return S.clone()
        want = run(0, 1)
        for offset, stride in [(1, 1), (2, 1), (4, 1), (0, 3)]:
            assert torch.equal(run(offset, stride), want), (offset, stride)
