"""Calls of one plan on several streams, captured calls and small calls (GPU).

A plan's kernels run on the caller's stream when a call is one chunk; its fits
share a task counter, so calls on different streams must still give what each
gives alone.  Every result is compared bit for bit with the same frames in one
plain call: the fit of a frame does not depend on its batch.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("amps", "params", "rss", "iters", "status")


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _plan_and_frames(dev, geom, n, **opts):
    s = synth.make_stream(geom, synth.BASE_SEED + 77)
    frames = synth.frames(s, n, snr_db=30.0, center_amp_hz=20e6, device=dev)["frames"]
    ref = np.full(geom.n_teeth, 512.0 * np.sqrt(2.0 / geom.n_teeth) * geom.frame_len / 2.0) * s.envelope
    return cg.Plan(geom.sample_rate, geom.frame_len, geom.tooth_freqs, geom.tooth_x, ref, **opts), frames


def _same(a, b):
    return all(torch.equal(a[k], b[k]) for k in KEYS)


@pytest.mark.parametrize("chunk", [0, 30_000])
def test_calls_on_several_streams(dev, chunk):
    plan, frames = _plan_and_frames(dev, synth.PAPER_RATE, 120_000, chunk_frames=chunk)
    with plan:
        want = plan.process(frames)
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream(dev) for _ in range(3)]
        got = []
        for i in range(9):
            n = (120_000, 70_001, 4_000)[i % 3]
            with torch.cuda.stream(streams[i % 3]):
                got.append((n, plan.process(frames[:n])))
        torch.cuda.synchronize()
        for n, o in got:
            assert _same(o, {k: want[k][:n] for k in KEYS}), n


@pytest.mark.parametrize("n", [500, 100_000])
def test_captured_call(dev, n):
    plan, frames = _plan_and_frames(dev, synth.PAPER_RATE, n)
    with plan:
        want = plan.process(frames)
        other = torch.cuda.Stream(dev)
        with torch.cuda.stream(other):        # the plan's last call is on another stream
            plan.process(frames)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = plan.process(frames)
        for _ in range(2):
            for k in KEYS:
                out[k].zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert _same(out, want)
        assert _same(plan.process(frames), want)


@pytest.mark.parametrize("geom", [synth.TINY, synth.PAPER_RATE, synth.WIDE], ids=["tiny", "paper_rate", "wide"])
def test_small_calls_equal_the_batch(dev, geom):
    plan, frames = _plan_and_frames(dev, geom, 20_000)
    with plan:
        want = plan.process(frames)
        sms = torch.cuda.get_device_properties(dev).multi_processor_count
        for n in (1, 2, 31, 33, 4 * sms - 1, 4 * sms, 4 * sms + 1, 16 * sms + 5, 16 * sms * 8 + 1):
            o = plan.process(frames[:n])
            assert _same(o, {k: want[k][:n] for k in KEYS}), n
