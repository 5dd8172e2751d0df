"""Captured calls of one plan share nothing with other calls in flight (GPU).

A captured fit walks its tasks at a fixed stride, a live one claims them from a
counter: both give the same bits at every batch size and fit kernel.  Calls on
two branches of one capture, two graphs replayed on two streams and a replay
beside live calls give what each call gives alone; with the learned guess,
whose fallback list belongs to the plan, two branches of one capture do.
"""
import os

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("params", "rss", "iters", "status")
GEOMETRIES = {
    "tiny": (synth.TINY, {}),                                  # one lane per frame
    "paper_rate": (synth.PAPER_RATE, {}),                      # two
    "wide": (synth.WIDE, {}),                                  # four
    "teeth 80": (synth.Geometry(1.1e9, 1100, -40, 39), {}),    # register kernels
    "lanes 1": (synth.Geometry(1.1e9, 1100, -40, 39), dict(lanes_per_frame=1)),
    "lanes 32": (synth.PAPER_RATE, dict(lanes_per_frame=32)),
    "fp64": (synth.PAPER_RATE, dict(solve_f64=1)),
}


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _plan_and_frames(dev, geom, n, **opts):
    s = synth.make_stream(geom, synth.BASE_SEED + 91)
    frames = synth.frames(s, n, snr_db=20.0, center_amp_hz=20e6, device=dev)["frames"]
    ref = np.full(geom.n_teeth, 512.0 * np.sqrt(2.0 / geom.n_teeth) * geom.frame_len / 2.0) * s.envelope
    return cg.Plan(geom.sample_rate, geom.frame_len, geom.tooth_freqs, geom.tooth_x, ref, **opts), frames


def _same(a, b):
    return all(torch.equal(a[k], b[k]) for k in KEYS)


def _clear(*outs):
    for o in outs:
        for k in KEYS:
            o[k].zero_()


def _capture(call):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call()
    return graph, out


@pytest.mark.parametrize("name", list(GEOMETRIES))
@pytest.mark.parametrize("n", [1, 37, 20_011, 100_003])
def test_captured_equals_live(dev, name, n):
    geom, opts = GEOMETRIES[name]
    plan, frames = _plan_and_frames(dev, geom, n, **opts)
    with plan:
        want = plan.process(frames)
        fits = plan.fit(want["y"])
        graph, out = _capture(lambda: (plan.process(frames), plan.fit(want["y"])))
        _clear(*out)
        graph.replay()
        torch.cuda.synchronize()
        assert _same(out[0], want)
        assert _same(out[1], fits)


def _calls(plan, frames, y):
    return {"process": lambda: plan.process(frames), "fit": lambda: plan.fit(y)}


@pytest.mark.parametrize("kind", ["process", "fit"])
def test_two_branches_two_graphs_and_a_live_call(dev, kind):
    plan, frames = _plan_and_frames(dev, synth.PAPER_RATE, 100_000)
    with plan:
        y = plan.process(frames)["y"]
        call = _calls(plan, frames, y)[kind]
        want = call()
        torch.cuda.synchronize()
        side = torch.cuda.Stream(dev)

        def branches():
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                b = call()
            a = call()
            torch.cuda.current_stream().wait_stream(side)
            return a, b

        graph, (a, b) = _capture(branches)
        for _ in range(5):
            _clear(a, b)
            graph.replay()
            torch.cuda.synchronize()
            assert _same(a, want) and _same(b, want)

        one, out1 = _capture(call)
        two, out2 = _capture(call)
        s1, s2, s3 = (torch.cuda.Stream(dev) for _ in range(3))
        for _ in range(10):
            _clear(out1, out2)
            torch.cuda.synchronize()
            with torch.cuda.stream(s1):
                one.replay()
            with torch.cuda.stream(s2):
                two.replay()
            with torch.cuda.stream(s3):
                live = call()
            torch.cuda.synchronize()
            assert _same(out1, want) and _same(out2, want) and _same(live, want)


def test_learned_guess_on_two_branches(dev):
    blob = open(os.path.join(os.path.dirname(cg.__file__), "data", "mlp_wide_t221.cgmlp"), "rb").read()
    plan, frames = _plan_and_frames(dev, synth.WIDE, 30_000, init=cg.INIT_MLP, polish_iter=1)
    with plan:
        plan.mlp_load(blob)
        want = [plan.process(frames), plan.process(frames.flip(0).contiguous())]
        assert (want[0]["status"] & cg.FIT_FALLBACK).any()
        flipped = frames.flip(0).contiguous()
        torch.cuda.synchronize()
        side = torch.cuda.Stream(dev)

        def branches():
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                b = plan.process(flipped)
            a = plan.process(frames)
            torch.cuda.current_stream().wait_stream(side)
            return a, b

        graph, out = _capture(branches)
        for _ in range(5):
            _clear(*out)
            graph.replay()
            torch.cuda.synchronize()
            assert _same(out[0], want[0]) and _same(out[1], want[1])
