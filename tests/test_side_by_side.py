"""Fits of one plan on several streams and from several threads (GPU).

A fit on one stream does not wait for a fit that another stream has not begun;
more streams than task counters, and threads with a stream each, give what each
call gives alone, bit for bit.
"""
import threading

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2307_12988_gb300")

pytestmark = pytest.mark.gpu

KEYS = ("params", "rss", "iters", "status")
N = 60_000   # more tasks than warps: the counters are used


@pytest.fixture(scope="module")
def plan_and_spectra():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.PAPER_RATE
    s = synth.make_stream(g, synth.BASE_SEED + 92)
    frames = synth.frames(s, N, snr_db=20.0, center_amp_hz=20e6, device=torch.device("cuda:0"))["frames"]
    ref = np.full(g.n_teeth, 512.0 * np.sqrt(2.0 / g.n_teeth) * g.frame_len / 2.0) * s.envelope
    plan = cg.Plan(g.sample_rate, g.frame_len, g.tooth_freqs, g.tooth_x, ref)
    y = plan.process(frames)["y"]
    want = plan.fit(y)
    torch.cuda.synchronize()
    yield plan, y, want
    plan.close()


def _same(a, b, n=N):
    return all(torch.equal(a[k][:n], b[k][:n]) for k in KEYS)


def test_a_waiting_stream_holds_no_other(plan_and_spectra):
    plan, y, want = plan_and_spectra
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    for s in (one, two):                      # workspaces of both streams
        with torch.cuda.stream(s):
            plan.fit(y)
    torch.cuda.synchronize()
    with torch.cuda.stream(one):
        torch.cuda._sleep(1_000_000_000)      # about half a second
        a = plan.fit(y)
        done = torch.cuda.Event()
        done.record()
    with torch.cuda.stream(two):
        b = plan.fit(y)
    two.synchronize()
    assert not done.query()
    torch.cuda.synchronize()
    assert _same(a, want) and _same(b, want)


def test_more_streams_than_counters(plan_and_spectra):
    plan, y, want = plan_and_spectra
    streams = [torch.cuda.Stream() for _ in range(13)]
    out = []
    for i in range(52):
        n = (N, 40_001, 25_000)[i % 3]
        with torch.cuda.stream(streams[i % 13]):
            out.append((n, plan.fit(y[:n])))
    torch.cuda.synchronize()
    assert all(_same(o, want, n) for n, o in out)


def test_threads_with_a_stream_each(plan_and_spectra):
    plan, y, want = plan_and_spectra
    bad = []

    def work():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            outs = [plan.fit(y) for _ in range(20)]
        s.synchronize()
        bad.extend(i for i, o in enumerate(outs) if not _same(o, want))

    threads = [threading.Thread(target=work) for _ in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
