"""Workloads whose time is tracked: what a program that uses this library has
it do, through the public entry points, over the sizes it is used at.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``process``  ``Plan.process`` on resident frames: readout, starting point and
  Lorentzian fit of every frame (``paper8``: the 8-bit configuration, with the
  median-filtered centre and the boxed Fano fit);
* ``readout``  ``Plan.readout`` of an instrument whose teeth lie on arbitrary
  bins (no comb structure to exploit);
* ``fit``      ``Plan.fit`` on spectra that were normalised elsewhere;
* ``guess``    ``Plan.mlp_infer``: the learned starting point;
* ``train``    ``Mlp.train_epoch``: one epoch of that network's training;
* ``psd``      ``Psd.welch`` of the fitted centres and ``Psd.resonance``.

``listed()`` gives the fixed cases, ``draw()`` further ones of the same ranges,
``prepare()`` what the program has in hand before the call, ``run()`` one call,
``work()`` the bytes and operations a call cannot do without, and ``exact()``
the result in 64-bit arithmetic by plain torch or numpy.
"""
import math
import os
import struct

import numpy as np
import torch

import paper_2307_12988_gb300 as cg

HERE = os.path.dirname(os.path.abspath(__file__))
SHIPPED_NET = os.path.join(os.path.dirname(HERE), "paper_2307_12988_gb300", "data", "mlp_wide_t221.cgmlp")

# Instruments: digitiser rate, samples per frame, lowest and highest tooth, bits
# per sample.  Teeth lie at |51 + 10 k| MHz; the fit abscissa is 10 k MHz.
INSTRUMENTS = {
    "tiny": (1.0e9, 1000, -10, 10, 12),
    "paper_rate": (1.1e9, 1100, -49, 49, 12),
    "wide": (2.5e9, 2500, -110, 110, 12),
    "serve4096": (2.0e9, 4096, -100, 100, 12),
    "paper8": (2.2e9, 2200, -49, 49, 8),
}
# frames above which a call of that instrument exceeds 2.6 GB of input and output
MOST_FRAMES = {"tiny": 1_000_000, "paper_rate": 1_000_000, "wide": 400_000, "serve4096": 250_000, "paper8": 750_000}
FWHM = 80e6          # cavity linewidth
DRIVE = 23.686e3     # mechanical resonance that drives the centre
DEPTH = 0.7          # depth of the cavity dip
SNR_DB = 30.0        # time-domain signal to noise
FANO_Q = 0.3         # asymmetry of the Fano profile
HIDDEN = 256         # hidden width of the network


def listed():
    return [
        # one small batch, as a control loop or a serving stream hands over: latency and launches
        {"name": "process_batch_200", "kind": "process", "instrument": "paper_rate", "n": 200},
        # a short record of the smallest instrument, no multiple of anything
        {"name": "process_tiny_ragged", "kind": "process", "instrument": "tiny", "n": 9973},
        # one second of frames at the paper's rate: the headline workload
        {"name": "process_paper_rate_1s", "kind": "process", "instrument": "paper_rate", "n": 1_000_000},
        # a tenth of a second of the wide comb, odd count
        {"name": "process_wide_ragged", "kind": "process", "instrument": "wide", "n": 100_003},
        # the serving stream with 2.048 us frames (teeth between bins: full transform)
        {"name": "process_serve4096", "kind": "process", "instrument": "serve4096", "n": 30_000},
        # the paper's own configuration: 8-bit samples, median-filtered centre, boxed Fano fit
        {"name": "process_paper8_fano", "kind": "process", "instrument": "paper8", "n": 250_000},
        # an instrument without comb structure: teeth on arbitrary bins
        {"name": "readout_arbitrary", "kind": "readout", "samples": 2640, "teeth": 80, "n": 20_000},
        # spectra that were read out and normalised elsewhere: the fit alone
        {"name": "fit_spectra", "kind": "fit", "instrument": "paper_rate", "n": 100_000},
        # the learned starting point of the wide comb, with the shipped network
        {"name": "guess_wide", "kind": "guess", "instrument": "wide", "n": 250_000},
        # training that network: one epoch over a part of the set, the last batch short
        {"name": "train_epoch", "kind": "train", "teeth": 221, "n": 20_000, "batch": 1024},
        # displacement spectrum of one second of centres, straight from the parameter rows
        {"name": "psd_1s", "kind": "psd", "n": 1_000_000, "segment": 32768, "stride": 4},
        # and of ten minutes of centres
        {"name": "psd_10min", "kind": "psd", "n": 600_000_000, "segment": 32768, "stride": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["process", "process", "process", "readout", "fit", "guess", "train", "psd"])
    if kind == "process":
        name = rng.choice(sorted(INSTRUMENTS))
        return {"kind": kind, "instrument": name, "n": _log_int(rng, 32, MOST_FRAMES[name])}
    if kind == "readout":
        while True:   # lengths of the radices the transforms are built from
            n_samples = 2 ** rng.randint(2, 6) * 3 ** rng.randint(0, 2) * 5 ** rng.randint(0, 2) * 11 ** rng.randint(0, 1)
            if 200 <= n_samples <= 4400:
                break
        teeth = rng.randint(21, min(100, n_samples // 2 - 2) - 1)
        return {"kind": kind, "samples": n_samples, "teeth": teeth, "n": _log_int(rng, 32, 200_000)}
    if kind == "fit":
        return {"kind": kind, "instrument": rng.choice(["tiny", "paper_rate", "serve4096", "wide"]),
                "n": _log_int(rng, 32, 400_000)}
    if kind == "guess":
        return {"kind": kind, "instrument": rng.choice(["tiny", "paper_rate", "serve4096", "wide"]),
                "n": _log_int(rng, 32, 1_000_000)}
    if kind == "train":
        batch = _log_int(rng, 64, 4096)
        return {"kind": kind, "teeth": rng.choice([21, 99, 201, 221]), "batch": batch,
                "n": int(batch * rng.uniform(1.0, 12.0))}
    return {"kind": kind, "n": _log_int(rng, 200_000, 100_000_000), "segment": rng.choice([4096, 8192, 16384, 32768]),
            "stride": rng.choice([1, 4])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda:0")


def _generator(seed, stream):
    g = torch.Generator(device=_device())
    g.manual_seed((int(seed) * 1_000_003 + 7919 * stream) % (1 << 62))
    return g


def _host_rng(seed, stream):
    return np.random.default_rng(np.random.SeedSequence([int(seed), stream]))


def _abscissa(instrument):
    _, _, lo, hi, _ = INSTRUMENTS[instrument]
    return 10e6 * np.arange(lo, hi + 1, dtype=np.float64)


def _dip(x, centre, half_width, depth):
    """Lorentzian dip at abscissae x (torch [T]) for per-frame centres [n]."""
    d = x[None, :] - centre[:, None]
    return 1.0 - depth * half_width ** 2 / (d * d + half_width ** 2)


def _fano(x, centre, half_width, depth):
    e = (x[None, :] - centre[:, None]) / half_width
    return (1.0 - depth) + depth * (FANO_Q + e) ** 2 / (1.0 + e * e)


def _quantised(clean, sigma, full, gen, dtype):
    clean.add_(torch.randn(clean.shape, generator=gen, device=clean.device), alpha=sigma)
    return clean.round_().clamp_(-full, full - 1).to(dtype)


def _comb_frames(instrument, n, seed, cavity):
    """Digitised frames [n, N] of a comb instrument: every tooth's amplitude
    shaped by the cavity, whose centre follows the mechanical drive."""
    fs, N, lo, hi, bits = INSTRUMENTS[instrument]
    dev = _device()
    rng = _host_rng(seed, 1)
    T = hi - lo + 1
    full = 2.0 ** (bits - 1)
    rms = full / 4.0
    freq = 51e6 + 10e6 * np.arange(lo, hi + 1, dtype=np.float64)
    envelope = rng.uniform(0.9, 1.1, T)
    phase = rng.uniform(0.0, 2.0 * math.pi, T)
    drive_phase = rng.uniform(0.0, 2.0 * math.pi)
    cycles = np.mod(np.outer(freq, np.arange(N)) / fs, 1.0)
    angle = 2.0 * math.pi * cycles + phase[:, None]
    scale = (rms * math.sqrt(2.0 / T) * envelope)[:, None]
    cos_n = torch.tensor(scale * np.cos(angle), dtype=torch.float32, device=dev)
    sin_n = torch.tensor(scale * np.sin(angle), dtype=torch.float32, device=dev)
    x = torch.tensor(_abscissa(instrument), device=dev)
    f = torch.tensor(freq, device=dev)
    gen = _generator(seed, 2 if cavity else 3)
    out = torch.empty((n, N), dtype=torch.int8 if bits == 8 else torch.int16, device=dev)
    for s in range(0, n, 65536):
        m = min(65536, n - s)
        t0 = (torch.arange(s, s + m, device=dev, dtype=torch.float64)) * (N / fs)
        shape = torch.ones((m, T), dtype=torch.float64, device=dev)
        if cavity:
            centre = 20e6 * torch.sin(2.0 * math.pi * DRIVE * t0 + drive_phase)
            shape = (_fano if bits == 8 else _dip)(x, centre, FWHM / 2.0, DEPTH)
        psi = 2.0 * math.pi * torch.remainder(t0[:, None] * f[None, :], 1.0)
        re = (shape * torch.cos(psi)).float()
        im = (shape * torch.sin(psi)).float()
        sig = re @ cos_n - im @ sin_n
        out[s:s + m] = _quantised(sig, rms / 10.0 ** (SNR_DB / 20.0), full, gen, out.dtype)
    return out


def _magnitudes(frames, bins):
    """|X| at the bins in 64 bits, frames in slices."""
    idx = torch.as_tensor(bins, device=frames.device)
    out = torch.empty((frames.shape[0], idx.numel()), dtype=torch.float64, device=frames.device)
    step = max(1, (1 << 27) // frames.shape[1])
    for s in range(0, frames.shape[0], step):
        out[s:s + step] = torch.fft.rfft(frames[s:s + step].double(), dim=1)[:, idx].abs()
    return out


def _comb_bins(instrument):
    fs, N, lo, hi, _ = INSTRUMENTS[instrument]
    b = np.floor(np.abs(51e6 + 10e6 * np.arange(lo, hi + 1)) * N / fs + 0.5).astype(np.int64) % N
    return np.where(b > N // 2, N - b, b)


def _comb_reference(instrument, seed):
    frames = _comb_frames(instrument, 512, seed, cavity=False)
    return _magnitudes(frames, _comb_bins(instrument)).mean(dim=0).cpu().numpy()


def _fano_options():
    return dict(model=cg.MODEL_FANO, init=cg.INIT_MEDIAN, fano_q=FANO_Q, fano_gamma=FWHM / 2.0, fano_A=DEPTH,
                fano_B=1.0 - DEPTH, fano_box=0.1)


def _comb_plan(instrument, ref, **options):
    fs, N, lo, hi, _ = INSTRUMENTS[instrument]
    return cg.Plan(fs, N, 51e6 + 10e6 * np.arange(lo, hi + 1, dtype=np.float64), _abscissa(instrument), ref, **options)


def _arbitrary(case, seed):
    """Frames, bins, abscissa and reference of an instrument whose teeth lie
    on random distinct bins in random order."""
    dev, rng = _device(), _host_rng(seed, 4)
    N, T, n = case["samples"], case["teeth"], case["n"]
    bins = rng.choice(np.arange(2, N // 2 - 1), size=T, replace=False)
    x = np.cumsum(rng.uniform(0.6, 1.4, T)) * 10e6
    x -= x.mean()
    g = rng.uniform(2.0, 5.0) * (x[-1] - x[0]) / (T - 1)
    c = rng.uniform(-0.2, 0.2) * (x[-1] - x[0])
    amp = 512.0 * math.sqrt(2.0 / T) * rng.uniform(0.9, 1.1, T)
    angle = 2.0 * math.pi * np.mod(np.outer(bins, np.arange(N)), N) / N + rng.uniform(0.0, 2.0 * math.pi, T)[:, None]
    basis = torch.tensor(amp[:, None] * np.cos(angle), dtype=torch.float32, device=dev)
    gen = _generator(seed, 5)
    frames = torch.empty((n, N), dtype=torch.int16, device=dev)
    xt = torch.tensor(x, device=dev)
    for s in range(0, n, 65536):
        m = min(65536, n - s)
        centre = c + 0.02 * (x[-1] - x[0]) * torch.randn(m, generator=gen, device=dev, dtype=torch.float64)
        frames[s:s + m] = _quantised(_dip(xt, centre, g, DEPTH).float() @ basis, 20.0, 2048.0, gen, torch.int16)
    return frames, bins, x, amp * N / 2.0


def _spectra(instrument, n, seed, wander):
    """Normalised tooth spectra [n, T] as the readout gives them: bin noise of
    20 to 40 dB on each tooth phasor, dips of 60 to 100 MHz; also the true
    (c, g, A, B) of each."""
    fs, N, lo, hi, _ = INSTRUMENTS[instrument]
    dev, gen = _device(), _generator(seed, 6)
    T = hi - lo + 1

    def uniform(a, b):
        return a + (b - a) * torch.rand(n, generator=gen, device=dev, dtype=torch.float32)

    c = uniform(-wander, wander)
    g = uniform(30e6, 50e6)
    snr = uniform(20.0, 40.0)
    depth = uniform(0.6, 0.8)
    noise = 512.0 * 10.0 ** (-snr / 20.0) * math.sqrt(N / 2.0) / (512.0 * math.sqrt(2.0 / T) * N / 2.0)
    x = torch.tensor(_abscissa(instrument), dtype=torch.float32, device=dev)
    d = x[None, :] - c[:, None]
    clean = 1.0 - depth[:, None] * (g * g)[:, None] / (d * d + (g * g)[:, None])
    re = clean + noise[:, None] * torch.randn((n, T), generator=gen, device=dev)
    im = noise[:, None] * torch.randn((n, T), generator=gen, device=dev)
    return torch.sqrt(re * re + im * im), torch.stack([c, g, -depth, torch.ones_like(c)], dim=1)


def _net_arrays(blob):
    """(n_in, in_mean, in_scale, out_mean, out_scale, theta) of a saved network."""
    n_in, hidden, n_out, _ = struct.unpack("<4i", blob[8:24])
    v = np.frombuffer(blob[24:], dtype="<f4").astype(np.float64)
    cut = np.cumsum([n_in, n_in, n_out, n_out])
    return (n_in, *np.split(v, cut))


def _net_blob(instrument, seed):
    """A network for the instrument's tooth count: the shipped one where there
    is one, else freshly initialised weights in the saved format."""
    T = _abscissa(instrument).size
    if T == 221:
        with open(SHIPPED_NET, "rb") as f:
            return f.read()
    rng = _host_rng(seed, 7)
    layers = [rng.uniform(-1, 1, (HIDDEN, T)) / math.sqrt(T), 0.1 * rng.uniform(-1, 1, HIDDEN),
              rng.uniform(-1, 1, (HIDDEN, HIDDEN)) / math.sqrt(HIDDEN), 0.1 * rng.uniform(-1, 1, HIDDEN),
              rng.uniform(-1, 1, (4, HIDDEN)) / math.sqrt(HIDDEN), 0.1 * rng.uniform(-1, 1, 4)]
    norm = [np.full(T, 0.9), np.full(T, 5.0), np.array([0.0, 40e6, -0.7, 1.0]), np.array([58e6, 6e6, 0.06, 0.02])]
    body = np.concatenate([a.ravel() for a in norm + layers]).astype("<f4").tobytes()
    return b"CGMLP001" + struct.pack("<4i", T, HIDDEN, 4, 0) + body


def _training_set(case, seed):
    name = {21: "tiny", 99: "paper_rate", 201: "serve4096", 221: "wide"}[case["teeth"]]
    y, p = _spectra(name, case["n"], seed, 0.1 * float(np.ptp(_abscissa(name))) / 2.0)
    gen = _generator(seed, 8)
    p[:, 3] += 0.02 * torch.randn(case["n"], generator=gen, device=y.device)
    x = ((y - y.mean(dim=0)) / y.std(dim=0).clamp_min(1e-6)).contiguous()
    t = ((p - p.mean(dim=0)) / p.std(dim=0)).contiguous()
    perm = torch.randperm(case["n"], generator=gen, device=y.device).to(torch.int32)
    return x, t, perm


def _first_weights(case, seed):
    T = case["teeth"]
    rng = _host_rng(seed, 9)
    parts = [(HIDDEN * T, T), (HIDDEN, 0), (HIDDEN * HIDDEN, HIDDEN), (HIDDEN, 0), (4 * HIDDEN, HIDDEN), (4, 0)]
    return np.concatenate([rng.uniform(-1, 1, k) / math.sqrt(fan) if fan else np.zeros(k)
                           for k, fan in parts]).astype(np.float32)


def _centres(case, seed):
    """Fitted centres at 1 MHz: the thermally driven resonator (23.7 kHz,
    Q = 120, 2 MHz RMS) over a white floor; a record of 2^22 samples is
    repeated with fresh floor noise.  With stride 4 they are column 0 of
    parameter rows."""
    dev, gen = _device(), _generator(seed, 10)
    n, stride = case["n"], case["stride"]
    m = 1 << 22
    f = torch.fft.rfftfreq(m, d=1e-6, device=dev, dtype=torch.float32)
    f0, Q = 23.7e3, 120.0
    shape = f0 * f0 / torch.sqrt((f0 * f0 - f * f) ** 2 + (f * f0 / Q) ** 2)
    z = torch.randn((2, f.numel()), generator=gen, device=dev)
    record = torch.fft.irfft(torch.complex(z[0], z[1]) * shape, n=m)
    record *= 2e6 / record.std()
    out = torch.empty(n * stride, dtype=torch.float32, device=dev)
    if stride > 1:
        out.view(n, stride)[:, 1:] = torch.tensor([FWHM / 2.0, -DEPTH, 1.0], device=dev)
    column = out.view(n, stride)[:, 0]
    for s in range(0, n, m):
        k = min(m, n - s)
        column[s:s + k] = record[:k] + 2e4 * torch.randn(k, generator=gen, device=dev)
    return out


# ---------------------------------------------------------------------------
# a case's state and one call
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "process":
        name = case["instrument"]
        state["frames"] = _comb_frames(name, case["n"], seed, cavity=True)
        options = _fano_options() if name == "paper8" else {}
        state["plan"] = _comb_plan(name, _comb_reference(name, seed), **options)
    elif kind == "readout":
        frames, bins, x, ref = _arbitrary(case, seed)
        state["frames"] = frames
        state["plan"] = cg.Plan(1.0e9, case["samples"], bins * (1.0e9 / case["samples"]), x, ref)
    elif kind == "fit":
        state["y"], _ = _spectra(case["instrument"], case["n"], seed, 20e6)
        state["plan"] = _comb_plan(case["instrument"], None)
    elif kind == "guess":
        name = case["instrument"]
        state["y"], _ = _spectra(name, case["n"], seed, 0.1 * float(np.ptp(_abscissa(name))) / 2.0)
        state["plan"] = _comb_plan(name, None, init=cg.INIT_MLP)
        state["plan"].mlp_load(_net_blob(name, seed))
    elif kind == "train":
        state["x"], state["t"], state["perm"] = _training_set(case, seed)
        state["batch"] = case["batch"]
        state["net"] = cg.Mlp(case["teeth"], HIDDEN, 4, max_batch=case["batch"])
        state["net"].set_params(_first_weights(case, seed))
    else:
        state["x"] = _centres(case, seed)
        state["n"], state["stride"] = case["n"], case["stride"]
        state["psd"] = cg.Psd(case["segment"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "process":
        return state["plan"].process(state["frames"])
    if kind == "readout":
        return state["plan"].readout(state["frames"])
    if kind == "fit":
        return state["plan"].fit(state["y"])
    if kind == "guess":
        return state["plan"].mlp_infer(state["y"])
    if kind == "train":
        losses = state["net"].train_epoch(state["x"], state["t"], state["perm"], state["batch"], 1e-3)
        return {"losses": losses, "params": state["net"].params()}
    density, segments = state["psd"].welch(state["x"], 1e6, stride=state["stride"], n=state["n"])
    return density, segments, cg.Psd.resonance(density, 1e6 / state["psd"].seg_len, 18e3, 30e3)


# ---------------------------------------------------------------------------
# the work a call cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "process":
        _, N, lo, hi, bits = INSTRUMENTS[case["instrument"]]
        T = hi - lo + 1
        # samples in; amplitudes, spectra, parameters, chi^2, steps and status out
        return {"bytes": n * (N * (1 if bits == 8 else 2) + 8 * T + 16 + 4 + 2 + 2),
                "flops": n * (2.5 * N * math.log2(N) + 4 * 35 * T)}
    if kind == "readout":
        N, T = case["samples"], case["teeth"]
        return {"bytes": n * (2 * N + 8 * T), "flops": n * 2.5 * N * math.log2(N)}
    if kind == "fit":
        T = _abscissa(case["instrument"]).size
        return {"bytes": n * (4 * T + 16 + 4 + 2 + 2), "flops": n * 4 * 35 * T}
    if kind == "guess":
        T = _abscissa(case["instrument"]).size
        weights = HIDDEN * (T + HIDDEN + 4)
        return {"bytes": n * (4 * T + 16) + 2 * weights, "flops": 2 * n * weights}
    if kind == "train":
        T = case["teeth"]
        weights = HIDDEN * (T + HIDDEN + 4)
        steps = -(-n // case["batch"])
        # a forward and two backward products per row; weights and both moments read and written per step
        return {"bytes": n * 4 * (T + 4 + 1) + steps * 6 * 4 * weights, "flops": 6 * n * weights}
    M = case["segment"]
    segments = (n - M) // (M // 2) + 1
    return {"bytes": 4 * n + 8 * (M // 2 + 1), "flops": segments * 2.5 * M * math.log2(M)}


# ---------------------------------------------------------------------------
# results in 64 bits
# ---------------------------------------------------------------------------
def _moment_start(y, u):
    """Starting (c, g, A, B) of a dip or peak from the spectrum's moments."""
    T = u.numel()
    order = torch.argsort(u.abs(), descending=True)
    B = y[:, order[:max(4, T // 5)]].median(dim=1).values
    d = y - B[:, None]
    sign = torch.sign(d.gather(1, d.abs().argmax(dim=1, keepdim=True)))
    w = (sign * d).clamp_min(0.0)
    A = sign[:, 0] * w.max(dim=1).values
    g = (w.sum(dim=1) / (math.pi * A.abs())).clamp(0.5, 0.5 * (T - 1))
    return torch.stack([(w * u).sum(dim=1) / w.sum(dim=1), g, A, B], dim=1)


def _lorentz(u, p):
    c, g, A, B = (v[:, None] for v in p.unbind(1))
    d = u[None, :] - c
    q = 1.0 / (d * d + g * g)
    L = g * g * q
    return B + A * L, torch.stack([2.0 * A * d * L * q, 2.0 * A * g * q * (1.0 - L), L, torch.ones_like(L)], dim=2)


def _least_squares(y, u, p, model, lo=None, hi=None, steps=40):
    """Levenberg-Marquardt on every row of y at once, run to the optimum;
    lo and hi: bounds of the parameters (a bound whose gradient points outward
    holds its parameter)."""
    m, J = model(u, p)
    r = y - m
    chi = (r * r).sum(dim=1)
    lam = torch.full_like(chi, 1e-3)
    eye = torch.eye(p.shape[1], dtype=p.dtype, device=p.device)
    for _ in range(steps):
        H = J.transpose(1, 2) @ J
        b = (J.transpose(1, 2) @ r[:, :, None])[:, :, 0]
        if lo is not None:
            held = ((p <= lo) & (b < 0)) | ((p >= hi) & (b > 0))
            free = (~held).to(p.dtype)
            H = H * free[:, :, None] * free[:, None, :] + torch.diag_embed(held.to(p.dtype))
            b = b * free
        s = torch.rsqrt(torch.diagonal(H, dim1=1, dim2=2).clamp_min(1e-300))
        Hs = H * s[:, :, None] * s[:, None, :] + lam[:, None, None] * eye
        step = s * torch.linalg.solve(Hs, (s * b)[:, :, None])[:, :, 0]
        trial = p + step
        if lo is not None:
            trial = torch.minimum(torch.maximum(trial, lo), hi)
        mt, Jt = model(u, trial)
        rt = y - mt
        ct = (rt * rt).sum(dim=1)
        good = ct <= chi
        p = torch.where(good[:, None], trial, p)
        r = torch.where(good[:, None], rt, r)
        J = torch.where(good[:, None, None], Jt, J)
        chi = torch.where(good, ct, chi)
        lam = torch.where(good, lam * 0.1, lam * 10.0).clamp(1e-12, 1e12)
    return p, chi


def _fit64(y, x, fano):
    """Optimum (c, g, A, B) and chi^2 of every row, abscissa units."""
    x = torch.as_tensor(x, dtype=torch.float64, device=y.device)
    mid, scale = 0.5 * (x.min() + x.max()), (x.max() - x.min()) / (x.numel() - 1)
    u = (x - mid) / scale
    params = torch.empty((y.shape[0], 4), dtype=torch.float64, device=y.device)
    rss = torch.empty(y.shape[0], dtype=torch.float64, device=y.device)
    width = FWHM / 2.0 / scale

    def fano_model(u, p):
        c, A, B = (v[:, None] for v in p.unbind(1))
        e = (u[None, :] - c) / width
        F = (FANO_Q + e) ** 2 / (1.0 + e * e)
        dF = 2.0 * (FANO_Q + e) * (1.0 - FANO_Q * e) / (1.0 + e * e) ** 2
        return B + A * F, torch.stack([-A * dF / width, F, torch.ones_like(F)], dim=2)

    for s in range(0, y.shape[0], 100_000):
        rows = y[s:s + 100_000].double()
        if fano:
            c0 = u[rows.argmin(dim=1)] + FANO_Q * width
            p0 = torch.stack([c0, torch.full_like(c0, DEPTH), torch.full_like(c0, 1.0 - DEPTH)], dim=1)
            big = 1e30
            lo = torch.tensor([-big, 0.9 * DEPTH, 0.9 * (1.0 - DEPTH)], dtype=torch.float64, device=y.device)
            hi = torch.tensor([big, 1.1 * DEPTH, 1.1 * (1.0 - DEPTH)], dtype=torch.float64, device=y.device)
            p, chi = _least_squares(rows, u, p0, fano_model, lo, hi)
            p = torch.stack([p[:, 0], torch.ones_like(c0) * width, p[:, 1], p[:, 2]], dim=1)
        else:
            p, chi = _least_squares(rows, u, _moment_start(rows, u), _lorentz)
        params[s:s + 100_000] = torch.stack([mid + scale * p[:, 0], scale * p[:, 1].abs(), p[:, 2], p[:, 3]], dim=1)
        rss[s:s + 100_000] = chi
    return params, rss


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _layers(theta, n_in):
    sizes = [HIDDEN * n_in, HIDDEN, HIDDEN * HIDDEN, HIDDEN, 4 * HIDDEN, 4]
    W1, b1, W2, b2, W3, b3 = torch.split(theta, sizes)
    return W1.view(HIDDEN, n_in), b1, W2.view(HIDDEN, HIDDEN), b2, W3.view(4, HIDDEN), b3


def _forward(theta, x):
    W1, b1, W2, b2, W3, b3 = _layers(theta, x.shape[1])
    return _gelu(_gelu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def _train64(case, seed):
    x, t, perm = _training_set(case, seed)
    x, t, perm = x.double(), t.double(), perm.long()
    theta = torch.tensor(_first_weights(case, seed).astype(np.float64), device=x.device, requires_grad=True)
    m1, m2 = torch.zeros_like(theta), torch.zeros_like(theta)
    losses = []
    for k, s in enumerate(range(0, case["n"], case["batch"]), start=1):
        rows = perm[s:s + case["batch"]]
        loss = ((_forward(theta, x[rows]) - t[rows]) ** 2).mean()
        (g,) = torch.autograd.grad(loss, theta)
        losses.append(loss.detach())
        with torch.no_grad():
            m1 = 0.9 * m1 + 0.1 * g
            m2 = 0.999 * m2 + 0.001 * g * g
            theta -= 1e-3 * (m1 / (1.0 - 0.9 ** k)) / (torch.sqrt(m2 / (1.0 - 0.999 ** k)) + 1e-8)
    return {"losses": torch.stack(losses), "params": theta.detach()}


def _welch64(x, n, stride, M, fs):
    x = x.view(n, stride)[:, 0]
    window = 0.5 - 0.5 * torch.cos(2.0 * math.pi * torch.arange(M, device=x.device, dtype=torch.float64) / M)
    segments = (n - M) // (M // 2) + 1
    total = torch.zeros(M // 2 + 1, dtype=torch.float64, device=x.device)
    step = max(1, (1 << 26) // M)
    for s in range(0, segments, step):
        k = min(step, segments - s)
        block = x[s * (M // 2):(s + k - 1) * (M // 2) + M].unfold(0, M, M // 2).double()
        block = (block - block.mean(dim=1, keepdim=True)) * window
        z = torch.fft.rfft(block, dim=1)
        total += (z.real ** 2 + z.imag ** 2).sum(dim=0)
    total *= 2.0 / (segments * fs * (window * window).sum())
    total[0] *= 0.5
    total[-1] *= 0.5
    return total, segments


def _resonance64(S, df, f_lo, f_hi):
    """(f0, Q, A, B, their standard errors, chi^2, steps, status, bins) of the
    driven oscillator over a floor, fitted to ln S by Levenberg-Marquardt."""
    k = np.arange(max(1, math.ceil(f_lo / df)), min(S.size - 1, math.floor(f_hi / df)) + 1)
    f, logS, S = k * df, np.log(S[k]), S[k]
    kp, B = int(np.argmax(S)), float(S.min())
    half = B + 0.5 * (S[kp] - B)
    lo = hi = kp
    while lo > 0 and S[lo - 1] > half:
        lo -= 1
    while hi < S.size - 1 and S[hi + 1] > half:
        hi += 1
    fl = f[lo] if lo == 0 else f[lo - 1] + (half - S[lo - 1]) / (S[lo] - S[lo - 1]) * df
    fh = f[hi] if hi == S.size - 1 else f[hi] + (S[hi] - half) / (S[hi] - S[hi + 1]) * df
    Q = f[kp] / max(fh - fl, df)
    p = np.array([f[kp], Q, (S[kp] - B) / (Q * Q), B])

    def at(p):
        f0, Q, A, B = p
        a = f0 * f0 - f * f
        c = f * f0 / Q
        D = a * a + c * c
        m = A * f0 ** 4 / D + B
        if not np.all(m > 0.0) or not np.all(np.isfinite(m)):
            return None
        dD = 4.0 * f0 * a + 2.0 * f * f * f0 / (Q * Q)
        J = np.stack([A * (4.0 * f0 ** 3 / D - f0 ** 4 * dD / (D * D)), 2.0 * A * f0 ** 4 * c * c / (Q * D * D),
                      f0 ** 4 / D, np.ones_like(f)], axis=1) / m[:, None]
        return J, logS - np.log(m)

    J, r = at(p)
    chi, lam, steps, status = float(r @ r), 1e-3, 0, 1
    while steps < 200:
        steps += 1
        H = J.T @ J
        s = 1.0 / np.sqrt(np.diag(H))
        step = s * np.linalg.solve(H * np.outer(s, s) + lam * np.eye(4), s * (J.T @ r))
        new = at(p + step)
        c2 = math.inf if new is None else float(new[1] @ new[1])
        if math.isfinite(c2) and abs(c2 - chi) <= 1e-12 * chi:
            if c2 <= chi:
                p, chi, (J, r) = p + step, c2, new
            status = 0
            break
        if c2 < chi:
            p, chi, (J, r) = p + step, c2, new
            lam *= 0.1
        else:
            lam *= 10.0
    H = J.T @ J
    s = 1.0 / np.sqrt(np.diag(H))
    errors = s * np.sqrt(np.diag(np.linalg.inv(H * np.outer(s, s))) * chi / (f.size - 4))
    return np.concatenate([p, errors, [chi, steps, status, f.size]])


def exact(case, seed):
    kind = case["kind"]
    if kind == "process":
        name = case["instrument"]
        frames = _comb_frames(name, case["n"], seed, cavity=True)
        ref = _comb_reference(name, seed)
        amps = _magnitudes(frames, _comb_bins(name))
        del frames
        y = amps / torch.tensor(ref, device=amps.device)
        params, rss = _fit64(y, _abscissa(name), fano=name == "paper8")
        return {"amps": amps, "y": y, "params": params, "rss": rss, "iters": None, "status": None}
    if kind == "readout":
        frames, bins, _, ref = _arbitrary(case, seed)
        amps = _magnitudes(frames, bins)
        return amps, amps / torch.tensor(ref, device=amps.device)
    if kind == "fit":
        y, _ = _spectra(case["instrument"], case["n"], seed, 20e6)
        params, rss = _fit64(y, _abscissa(case["instrument"]), fano=False)
        return {"y": None, "params": params, "rss": rss, "iters": None, "status": None}
    if kind == "guess":
        name = case["instrument"]
        x = _abscissa(name)
        y, _ = _spectra(name, case["n"], seed, 0.1 * float(np.ptp(x)) / 2.0)
        _, *arrays = _net_arrays(_net_blob(name, seed))
        in_mean, in_scale, out_mean, out_scale, theta = (torch.tensor(a, device=y.device) for a in arrays)
        out = torch.empty((case["n"], 4), dtype=torch.float64, device=y.device)
        for s in range(0, case["n"], 100_000):
            rows = (y[s:s + 100_000].double() - in_mean) * in_scale
            out[s:s + 100_000] = _forward(theta, rows) * out_scale + out_mean
        dx = float(np.ptp(x)) / (x.size - 1)
        out[:, 1] = out[:, 1].abs().clamp(0.5 * dx, 0.5 * float(np.ptp(x)))
        return out
    if kind == "train":
        return _train64(case, seed)
    x = _centres(case, seed)
    M = case["segment"]
    density, segments = _welch64(x, case["n"], case["stride"], M, 1e6)
    return density, segments, _resonance64(density.cpu().numpy(), 1e6 / M, 18e3, 30e3)
