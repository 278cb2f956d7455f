"""Workloads of the correlator, through its public binding.

A case is one of four kinds:

  scan    one handle correlates a whole (short) scan, integration after
          integration.  ``path`` says where the samples live and the results
          go: "device" (attached device memory, results on the device), "host"
          (pinned host memory read over the host link, results copied to the
          host) or "push" (each pass resets the handle, pushes the recording
          from pinned host memory and copies the results to the host).
  batch   several scans of uneven shape, one integration each, as one graph.
  fringe  the delay-rate search of one baseline.

Samples are independent 2-bit codes with the code probabilities of a unit
Gaussian quantised at +-0.98 sigma, which is what noise-dominated recordings
hold.  Delays follow a spacecraft (station 0: 0.3..1.2 s, up to 3e-5 s/s) and
ground stations (a daily sinusoid of up to 20 ms), as quintic segments with a
boundary inside the scan.
"""
import math
import random

import numpy as np
import torch

from paper_1502_06894_gb300 import corr

DEV = "cuda:0"
LEVELS = (-3.336, -1.0, 1.0, 3.336)
PAYLOAD = 10000  # Mark5B payload bytes per frame
HEADER = 16
SYNC = 0xABADDEED


def _scan(name, stations, subbands, pols, nchan, samples, integrations=1, fs=32e6, precision=0, pre=False, cross=False,
          framed=False, path="device"):
    return {"name": name, "kind": "scan", "stations": stations, "subbands": subbands, "pols": pols, "nchan": nchan,
            "samples": samples, "integrations": integrations, "fs": fs, "precision": precision, "pre": pre,
            "cross": cross, "framed": framed, "path": path}


def listed():
    return [
        # the smallest calls: a few milliseconds of three stations, what a
        # setup check or a real-time monitor correlates; launches count
        _scan("check-3st", 3, 2, 2, 256, 128000, integrations=2),
        # first fringes: the spacecraft and one ground station, one subband,
        # 256 channels, one integration of 1 s
        _scan("pair-1s", 2, 1, 1, 256, 32000000),
        # the production scan: 10 stations, 8 subbands x 2 polarisations,
        # 1024 channels, 1 s integrations, in FP32
        _scan("ten-fp32", 10, 8, 2, 1024, 32000000, integrations=2),
        # the same with FP16 spectra
        _scan("ten-fp16", 10, 8, 2, 1024, 32000000, integrations=2, precision=1),
        # the production scan at a spacecraft's delay rate (fringe rotation
        # before the transform), end to end: samples in pinned host memory,
        # visibilities copied back
        _scan("ten-pre-host", 10, 8, 2, 1024, 16000000, pre=True, path="host"),
        # polarisation science: all four hand products of the production scan
        _scan("ten-cross", 10, 8, 2, 1024, 16000000, cross=True),
        # a large array: 64 stations, 16 subbands x 2 polarisations at
        # 64 Msample/s, 4096 channels, a 0.125 s integration (976.6 blocks)
        _scan("array-fp32", 64, 16, 2, 4096, 8000000, fs=64e6),
        # the same in E4M3 on the tensor cores
        _scan("array-e4m3", 64, 16, 2, 4096, 8000000, fs=64e6, precision=2),
        # an odd mid-size network on the tensor cores: 17 stations, 7 subbands
        # of one polarisation, 2048 channels, a ragged integration
        _scan("odd-fp16", 17, 7, 1, 2048, 9000001, precision=1),
        # Mark5B-framed recordings of five stations pushed from host memory,
        # a few frames lost, results on the host
        _scan("mark5b-push", 5, 4, 2, 512, 8000000, framed=True, path="push"),
        # a correlator centre's queue: uneven scans in one graph
        {"name": "batch-6", "kind": "batch", "scans": 6, "mix": 4, "samples": 3200000, "precision": 1},
        # the wide-window fringe search of one baseline
        {"name": "fringe-512x8192", "kind": "fringe", "sub": 256, "nchan": 1024, "pad_rate": 512, "pad_delay": 8192},
    ]


def draw(rng):
    r = rng.random()
    if r < 0.15:
        ls, lc = rng.randint(4, 9), rng.randint(7, 13)
        sub = rng.randint((1 << ls) // 2 + 1, 1 << ls)
        return {"kind": "fringe", "sub": sub, "nchan": 1 << lc, "pad_rate": 1 << (ls + rng.randint(0, 1)),
                "pad_delay": 1 << min(14, lc + rng.randint(0, 3))}
    if r < 0.25:
        return {"kind": "batch", "scans": rng.randint(2, 8), "mix": rng.randint(5, 1 << 20),
                "samples": int(math.exp(rng.uniform(math.log(200000), math.log(3200000)))), "precision": rng.choice((0, 1, 2))}
    path = "push" if r < 0.35 else rng.choice(("device", "device", "device", "host"))
    while True:
        stations = int(round(math.exp(rng.uniform(math.log(2), math.log(64)))))
        subbands, pols = rng.randint(1, 16), rng.randint(1, 2)
        nchan = 1 << rng.randint(7, 13)
        fs = rng.choice((32e6, 32e6, 64e6))
        precision = rng.choice((0, 0, 1, 2))
        cross = pols == 2 and stations <= 32 and rng.random() < 0.25
        pre = nchan <= 4096 and rng.random() < 0.25
        integrations = rng.randint(1, 3)
        rows = stations * (2 if cross else 1)
        # station-samples of the pass, weighted by the cross products' share
        most = 2.5e10 / (1 + rows / 20) / (2 if pre else 1) / (1 if path == "device" else 4)
        total = math.exp(rng.uniform(math.log(2e7), math.log(most)))
        samples = int(total / (stations * subbands * pols * integrations))
        if 16 * nchan <= samples <= 64000000:
            break
    case = _scan("", stations, subbands, pols, nchan, samples, integrations, fs, precision, pre, cross,
                 path == "push" and rng.random() < 0.5, path)
    del case["name"]
    return case


# ---------------------------------------------------------------- inputs


def _delays(case, rng):
    """Per station two quintic segments (t0, coeffs) around the scan's middle."""
    dur = case["samples"] * case["integrations"] / case["fs"]
    t0s = (0.5 * dur - 120.0, 0.5 * dur)
    out = []
    for s in range(case["stations"]):
        segs = []
        if s == 0:
            tau0, rate = rng.uniform(0.3, 1.2), rng.uniform(-3e-5, 3e-5)
            acc, jerk = rng.uniform(-1, 1) * 1e-9, rng.uniform(-1, 1) * 1e-12
            for t in t0s:
                d = (tau0 + rate * t + acc * t ** 2 / 2 + jerk * t ** 3 / 6, rate + acc * t + jerk * t ** 2 / 2,
                     acc + jerk * t, jerk, 0.0, 0.0)
                segs.append((t, [x / math.factorial(i) for i, x in enumerate(d)]))
        else:
            amp, w, p = rng.uniform(-20e-3, 20e-3), 7.29e-5, rng.uniform(0, 2 * math.pi)
            for t in t0s:
                segs.append((t, [amp * w ** i * math.sin(w * t + p + i * math.pi / 2) / math.factorial(i)
                                 for i in range(6)]))
        out.append(segs)
    return out


def _tau(segs, t):
    """tau(t) of the segments in FP64, Horner's rule with one rounding a step
    (the long double holds the products exactly)."""
    t = np.asarray(t, np.float64)
    out = np.empty_like(t)
    rate = np.empty_like(t)
    for q, (t0, c) in enumerate(segs):
        m = (t >= t0) if q + 1 == len(segs) else (t >= t0) & (t < segs[q + 1][0])
        u = (t[m] - t0).astype(np.longdouble)
        v = np.full(u.shape, c[5])
        for k in range(4, -1, -1):
            v = (v.astype(np.longdouble) * u + np.longdouble(c[k])).astype(np.float64)
        d = np.zeros(u.shape)
        for k in range(5, 0, -1):
            d = (d.astype(np.longdouble) * u + np.longdouble(k * c[k])).astype(np.float64)
        out[m], rate[m] = v, d
    return out, rate


def _codes(nbytes, seed):
    """Packed bytes of quantised-Gaussian 2-bit codes (code 0..3 with
    probabilities 0.164, 0.336, 0.336, 0.164), made on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(seed & 0x7FFFFFFF)
    words = torch.empty((nbytes + 3) // 4, dtype=torch.int32, device=DEV)
    step = 1 << 25
    for o in range(0, words.numel(), step):
        n = min(step, words.numel() - o)

        def bits():
            return torch.randint(-2 ** 31, 2 ** 31, (n,), generator=g, device=DEV, dtype=torch.int32)

        high = bits()                       # each bit set with probability 21/64 = 0.328
        for k in range(5):
            high = high & bits() if k % 2 == 0 else high | bits()
        sign = bits()
        low = ~((sign >> 1) ^ high)
        words[o:o + n] = (sign & -1431655766) | (low & 1431655765)
    return words.view(torch.uint8)[:nbytes]


def _plan(case, seed):
    """Delay segments, sky frequencies and each station's window of samples."""
    rng = random.Random(seed * 1000003 + 17)
    delays = _delays(case, rng)
    span = case["samples"] * case["integrations"]
    n = 2 * case["nchan"]
    grid = np.linspace(0.0, span / case["fs"], 129)
    start, count = [], []
    for segs in delays:
        tau = _tau(segs, grid)[0]
        lo = (int(math.floor(tau.min() * case["fs"])) - 64) // 16 * 16
        hi = span + int(math.ceil(tau.max() * case["fs"])) + n + 64
        start.append(lo)
        count.append((hi - lo + 15) // 16 * 16)
    nu0 = [4.8e9 + 16e6 * sb for sb in range(case["subbands"])]
    return delays, nu0, start, count


def _lost(case, seed, station, frames):
    """Frames of a station that carry no sync word."""
    rng = random.Random(seed * 7919 + station)
    return sorted(rng.sample(range(frames), min(frames, 1 + frames // 4000)))


def _frames(payload, lost):
    """Mark5B-style frames (a 16-byte header and PAYLOAD bytes) of a stream."""
    nf = -(-payload.numel() // PAYLOAD)
    out = torch.zeros((nf, HEADER + PAYLOAD), dtype=torch.uint8, device=payload.device)
    body = torch.zeros(nf * PAYLOAD, dtype=torch.uint8, device=payload.device)
    body[:payload.numel()] = payload
    out[:, HEADER:] = body.view(nf, PAYLOAD)
    head = np.zeros((nf, 4), np.uint32)
    head[:, 0] = SYNC
    head[:, 1] = np.arange(nf) & 0x7FFF
    head[lost, 0] = 0
    out[:, :HEADER] = torch.from_numpy(head.view(np.uint8)).to(payload.device)
    return out.view(-1)


def _station_bytes(case, count):
    return (count * case["subbands"] * case["pols"] // 4 + 15) // 16 * 16


class _Scan:
    """A configured correlator, its samples and its result buffers."""

    def __init__(self, case, seed):
        self.case = case
        delays, nu0, start, count = _plan(case, seed)
        c = corr.Correlator(case["stations"], case["subbands"], case["pols"], case["nchan"],
                            case["samples"] / case["fs"], fs=case["fs"])
        for sb, nu in enumerate(nu0):
            c.set_sky_freq(sb, nu)
        c.set_precision(case["precision"])
        if case["cross"]:
            c.set_pol_products(corr.CORR_POL_CROSS)
        if case["pre"]:
            c.set_fringe_rotation(corr.CORR_ROT_PRE_F)
        if case["framed"]:
            c.set_frame_format(PAYLOAD)
        self.data = []
        for s, segs in enumerate(delays):
            for t0, coeffs in segs:
                c.set_delay_poly(s, t0, coeffs)
            c.set_stream_start(s, start[s])
            x = _codes(_station_bytes(case, count[s]), seed * 131 + s)
            if case["framed"]:
                x = _frames(x, _lost(case, seed, s, -(-x.numel() // PAYLOAD)))
            if case["path"] != "device":
                host = torch.empty(x.numel(), dtype=torch.uint8, pin_memory=True)
                host.copy_(x)
                x = host
            self.data.append(x)
            if case["path"] == "device":
                c.attach_device(s, x)
            elif case["path"] == "host":
                c.attach_host(s, x)
            else:
                c.reserve(s, x.numel())
        products = 4 if case["cross"] else case["pols"]
        shape = (c.nbl, case["subbands"], products, case["nchan"])
        where = {"device": DEV} if case["path"] == "device" else {"pin_memory": True}
        self.vis = [torch.empty(shape, dtype=torch.complex64, **where) for _ in range(case["integrations"])]
        self.weights = [torch.empty(c.nbl, dtype=torch.float64, **where) for _ in range(case["integrations"])]
        self.c = c
        torch.cuda.synchronize()  # the correlator's streams are its own

    def __del__(self):
        c = getattr(self, "c", None)
        if c is not None:
            c.close()


def _mix(case):
    """The scans of a batch: uneven shapes, one integration of about `samples`
    samples of up to 4e9 station-samples each."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["scans"]):
        stations, subbands, pols = rng.randint(2, 20), rng.randint(1, 16), rng.randint(1, 2)
        nchan = 1 << rng.randint(7, 13)
        n = 2 * nchan
        blocks = max(4, int(case["samples"] * rng.uniform(0.25, 1.0)) // n)
        out.append(_scan("", stations, subbands, pols, nchan, blocks * n, precision=case["precision"]))
    return out


def prepare(case, seed):
    if case["kind"] == "scan":
        return _Scan(case, seed)
    if case["kind"] == "batch":
        scans = [_Scan(c, seed * 64 + q) for q, c in enumerate(_mix(case))]
        for s in scans:
            s.c.flush()
        return scans
    g = torch.Generator(device=DEV).manual_seed(seed & 0x7FFFFFFF)
    t, k = case["sub"], case["nchan"]
    rng = random.Random(seed)
    # a fringe at a residual delay and rate, in noise
    lag, rate = rng.uniform(-0.4, 0.4), rng.uniform(-0.4, 0.4)
    ph = 2 * math.pi * (lag * torch.arange(k, device=DEV, dtype=torch.float64)[None]
                        + rate * torch.arange(t, device=DEV, dtype=torch.float64)[:, None])
    noise = torch.randn((t, k, 2), generator=g, device=DEV)
    return {"case": case, "vis": (torch.view_as_complex(noise) + 0.5 * torch.polar(torch.ones_like(ph), ph)).to(torch.complex64)}


# ---------------------------------------------------------------- one pass


def run(state):
    if isinstance(state, _Scan):
        c, path = state.c, state.case["path"]
        if path == "push":
            c.reset()
            for s, x in enumerate(state.data):
                c.push_async(s, x)
        else:
            c.rewind()
        for v, w in zip(state.vis, state.weights):
            rc = c.correlate_device(v, w) if path == "device" else c.correlate_into(v, w)
            if rc != corr.CORR_OK:
                raise corr.CorrError(rc, corr.corr_last_error(c.h).decode())
        if path == "push":
            c.wait_pushes()
        return {"vis": state.vis, "weights": state.weights}
    if isinstance(state, list):
        for s in state:
            s.c.rewind()
        corr.batch_run([s.c for s in state], [s.vis[0] for s in state], [s.weights[0] for s in state])
        return {"vis": [s.vis[0] for s in state], "weights": [s.weights[0] for s in state]}
    case = state["case"]
    m, peak = corr.fringe_search(state["vis"], case["pad_rate"], case["pad_delay"])
    return {"map": m, "peak": [peak[0], peak[1], peak[2], peak[3].real, peak[3].imag]}


def _blocks(case):
    n = 2 * case["nchan"]
    return [(-(-i * case["samples"] // n), -(-(i + 1) * case["samples"] // n)) for i in range(case["integrations"])]


def work(case):
    if case["kind"] == "batch":
        parts = [work(c) for c in _mix(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if case["kind"] == "fringe":
        t, k, nr, nd = case["sub"], case["nchan"], case["pad_rate"], case["pad_delay"]
        return {"bytes": 8 * (t * k + nr * nd), "flops": 5 * nd * math.log2(nd) * t + 5 * nr * math.log2(nr) * nd + 3 * nr * nd}
    s, g, nch = case["stations"], case["subbands"] * case["pols"], case["nchan"]
    n, blocks = 2 * nch, _blocks(case)[-1][1]
    rows, streams = (2 * s, case["subbands"]) if case["cross"] else (s, g)
    out = s * (s + 1) // 2 * case["subbands"] * (4 if case["cross"] else case["pols"]) * nch * 8 * case["integrations"]
    # a real transform (with the rotation before it a complex one and a
    # rotated sample), the phase of every channel, and every product
    fft = (5 * n * math.log2(n) + 2 * n) if case["pre"] else 2.5 * n * math.log2(n)
    flops = blocks * (s * g * (fft + 6 * nch) + rows * (rows + 1) / 2 * streams * nch * 8)
    return {"bytes": s * blocks * n * g / 4 + out, "flops": flops}


# ---------------------------------------------------------------- the definition in 64 bits


def _exact_scan(case, seed):
    delays, nu0, start, count = _plan(case, seed)
    s, g, nch, fs = case["stations"], case["subbands"] * case["pols"], case["nchan"], case["fs"]
    n = 2 * nch
    data, levels = [], torch.tensor(np.array(LEVELS, np.float32).astype(np.float64), device=DEV)
    for q in range(s):
        data.append(_codes(_station_bytes(case, count[q]), seed * 131 + q))
    vis, weights = [], []
    k = torch.arange(nch, device=DEV, dtype=torch.float64)
    pairs = [(a, b) for a in range(s) for b in range(a, s)]
    ia = torch.tensor([a for a, _ in pairs], device=DEV)
    ib = torch.tensor([b for _, b in pairs], device=DEV)
    for b0, b1 in _blocks(case):
        nb = b1 - b0
        tc = (np.arange(b0, b1, dtype=np.float64) * n + n // 2) / fs
        first, ok, phi, step, slope = [], [], [], [], []
        for q in range(s):
            tau, rate = _tau(delays[q], tc)
            whole = np.floor((tau.astype(np.longdouble) * fs + 0.5).astype(np.float64))
            eps = tau - whole / fs
            rel = (np.arange(b0, b1, dtype=np.int64) * n + whole.astype(np.int64)) - start[q]
            bytes_ = _station_bytes(case, count[q])
            if case["framed"]:
                frames = -(-bytes_ // PAYLOAD)
                bad = np.zeros(frames, np.int64)
                bad[_lost(case, seed, q, frames)] = 1
                have = frames * PAYLOAD * 4 // g
                before = np.concatenate(([0], np.cumsum(bad)))
                fa = np.clip((2 * rel * g) // 8 // PAYLOAD, 0, frames)
                fb = np.clip((2 * (rel + n) * g - 1) // 8 // PAYLOAD + 1, 0, frames)
                good = (rel >= 0) & (rel + n <= have) & (before[fb] - before[fa] == 0)
            else:
                good = (rel >= 0) & (rel + n <= bytes_ * 4 // g)
            first.append(torch.from_numpy(rel).to(DEV))
            ok.append(torch.from_numpy(good).to(DEV))
            phi.append(torch.from_numpy(np.stack([nu * tau - np.floor(nu * tau) for nu in nu0])).to(DEV))
            step.append(torch.from_numpy(np.stack([nu * rate / fs for nu in nu0])).to(DEV))
            slope.append(torch.from_numpy(eps * fs / n).to(DEV))
        okf = torch.stack(ok).double()
        w = (okf @ okf.T)[ia, ib]
        products = 4 if case["cross"] else case["pols"]
        out = torch.zeros((len(pairs), case["subbands"], products, nch), dtype=torch.complex128, device=DEV)
        chunk = max(1, min(nb, (1 << 28) // (s * n * (2 if case["cross"] else 1))))

        def spectra(j, lo, hi):
            """[station, block, channel] of stream j, blocks b0 + lo .. b0 + hi."""
            sb = j // case["pols"]
            t = torch.arange(n, device=DEV)
            x = torch.empty((s, hi - lo, nch), dtype=torch.complex128, device=DEV)
            for q in range(s):
                bit = 2 * ((first[q][lo:hi, None] + t) * g + j)
                top = data[q].numel() - 1
                code = (data[q][(bit >> 3).clamp_(0, top)] >> (bit & 7).to(torch.uint8)) & 3
                v = levels[code.long()] * ok[q][lo:hi, None]
                ramp = slope[q][lo:hi, None] * k
                if case["pre"]:
                    ph = phi[q][sb, lo:hi, None] + step[q][sb, lo:hi, None] * (t - n // 2)
                    ph = 2 * math.pi * (ph - torch.floor(ph))
                    f = torch.fft.fft(v * torch.polar(torch.ones_like(ph), ph))[:, :nch]
                else:
                    f = torch.fft.rfft(v)[:, :nch]
                    ramp = ramp + phi[q][sb, lo:hi, None]
                x[q] = f * torch.polar(torch.ones_like(ramp), 2 * math.pi * (ramp - torch.floor(ramp)))
            return x

        def products_of(x, y):
            """sum over blocks of x_a conj(y_b) for a <= b."""
            if s <= 12:
                return torch.stack([(x[a] * y[b].conj()).sum(0) for a, b in pairs])
            return torch.matmul(x.permute(2, 0, 1), y.permute(2, 1, 0).conj())[:, ia, ib].T

        for sb in range(case["subbands"]):
            for lo in range(0, nb, chunk):
                hi = min(nb, lo + chunk)
                x = [spectra(sb * case["pols"] + p, lo, hi) for p in range(case["pols"])] if case["cross"] else None
                for pq in range(products):
                    if case["cross"]:
                        out[:, sb, pq] += products_of(x[pq >> 1], x[pq & 1])
                    else:
                        y = spectra(sb * case["pols"] + pq, lo, hi)
                        out[:, sb, pq] += products_of(y, y)
        vis.append(out / (w.clamp(min=1.0) * n)[:, None, None, None])
        weights.append(w)
    return {"vis": vis, "weights": weights}


def _exact_seconds(case):
    """About how long the 64-bit evaluation takes."""
    w = work(case)
    return w["flops"] * (2 if case["stations"] > 12 else 1) / 6e11 + case["integrations"] * case["stations"] * 0.1


def exact(case, seed):
    if case["kind"] == "fringe":
        v = prepare(case, seed)["vis"].to(torch.complex128)
        m = torch.fft.ifft2(v, s=(case["pad_rate"], case["pad_delay"])) * (case["pad_rate"] * case["pad_delay"])
        at = int(m.abs().argmax())
        p = complex(m.view(-1)[at])
        return {"map": m, "peak": [at // case["pad_delay"], at % case["pad_delay"], abs(p), p.real, p.imag]}
    if case["kind"] == "batch":
        if sum(_exact_seconds(c) for c in _mix(case)) > 20:
            return None
        parts = [_exact_scan(c, seed * 64 + q) for q, c in enumerate(_mix(case))]
        return {k: [p[k][0] for p in parts] for k in ("vis", "weights")}
    if _exact_seconds(case) > 20:
        return None
    return _exact_scan(case, seed)
