"""Timed cases of the QTAM transform pair: what a program that uses this library has it do.

Sizes are those of the benchmark's workloads and of the tests (the 4 s FP64 check, 8 s serving
requests, 64 s segments with Q {4..64} x 128 rows, the uneven 1-32 s batch, 6 s glitch segments,
2 s dense tiles, a stream through 64 s chunks).  `draw` gives the same kinds of work at other
durations, sample rates, plane and row counts, batches and storage types.

Inputs are whitened strain: unit white noise with sine-Gaussian glitches, and a chirp in every
other segment.  `exact` is the transform's definition in 64 bits with torch only.
"""
import math

import numpy as np
import torch

from paper_2603_29785_gb300 import batch as qbatch
from paper_2603_29785_gb300 import qtam

MAX_ROW = 7680           # longest envelope with a factor of 3 or 5 that a plan takes (8192 alone is longer)


def listed():
    full = dict(fs=4096.0, n=262144, qs="4,8,16,32,64", f_max=2048.0, rows=128)
    return [
        # smallest call: one 4 s segment in FP64, analysis and synthesis (validation against double precision)
        dict(name="pair_4s_f64", kind="pair", fs=4096.0, n=16384, qs="8", f_max=1024.0, rows=64, batch=1, compute="f64"),
        # one serving request: three channels of 8 s at one Q, some rows zeroed, and back to strain
        dict(name="request_8s", kind="request", fs=4096.0, n=32768, qs="16", f_max=2048.0, rows=128, batch=3),
        # low latency: a single 64 s segment through every plane and back
        dict(name="pair_64s_one", kind="pair", batch=1, **full),
        # glitch classification: 6 s segments, 62 rows per plane at the minimal length, and the best plane of each
        dict(name="scan_6s", kind="scan", fs=4096.0, n=24576, qs="4,8,16,32,64", f_max=2048.0, rows=62, batch=128,
             clamp_hz=111.3),
        # offline analysis of a batch of 64 s segments (the benchmark's batch) ...
        dict(name="forward_64s", kind="forward", batch=64, **full),
        # ... and its synthesis
        dict(name="inverse_64s", kind="inverse", batch=64, **full),
        # envelopes kept in 16 bits: one batch analysed, a stored one synthesised
        dict(name="stored_64s_bf16", kind="stored", batch=16, envelope="bf16", **full),
        # the same on the tensor-core short DFT, which a plan takes for 16-bit envelopes at M = 8192
        dict(name="stored_64s_tensor", kind="stored", batch=16, envelope="bf16", n_out=8192, short_dft="auto", **full),
        # composite bank: one window family per plane
        dict(name="bank_64s", kind="pair", batch=16, windows="bisquare,tukey,kaiser,hann,planck", **full),
        # undemodulated tiles over the whole spectrum, and the canonical inverse
        dict(name="dense_2s", kind="pair", fs=4096.0, n=8192, qs="4,8,16", f_max=2048.0, rows=64, batch=64, eps=1e-3,
             remodulate=True),
        # a continuous stream in overlapping 64 s chunks, from its first sample, and back
        dict(name="stream_64s", kind="stream", batch=16, **full),
        # segments of 1 to 32 s at two rates, forward and inverse as one CUDA graph
        dict(name="uneven_graph", kind="uneven", fs=4096.0, n=131072, qs="8,16,32", f_max=2048.0, rows=128, batch=96),
    ]


# ------------------------------------------------------------------ drawn cases
_SECONDS = (1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64)
_RATES = (1000.0, 2000.0, 2048.0, 4096.0, 8192.0, 16384.0)
_QS = (4, 5, 6, 8, 10, 11.3, 16, 20, 24, 32, 45, 64)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["pair", "pair", "forward", "inverse", "request", "scan", "stored", "bank", "dense", "stream",
                           "uneven", "f64"])
        fs = rng.choice(_RATES)
        n = int(fs * rng.choice(_SECONDS))
        f_max = 2048.0 if fs >= 4096 else math.floor(0.49 * fs)
        k = rng.randint(1, 5)
        c = dict(kind=kind, fs=fs, n=n, qs=",".join("%g" % q for q in sorted(rng.sample(_QS, k))), f_max=f_max,
                 rows=rng.choice([40, 48, 62, 64, 96, 100, 128, 150]), batch=1)
        if kind == "bank":
            c["kind"] = "pair"
            c["windows"] = ",".join(rng.choice(["bisquare", "tukey", "kaiser", "hann", "planck"]) for _ in range(k))
        elif kind == "dense":
            c.update(kind="pair", eps=1e-3, remodulate=rng.random() < 0.7)
        elif kind == "f64":
            c.update(kind="pair", compute="f64")
        elif kind == "stored":
            c["envelope"] = rng.choice(["bf16", "f16"])
        elif kind == "request":
            c["qs"] = "%g" % rng.choice(_QS)
        elif kind == "scan" and rng.random() < 0.5:
            c["clamp_hz"] = round(rng.uniform(40, 120), 1)
        if kind == "uneven":
            # lengths are doubled up to this case's: at least 1 s, at most 32 s, at two rates
            c.update(fs=4096.0, n=rng.choice([8, 16, 32]) * 4096, f_max=2048.0, batch=rng.randint(8, 64))
            return c
        try:
            g = _geometry(c)
        except ValueError:
            continue
        if g.M > MAX_ROW and g.M != 8192 or n > (1 << 20):
            continue
        if kind == "stream":
            q = n // math.gcd(n, g.M)
            if q * 8 > n:                   # chunk edges fall on whole columns: too coarse a grid leaves no guard
                continue
        size = 8 * len(g.kc) * g.M * (2 if kind == "f64" else 1)
        most = (1 << {"forward": 30, "inverse": 30, "scan": 29, "dense": 28, "f64": 26}.get(kind, 29)) // size
        if most < 1:
            continue
        c["batch"] = min(_log_int(rng, 1, min(most, 512)), 32 if kind == "stream" else 512)
        return c


# ------------------------------------------------------------------ the definition, in 64 bits
class _Geometry:
    pass


def _smooth(m):
    while True:
        r = m
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            return m
        m += 1


def _params(case):
    names = case["windows"].split(",") if case.get("windows") else ["bisquare"] * len(case["qs"].split(","))
    return [(w, {"tukey": 0.5, "kaiser": 8.0, "planck": 0.3}.get(w, 0.0)) for w in names]


def _window(name, prm, h):
    """W'(0..h) of one window family, FP64."""
    u = torch.arange(h + 1, dtype=torch.float64) / h
    if name == "bisquare":
        return (1 - u * u) ** 2
    if name == "hann":
        return 0.5 * (1 + torch.cos(math.pi * u))
    if name == "kaiser":
        return torch.i0(prm * torch.sqrt((1 - u * u).clamp(min=0))) / torch.i0(torch.tensor(prm, dtype=torch.float64))
    if name == "tukey":
        return torch.where(u <= 1 - prm, torch.ones_like(u), 0.5 * (1 + torch.cos(math.pi * (u - (1 - prm)) / prm)))
    t = 1 - u
    inner = (t > 0) & (t < prm)
    ts = torch.where(inner, t, torch.full_like(t, prm / 2))
    w = 1 / (torch.exp((prm / ts - prm / (prm - ts)).clamp(-700, 700)) + 1)
    return torch.where(t >= prm, torch.ones_like(t), torch.where(inner, w, torch.zeros_like(t)))


def _geometry(case):
    """Rows, widths and the envelope length of a case (host)."""
    g = _Geometry()
    g.fs, g.N, g.K = case["fs"], case["n"], case["rows"]
    g.qs = [float(q) for q in case["qs"].split(",")]
    T, f0, f1 = g.N / g.fs, 20.0, case["f_max"]
    f = [f0 * math.pow(f1 / f0, k / (g.K - 1)) for k in range(g.K)]
    gap = case.get("clamp_hz", 0.0) or max(b - a for a, b in zip(f, f[1:]))
    h_max = math.ceil(T * gap) // 2
    g.kc = [int(math.floor(v * T + 0.5)) for _ in g.qs for v in f]
    g.h = [max(1, min(int(math.floor(v * T * math.sqrt(11.0) / q)), h_max)) for q in g.qs for v in f]
    L = 2 * max(g.h) + 1
    if case.get("eps"):
        L = max(L, g.N // 2 + 1)
    g.M = case.get("n_out") or _smooth(L)
    g.eps, g.remod = case.get("eps", 0.0), case.get("remodulate", False)
    if max(g.kc) > g.N // 2 + 1 or g.M < L:
        raise ValueError("no such case")
    return g


class _Bank:
    """Index and weight tables of one plane's rows, on the device: bin[k, i] and w[k, i] of envelope position i."""

    def __init__(self, case, dtype=torch.float64):
        g = self.g = _geometry(case)
        dev = "cuda"
        M, half = g.M, g.N // 2
        self.bins, self.w, self.kc = [], [], []
        self.P = torch.zeros(half + 1, dtype=torch.float64, device=dev)
        i = torch.arange(M, device=dev)
        for p, (name, prm) in enumerate(_params(case)):
            tabs, offs, c = [], [], []
            at, seen = 0, {}
            hs = g.h[p * g.K:(p + 1) * g.K]
            for h in hs:
                if h not in seen:
                    t = _window(name, prm, h)
                    seen[h] = (at, float(1 / torch.sqrt(2 * (t * t).sum() - t[0] * t[0])))
                    tabs.append(t)
                    at += h + 1
                offs.append(seen[h][0])
                c.append(seen[h][1])
            tab = torch.cat(tabs).to(dev)
            h = torch.tensor(hs, device=dev)[:, None]
            kc = torch.tensor(g.kc[p * g.K:(p + 1) * g.K], device=dev)[:, None]
            c = torch.tensor(c, dtype=torch.float64, device=dev)[:, None]
            off = torch.tensor(offs, device=dev)[:, None]
            if g.eps:      # every bin of the one-sided spectrum has its place
                f = (i[None] + kc) % M
                d = f - kc
                inside = f <= half
                f = f.clamp(max=half)
            else:
                d = torch.where(i[None] <= h, i[None], i[None] - M)
                f = kc + d
                inside = (d.abs() <= h) & (f >= 0) & (f <= half)
                f = f.clamp(0, half)
            w = tab[off + d.abs().clamp(max=h)]
            w = torch.where(d.abs() > h, torch.zeros_like(w), w)
            if g.eps:
                w = torch.where(w > 0, w, torch.full_like(w, g.eps))
            w = torch.where(inside, c * w, torch.zeros_like(w))
            self.P.index_add_(0, f.reshape(-1), (w * w).reshape(-1))
            self.bins.append(f)
            self.w.append(w.to(dtype))
            self.kc.append(kc)
        self.n = torch.arange(M, device=dev)

    def carrier(self, p):
        t = (self.kc[p] * self.n) % self.g.M
        a = t.to(torch.float64) * (2 * math.pi / self.g.M)
        return torch.polar(torch.ones_like(a), a)

    def forward(self, x):
        """[P, K, M] envelopes of one segment, in the precision of `x`."""
        g = self.g
        X = torch.fft.rfft(x)
        out = torch.empty((len(g.qs), g.K, g.M), dtype=X.dtype, device=x.device)
        for p in range(len(g.qs)):
            y = torch.fft.ifft(X[self.bins[p]] * self.w[p], norm="forward")
            if g.remod:
                y = y * self.carrier(p)
            out[p] = y / math.sqrt(g.M * g.N)
        return out

    def inverse(self, y, tau):
        g = self.g
        half = g.N // 2
        A = torch.zeros((half + 1, 2), dtype=torch.float64, device=y.device)
        for p in range(len(g.qs)):
            v = y[p] * self.carrier(p).conj() if g.remod else y[p]
            v = torch.fft.fft(v) * (math.sqrt(g.N / g.M) * self.w[p])
            A.index_add_(0, self.bins[p].reshape(-1), torch.view_as_real(v).reshape(-1, 2))
        keep = (self.P > 0) & (self.P >= tau * self.P.max())
        X = torch.view_as_complex(A) * torch.where(keep, 1 / self.P, torch.zeros_like(self.P))
        X.imag[0] = 0
        X.imag[half] = 0
        return torch.fft.irfft(X, n=g.N)


# ------------------------------------------------------------------ inputs
def _generator(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * salt + seed)


def _strain(batch, n, fs, seed, dtype=torch.float32, salt=0):
    """[batch, n] whitened strain: white noise, two glitches a segment, a chirp in every other one."""
    gen = _generator(seed, salt)
    x = torch.randn((batch, n), generator=gen, device="cuda", dtype=torch.float32)
    t = torch.arange(n, device="cuda", dtype=torch.float32) / fs
    T = n / fs
    u = torch.rand((batch, 8), generator=gen, device="cuda")
    for k in range(2):
        f0 = 30.0 * (min(1500.0, 0.45 * fs) / 30.0) ** u[:, 4 * k, None]
        q = 4.0 + 36.0 * u[:, 4 * k + 1, None]
        tau = q / (math.sqrt(2.0) * math.pi * f0)
        d = t[None] - T * u[:, 4 * k + 2, None]
        amp = (8.0 + 42.0 * u[:, 4 * k + 3, None]) / torch.sqrt(0.63 * tau * fs)
        x += amp * torch.exp(-(d / tau) ** 2) * torch.sin(2 * math.pi * f0 * d)
    left = (0.9 * T - t).clamp(min=1e-3) / (0.9 * T)
    sweep = torch.sin(2 * math.pi * 32.0 * T * left ** 0.625) * left ** -0.25 * (t < 0.9 * T)
    x[::2] += 20.0 / math.sqrt(float((sweep ** 2).sum()) + 1e-30) * sweep
    return x.to(dtype)


def _envelopes(case, batch, seed, salt):
    """Stored envelopes of `batch` segments, made by the definition in 32 bits."""
    bank = _Bank(case, torch.float32)
    x = _strain(batch, case["n"], case["fs"], seed, salt=salt)
    y = torch.stack([bank.forward(v) for v in x])
    if case.get("envelope") in ("bf16", "f16"):
        y = torch.view_as_real(y).to(torch.bfloat16 if case["envelope"] == "bf16" else torch.float16)
    return y


def _plan(case):
    g = _geometry(case)
    par = _params(case)
    kw = dict(max_window_hz=case.get("clamp_hz", 0.0), n_out=case.get("n_out", 0), compute=case.get("compute", "f32"),
              envelope=case.get("envelope"), short_dft=case.get("short_dft", "cuda"), stopband_eps=g.eps,
              remodulate=bool(g.remod))
    if case.get("windows"):
        kw.update(window=tuple(p[0] for p in par), window_param=tuple(p[1] for p in par))
    return qtam.Plan(g.fs, g.N, tuple(g.qs), 20.0, case["f_max"], g.K, device=0, **kw)


def _gain(case, seed):
    """Row gains of a masked synthesis: about a fifth of the rows zeroed."""
    P = len(case["qs"].split(","))
    r = torch.rand((case["batch"], P, case["rows"]), generator=_generator(seed, 7), device="cuda")
    return (r > 0.2).to(torch.float32)


def _uneven(case, seed):
    """Segments of 1, 2, 4 ... s up to the case's length, half of them at four times its rate."""
    top = case["n"] // int(case["fs"])
    secs = [1 << k for k in range(top.bit_length())]
    host = np.random.Generator(np.random.PCG64(12345))       # the mix of lengths is the case's, not the seed's
    segs, rates = [], []
    for i in range(case["batch"]):
        fs = case["fs"] * (4 if i % 2 else 1)
        segs.append((int(secs[int(host.integers(len(secs)))] * fs), fs))
        rates.append(fs)
    out = [None] * len(segs)
    for key in sorted(set(segs)):
        idx = [i for i, s in enumerate(segs) if s == key]
        x = _strain(len(idx), key[0], key[1], seed, salt=key[0] % 99991)
        for j, i in enumerate(idx):
            out[i] = x[j].cpu().numpy()
    return out, rates


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        segs, rates = _uneven(case, seed)
        cache = qbatch.PlanCache([float(q) for q in case["qs"].split(",")], 20.0, case["f_max"], case["rows"], device=0)
        ub = qbatch.UnevenBatch(segs, rates, cache, tune=False)
        ub.capture()
        return dict(case=case, ub=ub)
    s = dict(case=case, plan=_plan(case))
    if kind == "stream":
        s["stream"] = qtam.Stream(s["plan"], max_chunks=case["batch"])
        s["x"] = _strain(1, s["stream"].hop * case["batch"], case["fs"], seed)[0]
        return s
    if kind != "inverse":
        s["x"] = _strain(case["batch"], case["n"], case["fs"], seed,
                         torch.float64 if case.get("compute") == "f64" else torch.float32)
    if kind in ("inverse", "stored"):
        s["y"] = _envelopes(case, case["batch"], seed, 3)
    if kind == "request":
        s["gain"] = _gain(case, seed)
    return s


def run(state):
    kind = state["case"]["kind"]
    if kind == "uneven":
        ub = state["ub"]
        ub.replay()
        return [g.y for g in ub.groups] + [g.xh for g in ub.groups]
    p = state["plan"]
    if kind == "forward":
        return p.forward(state["x"])
    if kind == "inverse":
        return p.inverse(state["y"])
    if kind == "pair":
        y = p.forward(state["x"])
        return y, p.inverse(y)
    if kind == "request":
        y = p.forward(state["x"])
        p.scale_rows(y, state["gain"])
        return y, p.inverse(y)
    if kind == "scan":
        y = p.forward(state["x"])
        energy, peak, by_energy, by_peak = p.plane_metrics(y)
        return y, energy, peak, by_energy, by_peak
    if kind == "stored":
        return p.forward(state["x"]), p.inverse(state["y"])
    s = state["stream"]
    s.reset()
    y = s.forward(state["x"])
    return y, s.inverse(y)


def _row_flops(M):
    return 5.0 * M * math.log2(M)


def work(case):
    """Strain and envelopes read or written once in each direction; 5 m log2 m per transform of length m."""
    kind = case["kind"]
    if kind == "uneven":
        host = np.random.Generator(np.random.PCG64(12345))
        top = (case["n"] // int(case["fs"])).bit_length()
        total = dict(bytes=0.0, flops=0.0)
        for i in range(case["batch"]):
            fs = case["fs"] * (4 if i % 2 else 1)
            one = work(dict(case, kind="pair", fs=fs, n=int((1 << int(host.integers(top))) * fs), batch=1))
            total = {k: total[k] + one[k] for k in total}
        return total
    g = _geometry(case)
    size = 8 if case.get("compute") == "f64" else 4
    env = 2 * size if case.get("envelope") not in ("bf16", "f16") else 4
    rows, B, N = len(g.kc), case["batch"], g.N
    y, x = float(B * rows * g.M * env), float(B * N * size)
    flops = B * (rows * _row_flops(g.M) + 2.5 * N * math.log2(N))
    if kind == "stream":
        q = N // math.gcd(N, g.M)
        hop = N - 2 * q * ((N // 4) // q)
        kept = B * rows * (hop * g.M // N) * env
        return dict(bytes=2.0 * (kept + B * hop * size), flops=2 * flops)
    both = 2 if kind in ("pair", "request", "stored") else 1
    extra = 2 * 0.2 * y if kind == "request" else y if kind == "scan" else 0.0
    return dict(bytes=both * (x + y) + extra, flops=both * flops)


def exact(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        segs, rates = _uneven(case, seed)
        groups = {}
        for i, (x, fs) in enumerate(zip(segs, rates)):
            groups.setdefault((fs, len(x)), []).append(i)
        ys, xs = [], []
        for (fs, n), idx in sorted(groups.items(), key=lambda kv: -kv[0][1]):
            bank = _Bank(dict(case, fs=fs, n=n))
            y = [bank.forward(torch.from_numpy(segs[i]).cuda().double()) for i in idx]
            xs.append(torch.stack([bank.inverse(v, 1e-6) for v in y]))
            ys.append(torch.stack(y))
        return ys + xs
    bank = _Bank(case)
    g = bank.g
    tau = 0.0 if case.get("compute") == "f64" else 1e-6
    if kind == "stream":
        return _exact_stream(case, bank, seed)
    y = x = back = None
    if kind != "inverse":
        x = _strain(case["batch"], g.N, g.fs, seed).double()
        y = torch.stack([bank.forward(v) for v in x])
    if kind == "request":
        y = y * _gain(case, seed)[..., None].double()
    if kind in ("inverse", "stored"):
        src = _envelopes(case, case["batch"], seed, 3)
        src = torch.view_as_complex(src.double()) if kind == "stored" else src.to(torch.complex128)
        back = torch.stack([bank.inverse(v, tau) for v in src])
        if kind == "inverse":
            return back
        return torch.view_as_real(y), back
    if kind == "forward":
        return y
    if kind == "scan":
        a2 = torch.view_as_real(y).square().sum(-1)
        energy, peak = a2.sum((2, 3)), a2.amax((2, 3))
        return y, energy, peak, energy.argmax(1), peak.argmax(1)
    return y, torch.stack([bank.inverse(v, tau) for v in y])


def _exact_stream(case, bank, seed):
    """Overlap-save: chunk i holds the N samples from i hop - 2G on and keeps its central columns; rows carry the
    phase exp(-2 pi i k_c a / N) of their chunk's first sample a; the inverse runs the same chunks over the map."""
    g, J = bank.g, case["batch"]
    q = g.N // math.gcd(g.N, g.M)
    G = q * ((g.N // 4) // q)
    hop = g.N - 2 * G
    Hn, Gm = hop * g.M // g.N, G * g.M // g.N
    x = _strain(1, hop * J, g.fs, seed)[0].double()
    xp = torch.cat([x.new_zeros(2 * G), x])
    kc = torch.stack([k[:, 0] for k in bank.kc])

    def phase(a):
        t = ((kc * a) % g.N).to(torch.float64) * (-2 * math.pi / g.N)
        return torch.polar(torch.ones_like(t), t)[:, :, None]

    y = torch.cat([(bank.forward(xp[i * hop:i * hop + g.N]) * phase(i * hop - 2 * G))[:, :, Gm:Gm + Hn]
                   for i in range(J)], dim=2)
    yp = torch.cat([y.new_zeros((y.shape[0], y.shape[1], 2 * Gm)), y], dim=2)
    back = [bank.inverse(yp[:, :, i * Hn:i * Hn + g.M] * phase(i * hop - 3 * G).conj(), 1e-6)[G:G + hop] for i in range(J)]
    return y, torch.cat(back)
