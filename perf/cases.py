"""Performance cases of the butterfly-filtering library: searches through the public binding (bf.py) over the range
of sizes, sample rates, precisions and calls that its workloads use.

Every case is a dict of plain values:

  api        "correlate" (bf_correlate, results copied to host memory), "stream" (the same enqueued on a caller's
             stream with asynchronous copies into pinned buffers), "plan" (bf_plan_run of a captured search),
             "serve" (requests submitted to the serving loop and polled), "control" (the time-randomised control)
  precision  "split_bf16", "split_fp16", "bf16", "fp32" or "fft_fp32"
  generated  the bank keeps only its chirp parameters and its templates are made inside the call
  quad       quadrature bank (template and Hilbert partner)
  fs, T      sample rate (Hz) and template length (s)
  tracks, senses, durs, I, J, f_min, f_max   the chirp grid (durs sweep times from 0.2 T to T, one: T)
  n, n_min, n_max, noise, snr    number of series, shortest and longest (samples), kind of noise, injected signal
  host       the series are host arrays, else CUDA tensors
  hist, map, parseval, kappa    outputs and tail threshold

Inputs are synthetic, made from the seed alone; lengths, banks and options follow from the case alone.
"""
import math

import numpy as np
import torch

from paper_1802_01685_gb300 import bf

LINEAR, POWERLAW = 0, 1
ASC, DESC, BOTH = 0, 1, 2
TRACKS = {"linear": [LINEAR], "powerlaw": [POWERLAW], "both": [LINEAR, POWERLAW]}
SENSES = {"asc": [ASC], "two": [ASC, DESC], "butterfly": [BOTH]}


def _case(name=None, api="correlate", precision="split_bf16", generated=False, quad=False, fs=2048.0, T=1.0,
          tracks="linear", senses="two", durs=1, I=8, J=16, f_min=50.0, f_max=1000.0, n=1, n_min=8192, n_max=8192,
          noise="white", snr=8.0, host=False, hist=True, map=False, parseval=False, kappa=5.0):
    c = dict(api=api, precision=precision, generated=generated, quad=quad, fs=fs, T=T, tracks=tracks, senses=senses,
             durs=durs, I=I, J=J, f_min=f_min, f_max=f_max, n=n, n_min=n_min, n_max=n_max, noise=noise, snr=snr,
             host=host, hist=hist, map=map, parseval=parseval, kappa=kappa)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest search: 4 s at 2048 Hz from host memory against 256 linear chirps (a first look at a short
        # trigger, where latency and launches count)
        _case("trigger_4s", host=True),
        # follow-up of a short segment with an odd length in single precision
        _case("followup_fp32", precision="fp32", n=2, n_min=30011, n_max=32768, I=32, J=32),
        # a quick look in plain BF16 on the caller's stream, results into pinned buffers
        _case("quicklook_stream_bf16", api="stream", precision="bf16", n=1, n_min=131071, n_max=131071, I=64, J=64,
              noise="gw", f_min=20.0, hist=False),
        # one 16 s block of strain after another through a captured plan (FFT route)
        _case("block_plan_fft", api="plan", precision="fft_fp32", fs=4096.0, tracks="powerlaw", senses="asc", I=64,
              J=64, f_min=40.0, f_max=400.0, n_min=65536, n_max=65536, noise="gw"),
        # the same kind of block, two detectors, through a plan of the tensor-core route
        _case("block_plan_split", api="plan", fs=4096.0, tracks="powerlaw", senses="asc", I=32, J=32, f_min=40.0,
              f_max=400.0, n=2, n_min=65536, n_max=65536, noise="gw"),
        # 64 s of two detectors against a quarter of the GW bank, the default precision, stored bank
        _case("gw_pair_split", fs=4096.0, tracks="powerlaw", senses="asc", I=128, J=128, f_min=40.0, f_max=400.0, n=2,
              n_min=262144, n_max=262144, noise="gw", hist=False),
        # the GW step on the FFT route: two detectors and two controls against 65,536 generated templates
        _case("gw_step_fft_generated", precision="fft_fp32", generated=True, fs=4096.0, tracks="powerlaw",
              senses="asc", I=256, J=256, f_min=40.0, f_max=400.0, n=4, n_min=262144, n_max=262144, noise="gw"),
        # 42 light curves of 20-200 s in 0.5 ms bins (odd lengths, templates of 2000 samples) in one batch
        _case("grb_batch_fft", precision="fft_fp32", fs=2000.0, I=32, J=32, f_min=20.0, f_max=999.0, n=42,
              n_min=40001, n_max=399999, noise="counts"),
        # short and full-length sweeps of both kinds, generated, split-FP16 (a slice of the full bank)
        _case("full_bank_fp16_generated", precision="split_fp16", generated=True, tracks="both", durs=9, I=10, J=12,
              f_min=20.0, n_min=65536, n_max=65536, hist=False),
        # phase-blind search with predicted noise level: quadrature bank, Parseval tails, painted map
        _case("quadrature_parseval_map", precision="fft_fp32", quad=True, fs=4096.0, tracks="powerlaw", senses="asc",
              I=32, J=32, f_min=40.0, f_max=400.0, n_min=50003, n_max=50003, noise="gw", snr=60.0, map=True,
              kappa=12.0),
        # a few requests of different lengths served together
        _case("serve_mixed", api="serve", n=6, n_min=9001, n_max=131072, I=32, J=32, noise="white", host=True),
        # the control of one 64 s series
        _case("control_64s", api="control", fs=4096.0, n_min=262144, n_max=262144, noise="gw"),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["correlate", "correlate", "correlate", "stream", "plan", "plan", "serve", "control"])
    fs = rng.choice([2000.0, 2048.0, 4096.0, 4096.0])
    n_min = _spread(rng, 6000 if fs < 4000 else 9000, 300000)
    if api == "control":
        n = _spread(rng, 1000, 500000)
        return _case(api=api, fs=fs, n_min=n, n_max=n, noise=rng.choice(["white", "gw", "counts"]))
    precision = rng.choice(["split_bf16", "split_bf16", "fft_fp32", "fft_fp32", "fft_fp32", "bf16", "split_fp16", "fp32"])
    n = 1 if rng.random() < 0.5 else _spread(rng, 2, 12)
    quad = rng.random() < 0.2
    c = _case(api=api, precision=precision, fs=fs, quad=quad, generated=rng.random() < 0.3,
              tracks=rng.choice(["linear", "powerlaw", "both"]), senses=rng.choice(["asc", "two", "butterfly"]),
              durs=rng.choice([1, 1, 1, 3]), I=_spread(rng, 4, 64), J=_spread(rng, 4, 64),
              f_min=float(rng.randint(20, 60)), f_max=float(rng.randint(400, 990)), n=n, n_min=n_min,
              n_max=n_min if n == 1 else min(300000, int(n_min * rng.uniform(1.0, 4.0))),
              noise=rng.choice(["white", "gw", "counts"]), host=api == "serve" or rng.random() < 0.3,
              hist=rng.random() < 0.5 and precision in ("fp32", "fft_fp32"), parseval=api != "serve" and rng.random() < 0.2)
    # no dearer than the largest listed case: fewer templates where the correlation would be
    rate = {"fp32": 3e9, "fft_fp32": 1e11, "bf16": 8e10, "split_bf16": 2.5e10, "split_fp16": 2.5e10}[precision]
    while _lags(c) * _templates(c) * (2 if quad else 1) > 0.1 * rate:
        if c["I"] >= c["J"]:
            c["I"] = max(1, c["I"] // 2)
        else:
            c["J"] = max(1, c["J"] // 2)
        if c["I"] * c["J"] == 1:
            break
    return c


# ---------------------------------------------------------------- geometry

def _M(c):
    return int(math.floor(c["T"] * c["fs"] + 0.5))


def _durations(c):
    d = c["durs"]
    return [c["T"]] if d == 1 else [c["T"] * (0.2 + 0.8 * i / (d - 1)) for i in range(d)]


def _templates(c):
    return len(TRACKS[c["tracks"]]) * len(SENSES[c["senses"]]) * c["durs"] * c["I"] * c["J"]


def _lengths(c):
    n, lo, hi = c["n"], c["n_min"], c["n_max"]
    return [lo + int((hi - lo) * ((i * 0.6180339887498949) % 1.0)) for i in range(n)]


def _lags(c):
    return sum(x - _M(c) + 1 for x in _lengths(c))


def _grid(c):
    return dict(tracks=TRACKS[c["tracks"]], senses=SENSES[c["senses"]], durations=_durations(c), f_min=c["f_min"],
                f_max=c["f_max"], I=c["I"], J=c["J"])


def _slices(c):
    """serve: the template range of each request."""
    K = _templates(c)
    return [(i * K // (2 * c["n"]), K - (i * K) // (3 * c["n"])) for i in range(c["n"])]


# ---------------------------------------------------------------- inputs

def _signal(c):
    """An injected chirp that is on no bank's grid: 1 s, Hann envelope, unit norm."""
    M, fs = _M(c), c["fs"]
    t = torch.arange(M, dtype=torch.float64, device="cuda") / fs
    f = 45.0 + (380.0 - 45.0) * (t / c["T"]) ** 2
    w = torch.sin(math.pi * (t * fs + 0.5) / M) ** 2
    s = w * torch.sin(2 * math.pi * torch.cumsum(f, 0) / fs)
    return s / s.norm()


def _noise(c, n, g):
    fs = c["fs"]
    w = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    if c["noise"] == "white":
        return w
    f = torch.fft.rfftfreq(n, 1.0 / fs, device="cuda", dtype=torch.float64)
    if c["noise"] == "gw":              # 1/f below 30 Hz, flat above
        amp = torch.where(f < 30.0, 30.0 / f.clamp(min=1.0), torch.ones_like(f))
        amp[0] = 0.0
        y = torch.fft.irfft(torch.fft.rfft(w) * amp, n)
        return y / y.std()
    amp = f.clamp(min=fs / n) ** (-5.0 / 6.0)      # photon counts on a Kolmogorov field, 500 per second
    amp[0] = 0.0
    y = torch.fft.irfft(torch.fft.rfft(w) * amp, n)
    lam = (500.0 * (1.0 + 0.3 * y / y.std()) / fs).clamp(min=0.0)
    k = torch.poisson(lam, generator=g)
    return k - k.mean()


def _series(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    out, s = [], _signal(c)
    for n in _lengths(c):
        x = _noise(c, n, g)
        if c["api"] != "control":
            at = int(torch.randint(0, n - len(s) + 1, (1,), device="cuda", generator=g))
            x[at:at + len(s)] += c["snr"] * x.std() * s
        out.append(x.to(torch.float32))
    return out


# ---------------------------------------------------------------- the program's state

_ctx = None


def _context():
    """One context for the process, as a program keeps one."""
    global _ctx
    if _ctx is None:
        _ctx = bf.bf_init()
    return _ctx


class State:
    """What the program holds: the context, a bank, a plan where it uses one, the series."""

    def __init__(self, case, seed):
        c = self.case = dict(case)
        self.ctx = _context()
        self.bank = self.plan = None
        self.seed = int(seed)
        self.series = _series(c, seed)
        if c["host"]:
            self.series = [x.cpu().numpy() for x in self.series]
        if c["api"] == "control":
            self.out = torch.empty_like(self.series[0])
            return
        layout = {"fp32": bf.BF_BANK_FP32, "split_fp16": bf.BF_BANK_SPLIT_FP16}.get(c["precision"], bf.BF_BANK_SPLIT_BF16)
        storage = (bf.BF_BANK_GENERATED if c["generated"] else layout) | (bf.BF_BANK_QUADRATURE if c["quad"] else 0)
        self.bank = bf.bf_bank_create_grid(self.ctx, _grid(c), c["fs"], c["T"], storage)
        kw = dict(precision=c["precision"], want_hist=c["hist"], want_map=c["map"], kappa=c["kappa"],
                  want_tails=c["parseval"], tail_sigma=bf.BF_SIGMA_PARSEVAL if c["parseval"] else bf.BF_SIGMA_WHITE)
        if c["api"] == "stream":
            self.stream = torch.cuda.Stream()
            kw["stream"] = self.stream.cuda_stream
            K = _templates(c)
            self.pinned = []
            for _ in self.series:
                t = dict(max=torch.empty(K, dtype=torch.float32), argmax=torch.empty(K, dtype=torch.int32),
                         sigma=torch.empty(K, dtype=torch.float32))
                if c["hist"]:
                    t["hist"] = torch.empty(1024, dtype=torch.int32)
                t = {k: v.pin_memory() for k, v in t.items()}
                self.pinned.append({k: v.numpy().view(np.uint32) if k == "hist" else v.numpy() for k, v in t.items()})
        if c["api"] == "serve":
            self.opts = [bf.make_opts(bank_begin=a, bank_end=b, **kw) for a, b in _slices(c)]
        else:
            self.opts = bf.make_opts(**kw)
        if c["api"] == "plan":
            self.plan = bf.bf_plan_create(self.ctx, self.bank, _lengths(c), c["fs"], self.opts)

    def __del__(self):
        try:
            if self.plan is not None:
                bf.bf_plan_destroy(self.plan)
            if self.bank is not None:
                bf.bf_bank_destroy(self.bank)
        except Exception:
            pass


def prepare(case, seed):
    return State(case, seed)


def _outputs(c, res, s):
    got = bf.bf_result_copy_to_host(res, s, want_hist=c["hist"], want_map=c["map"])
    return {k: v for k, v in got.items() if v is not None}


def _gather(c, res):
    out = {"series": _few([_outputs(c, res, s) for s in range(c["n"])])}
    if c["n"] > 1:
        out["mean_max"] = bf.bf_result_copy_mean_max(res)
    if c["parseval"]:
        out["sigma_pred"] = np.stack([bf.bf_result_copy_sigma_pred(res, s) for s in range(c["n"])])
    return out


def _few(per):
    """The outputs of all series as one array each where there are many series."""
    if len(per) <= 4:
        return per
    return [{k: np.stack([p[k] for p in per]) for k in per[0]}]


def run(state):
    c = state.case
    if c["api"] == "control":
        bf.bf_control_randomize(state.ctx, state.series[0], state.seed, state.out)
        return state.out
    if c["api"] == "plan":
        return _gather(c, bf.bf_plan_run(state.plan, state.series))
    if c["api"] == "serve":
        tickets = [bf.bf_serve_submit(state.ctx, state.bank, x, c["fs"], o) for x, o in zip(state.series, state.opts)]
        out = []
        for t in tickets:
            _, res = bf.bf_serve_poll(state.ctx, t)
            out.append(_outputs(c, res, 0))
            bf.bf_result_destroy(res)
        return out
    res = bf.bf_correlate(state.ctx, state.bank, state.series, c["fs"], state.opts)
    if c["api"] == "stream":
        st = state.stream.cuda_stream
        per = [bf.bf_result_copy_to_host_async(res, s, state.pinned[s], st, want_hist=c["hist"]) for s in range(c["n"])]
        state.stream.synchronize()
        out = {"series": _few([{k: v for k, v in p.items() if v is not None} for p in per])}
        bf.bf_result_check(res)
    else:
        out = _gather(c, res)
    bf.bf_result_destroy(res)
    return out


# ---------------------------------------------------------------- work, tolerance, exact values

def work(case):
    c = case
    N, K, M = sum(_lengths(c)), _templates(c), _M(c)
    if c["api"] == "control":
        return {"bytes": 8 * N, "flops": 0}
    rows = K * (2 if c["quad"] else 1)
    lags = _lags(c)
    if c["api"] == "serve":
        pairs = sum((n - M + 1) * (b - a) for n, (a, b) in zip(_lengths(c), _slices(c)))
    else:
        pairs = lags * K
    pairs *= 2 if c["quad"] else 1
    # series once, templates once (parameters only where the bank keeps no more), outputs once
    nbytes = 4 * N + rows * (48 if c["generated"] else 4 * M) + c["n"] * (12 * K + (4096 if c["hist"] else 0))
    if c["map"]:
        nbytes += 4 * sum(math.ceil(n / (c["fs"] * 1e-3)) * math.ceil(c["fs"] / 8.0) for n in _lengths(c))
    # the direct method: 2 M per lag and template; the FFT route: 5 N log2 N per 8192-point transform over its lags
    flops = 5 * 8192 * 13 / (16385 - M) * pairs if c["precision"] == "fft_fp32" else 2.0 * M * pairs
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    c = case
    if c["api"] == "control":
        return "exact"
    # four times the distance from the 64-bit values (split-BF16 6e-6, split-FP16 2e-6, FP32 8e-7, FFT 2.4e-7);
    # plain BF16 rounds its operands the same way everywhere, so only its accumulation may differ, as split-BF16's.
    # Whole values: lags of near ties, and counts at the edges of the histogram's bins.
    rel = {"split_bf16": 2.4e-5, "bf16": 2.4e-5, "split_fp16": 1e-5, "fp32": 3e-6, "fft_fp32": 1e-6}[c["precision"]]
    return {"rel": rel, "max": 10 * rel, "differ": 5e-3 if c["precision"] in ("fp32", "fft_fp32") else 1e-2}


def _chirps(c):
    for tr in TRACKS[c["tracks"]]:
        for se in SENSES[c["senses"]]:
            for D in _durations(c):
                for i in range(c["I"]):
                    lo = c["f_min"] + (c["f_max"] - c["f_min"]) * i / c["I"]
                    for j in range(c["J"]):
                        yield tr, se, lo, lo + (c["f_max"] - lo) * (j + 1) / c["J"], D


def _rows64(c, chirps, quad):
    """Templates (quad: their Hilbert partners) of the given chirps at unit norm, in 64 bits."""
    M, fs = _M(c), c["fs"]
    p = torch.tensor(chirps, dtype=torch.float64, device="cuda")
    tr, se, lo, hi, D = (p[:, i:i + 1] for i in range(5))
    MD = torch.floor(D * fs + 0.5)
    first = torch.floor((M - MD) / 2)
    j = torch.arange(M, dtype=torch.float64, device="cuda")[None, :] - first
    inside = (j >= 0) & (j < MD)
    t = torch.where(inside, j, torch.zeros_like(j)) / fs
    lin = lo * t + (hi - lo) * t * t / (2 * D)
    tc = D / (1 - (lo / hi) ** (8.0 / 3.0))
    pw = 1.6 * lo * tc * (1 - (1 - t / tc).clamp(min=0.0) ** 0.625)
    cyc = torch.where(tr == LINEAR, lin, pw)
    ph = 2 * math.pi * (cyc - torch.round(cyc))
    w = torch.sin(math.pi * (j + 0.5) / MD) ** 2
    g = torch.where(inside, w * (torch.sin(ph) if quad else torch.cos(ph)), torch.zeros_like(j))
    rev = g.flip(1) * (-1.0 if quad else 1.0)
    h = torch.where(se == ASC, g, torch.where(se == DESC, rev, g + rev))
    return h / h.norm(dim=1, keepdim=True)


def exact(case, seed):
    c = case
    series = _series(c, seed)
    if c["api"] == "control":
        x = series[0].cpu().numpy()
        z = (np.arange(len(x), dtype=np.uint64) ^ np.uint64(int(seed))) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return torch.from_numpy(x[np.argsort(z ^ (z >> np.uint64(31)), kind="stable")])
    K, M, rows = _templates(c), _M(c), 2 if c["quad"] else 1
    if _lags(c) * K * rows > 3e10:
        return None                                     # over 20 seconds in 64 bits
    chirps = [tuple(map(float, x)) for x in _chirps(c)]
    slices = _slices(c) if c["api"] == "serve" else [(0, K)] * c["n"]
    per, preds = [], []
    for x32, (a, b) in zip(series, slices):
        x = x32.double()
        n, L = len(x), len(x) - M + 1
        F = 1 << (n - 1).bit_length()
        X = torch.fft.rfft(x, F)
        S = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.cumsum(x * x, 0)])
        inv = 1.0 / torch.sqrt(S[M:] - S[:-M])
        vmax, arg, sig, pred = [], [], [], []
        if c["parseval"]:
            G = 16384
            if n >= G:
                P = (torch.fft.fft(x.unfold(0, G, G // 2)).abs() ** 2).mean(0)
            else:
                P = torch.fft.fft(x, G).abs() ** 2 * (G / n)
        step = max(1, min(512, (1 << 27) // F))
        for k in range(a, b, step):
            r2 = 0.0
            s2 = 0.0
            for q in range(rows):
                h = _rows64(c, chirps[k:min(k + step, b)], q == 1)
                rho = torch.fft.irfft(X * torch.fft.rfft(h, F).conj(), F)[:, :L] * inv
                r2 = rho * rho if q == 0 else r2 + rho * rho
                if c["parseval"]:
                    s2 = s2 + (torch.fft.fft(h, 16384).abs() ** 2 * P).sum(1)
            m2, at = r2.max(1)
            vmax.append(m2.sqrt())
            arg.append(at)
            sig.append(r2.mean(1).sqrt())
            if c["parseval"]:
                pred.append(torch.sqrt(s2 / (16384.0 ** 2 * M * (x * x).mean())))
        o = {"max": torch.cat(vmax).cpu().numpy(), "argmax": torch.cat(arg).cpu().numpy().astype(np.int32),
             "sigma": torch.cat(sig).cpu().numpy()}
        if c["hist"]:
            o["hist"] = np.bincount(np.minimum((o["max"] * 1024).astype(np.int64), 1023), minlength=1024).astype(np.uint32)
        if c["map"]:
            o["map"] = None
        per.append(o)
        if pred:
            preds.append(torch.cat(pred).cpu().numpy())
    if c["api"] == "serve":
        return per
    out = {"series": _few(per)}
    if c["n"] > 1 and c["api"] != "stream":
        out["mean_max"] = np.mean([p["max"] for p in per], axis=0)
    if c["parseval"] and c["api"] != "stream":
        out["sigma_pred"] = np.stack(preds)
    return out
