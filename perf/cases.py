"""The work this X-engine is measured on: integrations of 4+4-bit frames through the public entry points.

A case is a dict of plain values; its "kind" names the entry points it goes through:

    frame    accumulate() once per input frame, then readout(reset=True)
    noalloc  correlate_noalloc() into a buffer of the caller's
    host     accumulate_host() from pinned memory, then readout_host(reset=True)
    batch    accumulate_batch() over frames of unlike sizes, then a readout of each
    gated    accumulate_gated() into G gates, then a readout of each
    lags     shift_lags(), the per-element delay before correlation

Inputs are Gaussian levels (sigma in quantisation steps), rounded, clipped to
[-8, 7] and packed as the library reads them: uint8 [T][F][N], high nibble =
real + 8, low nibble = imaginary + 8. Outputs are the int32 visibilities
[F][N(N+1)/2][2] (for lags: the shifted uint8 frame).
"""
import math

import torch

import paper_1503_06203_gb300 as xe

# ranges of the drawn cases
MAX_OPS = 2.0e12    # 4 N (N+1) F T summed over a pass
MAX_IN = 1 << 30    # input bytes of a pass
MAX_OUT = 1 << 30   # visibility bytes of a pass


def listed():
    return [
        # the smallest frame a user correlates: one array test, latency only
        {"name": "tiny", "kind": "frame", "N": 16, "F": 4, "T": 256, "frames": 1, "sigma": 2.5},
        # one stream of a serving system: 16 short frames into resident sums, then a readout
        {"name": "stream16", "kind": "frame", "N": 256, "F": 16, "T": 1024, "frames": 16, "sigma": 2.5},
        # the headline integration: 128 dual-polarisation feeds, 256 bands
        {"name": "pathfinder", "kind": "frame", "N": 256, "F": 256, "T": 16384, "frames": 1, "sigma": 2.5},
        # the largest array, a common tone on every input: as much output as the card writes in a frame
        {"name": "large_n", "kind": "frame", "N": 8192, "F": 4, "T": 2048, "frames": 1, "sigma": 2.5, "tone": 3.0},
        # a mid-size array, the served workload's middle stream
        {"name": "mid_n", "kind": "frame", "N": 1024, "F": 64, "T": 4096, "frames": 1, "sigma": 2.5},
        # an array whose element count fills no row or tile, and a time axis that fills no chunk
        {"name": "odd", "kind": "frame", "N": 250, "F": 61, "T": 4001, "frames": 1, "sigma": 1.5},
        # a real-time host that reserves every byte up front
        {"name": "noalloc", "kind": "noalloc", "N": 512, "F": 16, "T": 2048, "sigma": 2.5},
        # host buffers in, host buffers out, as a correlator node fed by its network card
        {"name": "host", "kind": "host", "N": 256, "F": 64, "T": 8192, "sigma": 2.5},
        # frames of several arrays that arrived together (N 64 to 2048)
        {"name": "batch_uneven", "kind": "batch", "frames": 16, "seed0": 3, "nmin": 64, "nmax": 2048, "fmax": 24,
         "tmin": 512, "tmax": 4096},
        # many small frames in one call
        {"name": "batch_small", "kind": "batch", "frames": 48, "seed0": 5, "nmin": 64, "nmax": 256, "fmax": 4,
         "tmin": 512, "tmax": 2048},
        # a pulsar binned into 8 gates of its period
        {"name": "gated", "kind": "gated", "N": 256, "F": 64, "T": 16384, "G": 8, "period": 1024, "phase": 100,
         "sigma": 2.5},
        # cable lengths taken out of a frame before it is correlated
        {"name": "lags", "kind": "lags", "N": 256, "F": 256, "T": 8192, "maxlag": 64, "sigma": 2.5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, nmax, odd):
    """An element count from 16 to nmax over its logarithm: a multiple of 16, or any number."""
    n = min(nmax, _log(rng, 16, nmax))
    return n if odd else max(16, n // 16 * 16)


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "batch", "gated", "lags", "noalloc", "host"])
    sigma = round(rng.uniform(1.5, 3.5), 2)
    if kind == "batch":
        nmin = rng.choice([64, 64, 128])
        nmax = rng.choice([n for n in (128, 256, 512, 1024, 2048) if n > nmin])
        frames = rng.randint(4, 48) if nmax <= 512 else rng.randint(4, 16)
        fmax = _log(rng, 2, 64) if nmax <= 512 else _log(rng, 2, 24)
        c = {"kind": "batch", "frames": frames, "seed0": rng.randrange(1 << 30), "nmin": nmin, "nmax": nmax,
             "fmax": fmax, "tmin": 512, "tmax": 256 * rng.randint(3, 16)}
        while True:  # within the caps
            w = work(c)
            if w["flops"] <= MAX_OPS and w["bytes"] <= MAX_IN + MAX_OUT:
                return c
            c["frames"] = max(1, c["frames"] // 2)
            c["fmax"] = max(1, c["fmax"] // 2)
    odd = rng.random() < 0.4 and kind != "noalloc"
    N = _size(rng, 1024 if kind in ("gated", "host") else 2048 if kind == "lags" else 8192, odd)
    T = _log(rng, 128, 16384)
    if kind != "lags":
        T = min(T, int(MAX_OPS / (4 * N * (N + 1))))
    if not odd:
        T = max(128, T // 128 * 128)
    if kind == "lags":
        F = max(1, min(_log(rng, 1, 256), (MAX_IN // 2) // (N * T)))
        return {"kind": "lags", "N": N, "F": F, "T": T, "maxlag": _log(rng, 1, 100), "sigma": sigma}
    reps = 1
    if kind == "frame" and rng.random() < 0.3:
        reps = max(1, min(rng.randint(2, 16), int(MAX_OPS / (4 * N * (N + 1) * T)), MAX_IN // (N * T)))
    if kind == "gated":
        reps = 8  # (a share of the cap: the gates' outputs)
    out = 4 * N * (N + 1)  # bytes of a band's visibilities
    cap = min(MAX_OPS / (4 * N * (N + 1) * T * (1 if kind == "gated" else reps)), MAX_IN / (N * T * reps),
              MAX_OUT / (out * (reps if kind == "gated" else 1)))
    if kind == "host":
        cap /= 4  # (pinned memory)
    F = max(1, min(_log(rng, 1, 256), int(cap)))
    if kind == "gated":
        G = rng.randint(2, 8)
        period = _log(rng, 128, 4096)
        return {"kind": kind, "N": N, "F": F, "T": T, "G": G, "period": period, "phase": rng.randrange(period),
                "sigma": sigma}
    c = {"kind": kind, "N": N, "F": F, "T": T, "sigma": sigma}
    if kind == "frame":
        c["frames"] = reps
    return c


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _frame(g, N, F, T, sigma, tone=0.0):
    """A packed frame uint8 [T][F][N]; tone: amplitude of a sequence common to all elements."""
    x = torch.empty(T, F, N, dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 26) // (F * N))
    w = 2 * math.pi * 37 / T
    for t in range(0, T, step):
        n = min(step, T - t)
        parts = []
        for k in range(2):
            v = torch.randn(n, F, N, generator=g, device="cuda").mul_(sigma)
            if tone:
                a = torch.arange(t, t + n, device="cuda", dtype=torch.float32) * w
                v += (tone * (a.sin() if k else a.cos())).reshape(n, 1, 1)
            parts.append(v.round_().clamp_(-8, 7).add_(8).to(torch.uint8))
        x[t:t + n] = (parts[0] << 4) | parts[1]
    return x


def _batch_frames(case):
    """(N, F, T, sigma) of each frame of a batch: sizes from powers of two, F and T uniform."""
    import random

    r = random.Random(case["seed0"])
    sizes = [n for n in (64, 128, 256, 512, 1024, 2048) if case["nmin"] <= n <= case["nmax"]]
    out = []
    for _ in range(case["frames"]):
        N = r.choice(sizes)
        out.append((N, r.randint(1, case["fmax"]), 256 * r.randint(case["tmin"] // 256, case["tmax"] // 256),
                    r.uniform(1.5, 3.5)))
    return out


def _vis(N, F):
    return torch.empty(F, N * (N + 1) // 2, 2, dtype=torch.int32, device="cuda")


def _inputs(case, seed):
    """The input frames of a case, on the GPU."""
    g = _gen(seed)
    if case["kind"] == "batch":
        return [_frame(g, N, F, T, s) for N, F, T, s in _batch_frames(case)]
    return [_frame(g, case["N"], case["F"], case["T"], case["sigma"], case.get("tone", 0.0))
            for _ in range(case.get("frames", 1))]


def _lags(case, seed):
    m = case["maxlag"]
    return torch.randint(-m, m, (case["N"],), generator=_gen(seed + 1), device="cuda", dtype=torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    xs = _inputs(case, seed)
    s = {"kind": kind, "x": xs}
    if kind == "batch":
        shapes = _batch_frames(case)
        s["c"] = [xe.Correlator(N, F, T) for N, F, T, _ in shapes]
        s["out"] = [_vis(N, F) for N, F, _, _ in shapes]
        return s
    N, F, T = case["N"], case["F"], case["T"]
    if kind == "frame":
        s["c"] = xe.Correlator(N, F, T)
        s["out"] = _vis(N, F)
    elif kind == "noalloc":
        s["out"] = _vis(N, F)
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "host":
        s["x"] = xs[0].cpu().pin_memory()
        s["c"] = xe.Correlator(N, F, T)
        s["out"] = torch.empty(F, N * (N + 1) // 2, 2, dtype=torch.int32, pin_memory=True)
    elif kind == "gated":
        s["c"] = [xe.Correlator(N, F, T) for _ in range(case["G"])]
        s["out"] = [_vis(N, F) for _ in range(case["G"])]
        s["period"], s["phase"] = case["period"], case["phase"]
    elif kind == "lags":
        s["lags"] = _lags(case, seed)
        s["out"] = torch.empty_like(xs[0])
    return s


def run(state):
    kind = state["kind"]
    if kind == "frame":
        c = state["c"]
        for x in state["x"]:
            c.accumulate(x)
        return c.readout(state["out"], reset=True)
    if kind == "noalloc":
        return xe.correlate_noalloc(state["x"][0], state["out"], state["status"])
    if kind == "host":
        state["c"].accumulate_host(state["x"])
        return state["c"].readout_host(state["out"], reset=True)
    if kind == "batch":
        xe.accumulate_batch(state["c"], state["x"])
        return [c.readout(o, reset=True) for c, o in zip(state["c"], state["out"])]
    if kind == "gated":
        xe.accumulate_gated(state["c"], state["x"][0], state["period"], state["phase"])
        return [c.readout(o, reset=True) for c, o in zip(state["c"], state["out"])]
    return xe.shift_lags(state["x"][0], state["lags"], state["out"])


def work(case):
    """Each input byte read once, each output byte written once; 8 operations per visibility and sample."""
    kind = case["kind"]
    if kind == "batch":
        dims = [(N, F, T) for N, F, T, _ in _batch_frames(case)]
    else:
        dims = [(case["N"], case["F"], case["T"])]
    reps = case.get("frames", 1) if kind == "frame" else 1
    nin = sum(N * F * T for N, F, T in dims) * reps
    if kind == "lags":
        return {"bytes": 2.0 * nin + 4.0 * case["N"], "flops": 0.0}
    nout = sum(4 * N * (N + 1) * F for N, F, _ in dims) * (case["G"] if kind == "gated" else 1)
    return {"bytes": float(nin + nout), "flops": float(sum(4 * N * (N + 1) * F * T for N, F, T in dims) * reps)}


def _correlate(frames, keep=None):
    """Packed visibilities of frames (all their samples, or those of the row mask `keep`), in 64 bits."""
    T, F, N = frames[0].shape
    iu = torch.triu_indices(N, N, device="cuda")
    flat = iu[0] * N + iu[1]
    del iu
    out = torch.empty(F, flat.numel(), 2, dtype=torch.int64, device="cuda")
    for f in range(F):
        re = torch.zeros(N, N, dtype=torch.float64, device="cuda")
        im = torch.zeros(N, N, dtype=torch.float64, device="cuda")
        for x in frames:
            b = x[:, f] if keep is None else x[keep, f]
            xr = (b >> 4).to(torch.float64) - 8
            xi = (b & 15).to(torch.float64) - 8
            re.addmm_(xr.T, xr).addmm_(xi.T, xi)
            im.addmm_(xi.T, xr).addmm_(xr.T, xi, alpha=-1)
        out[f, :, 0] = re.reshape(-1)[flat].to(torch.int64)
        out[f, :, 1] = im.reshape(-1)[flat].to(torch.int64)
    return out


def exact(case, seed):
    kind = case["kind"]
    if work(case)["flops"] > 1.5e12:  # (over about 10 seconds in 64 bits)
        return None
    xs = _inputs(case, seed)
    if kind == "batch":
        return [_correlate([x]) for x in xs]
    if kind == "gated":
        t = torch.arange(case["T"], device="cuda")
        gate = (t + case["phase"]) % case["period"] * case["G"] // case["period"]
        return [_correlate(xs, gate == g) for g in range(case["G"])]
    if kind == "lags":
        x = xs[0]
        lags = _lags(case, seed).cpu().tolist()
        y = torch.full_like(x, 0x88)
        T = x.shape[0]
        for i, lag in enumerate(lags):
            if abs(lag) < T:
                if lag >= 0:
                    y[lag:, :, i] = x[:T - lag, :, i]
                else:
                    y[:lag, :, i] = x[-lag:, :, i]
        return y
    out = _correlate(xs)
    return out.cpu() if kind == "host" else out
