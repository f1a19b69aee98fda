"""The work that the framework is timed on: one pass per case through the public entry points.

A case is a dict of plain values; `kind` says which entry point it goes through:

  call       Synth.render (or render_f32): one window of a tone set, from a cursor
  stream     Synth.render_stream: a record in pipelined chunks
  rearrange  seek + set_tones + set_chirps + render_stream into pinned host memory: a request end to end
  engine     Synth.render with the tensor-core static engine
  table      Synth.table_gemm: a whole periodic record
  mux        render_multiplexed: several channels interleaved
  replay     Synth.render behind a periodic hand-off (set_periodic in prepare)

All inputs are synthetic and made from the seed: tones in the 80-180 MHz band at 280 MS/s unless the
case says otherwise, as in paper_2403_15582_gb300/workloads.py.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_15582_gb300 as awg

FS = 280e6
LINEAR, MINJERK, EXPONENTIAL = awg.PROFILE_LINEAR, awg.PROFILE_MINJERK, awg.PROFILE_EXPONENTIAL

# The largest pass of each form of work: tone-samples of a direct render and of a tensor-core sum.
MAX_DIRECT = 10000 * (1 << 20)
MAX_GEMM = 10000 * (1 << 24)


def _call(name=None, *, K, n, start=0, chirps=0, profile="mixed", ms=35.0, ramps=0, f32=False, sine="sfu", **more):
    """A render case: K tones, `chirps` of them chirping for `ms` from sample 0 on, `ramps` of them with an
    amplitude ramp over the first 3/4 of the window, samples start .. start + n - 1."""
    c = dict(kind="call", K=K, n=n, start=start, chirps=chirps, profile=profile, ms=ms, ramps=ramps, f32=f32, sine=sine)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a few tones, some with chirps that start and end inside the window, FP32 sum
        # wanted too (the size of __graft_entry__.smoke): launches and latency
        _call("tiny", K=8, n=10000, chirps=5, ms=0.012, f32=True),
        # a static tweezer comb of 100 tones, 2^20 samples in one call (workloads.static_100)
        _call("comb_100", K=100, n=1 << 20),
        # a static comb of odd size on the rotator sine, from a cursor inside a tile, the ragged length of
        # the last chunk of a 35 ms record
        _call("rotator_777", K=777, n=100672, start=12345, sine="rotator"),
        # one 2^18-sample chunk in the middle of 1000 chirps: what a streaming program asks for every 0.94 ms
        _call("chunk_1000", K=1000, n=1 << 18, start=17 << 18, chirps=1000),
        # the playback record: 1000 tones chirped for 35 ms, 9.8M samples in 2^18-sample chunks
        _call("record_1000", K=1000, n=9800000, chirps=1000, kind="stream", chunk=1 << 18),
        # one 2^20-sample chunk of 10,000 tones that all chirp: the largest real-time load
        _call("chunk_10000", K=10000, n=1 << 20, start=3 << 20, chirps=10000),
        # tweezers switched on and off: 500 of 600 tones ramp their amplitude inside the window, FP32 sum
        _call("ramps_500", K=600, n=200000, start=1000, ramps=500, f32=True),
        # a rearrangement request end to end, host arrays to pinned host samples: 1500 tones, 100 of them
        # moved within 1 ms, 8 chunks of 2^16 samples
        _call("rearrange_1500", K=1500, n=1 << 19, chirps=100, ms=1.0, kind="rearrange", chunk=1 << 16),
        # streaming 10,000 tones with the tensor-core engine, groups of 100 chirping for 1 ms in turn
        # (workloads.stream_rotating): one 2^20-sample chunk
        dict(name="engine_10000", kind="engine", K=10000, n=1 << 20, start=0, groups=4, group=100, prec="fp16"),
        # a periodic table of 10,000 tones and 2^24 samples on the tensor cores (workloads.table_10000)
        dict(name="table_10000", kind="table", K=10000, log2=24, prec="bf16"),
        # four channels of 250 chirping tones each, interleaved for a four-channel card
        _call("mux_4", K=250, n=1 << 18, chirps=250, kind="mux", channels=4),
        # the static hold after a playback: 2^27 samples replayed from a periodic table of 2^24
        dict(name="replay", kind="replay", K=1000, log2=24, n=1 << 27, start=1 << 20),
    ]


def _log(rng, lo, hi):
    """An integer in lo .. hi, spread over the logarithm, odd about half of the time."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["call"] * 6 + ["stream", "stream", "rearrange", "engine", "table", "mux", "mux", "replay"])
    if kind == "table":
        K, log2 = _log(rng, 50, 10000), rng.randint(16, 24)
        return dict(kind=kind, K=K, log2=log2, prec=rng.choice(["fp16", "bf16"]))
    if kind == "replay":
        return dict(kind=kind, K=_log(rng, 1, 1000), log2=rng.randint(16, 24), n=_log(rng, 1 << 18, 1 << 27),
                    start=8 * rng.randint(0, 1 << 20) + rng.choice([0, 0, 0, 3]))
    if kind == "engine":
        K, group = _log(rng, 500, 10000), rng.choice([10, 50, 100])
        return dict(kind=kind, K=K, n=_log(rng, 1 << 16, 1 << 22), start=rng.randint(0, 100000), groups=rng.choice([0, 1, 2, 4]),
                    group=group, prec=rng.choice(["fp16", "bf16"]))
    channels = rng.choice([2, 3, 4, 8]) if kind == "mux" else 1
    K = _log(rng, 4, 1000) if kind == "mux" else _log(rng, 4, 10000)
    top = MAX_DIRECT // (K * channels)
    if kind == "call":
        n = _log(rng, 2000, min(1 << 22, top))
    elif kind == "mux":
        n = _log(rng, 1 << 13, min(1 << 20, top))
    else:
        n = _log(rng, 1 << 16, min(10000000, top))
    chirps = rng.choice([0, K, K, min(K, 100)])
    ms = rng.choice([rng.uniform(0.1, 2.0), rng.uniform(5.0, 35.0)])
    if kind == "rearrange":
        chirps, ms = min(K, rng.randint(1, 100)), rng.uniform(0.1, 2.0)
    # the cursor is at the start, or somewhere on the chirps
    c = _call(K=K, n=n, start=rng.choice([0, rng.randint(0, int(ms * 1e-3 * FS))]), chirps=chirps, ms=round(ms, 4),
              profile=rng.choice(["mixed", "mixed", "linear", "minjerk", "exponential"]), kind=kind)
    if kind == "call":
        c["f32"] = rng.random() < 0.3
        c["sine"] = rng.choice(["sfu", "sfu", "rotator"])
        c["ramps"] = rng.choice([0, 0, 0, K, K // 2])
    elif kind == "mux":
        c["channels"] = channels
    else:
        c["chunk"] = 1 << rng.randint(16, 20)
        c["start"] = 0
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _tones(case, seed):
    """Tones, chirps and ramps of one channel as numpy arrays."""
    rng = np.random.default_rng(seed)
    K = case["K"]
    w = {"f": rng.uniform(80e6, 180e6, K), "A": rng.uniform(0.5, 1.0, K) / K, "th": rng.uniform(0.0, 2.0 * math.pi, K),
         "chirps": None, "ramps": None}
    if case["kind"] == "engine":
        w["f"] = 80e6 + 1e4 * rng.choice(10000, K, replace=False)
        G = case["groups"] * case["group"]
        if G:
            # group m ramps linearly for 1 ms from sample m * 280,000 on
            L = int(round(1e-3 * FS))
            tone = np.sort(rng.choice(K, G, replace=False))
            w["chirps"] = dict(tone=tone, f0=w["f"][tone].copy(), f1=80e6 + 1e4 * rng.integers(0, 10000, G), dur=np.full(G, 1e-3),
                               profile=np.full(G, LINEAR), start=case["start"] + (np.arange(G) // case["group"]) * L)
        return w
    if case["kind"] in ("table", "replay"):
        w["f"] = 80e6 + 1e5 * 1000 / K * np.arange(K, dtype=np.float64)
        w["th"] = -math.pi * np.arange(K, dtype=np.float64) ** 2 / K + rng.uniform(0.0, 1.0, K)
        return w
    n_ch = case["chirps"]
    if n_ch:
        tone = np.sort(rng.choice(K, n_ch, replace=False))
        prof = {"mixed": np.arange(n_ch) % 2, "linear": np.full(n_ch, LINEAR), "minjerk": np.full(n_ch, MINJERK),
                "exponential": np.full(n_ch, EXPONENTIAL)}[case["profile"]]
        # chirps of a small window begin at different samples inside it
        start = case["start"] + rng.integers(0, 2000, n_ch) if case["n"] < 20000 else np.zeros(n_ch, dtype=np.int64)
        w["chirps"] = dict(tone=tone, f0=w["f"][tone].copy(), f1=rng.uniform(80e6, 180e6, n_ch), dur=np.full(n_ch, case["ms"] * 1e-3),
                           profile=prof, start=start)
    n_r = case["ramps"]
    if n_r:
        tone = np.sort(rng.choice(K, n_r, replace=False))
        w["ramps"] = dict(tone=tone, A1=np.where(np.arange(n_r) % 3 == 0, 0.0, rng.uniform(0.0, 1.0, n_r) / K),
                          dur=np.full(n_r, max(1, 3 * case["n"] // 4) / FS), profile=np.arange(n_r) % 2,
                          start=np.full(n_r, case["start"], dtype=np.int64))
    return w


def _set_chirps(s, c):
    s.set_chirps(c["tone"], c["f0"], c["f1"], c["dur"], c["profile"], c["start"])


def _synth(case, seed):
    s = awg.Synth(FS)
    w = _tones(case, seed)
    s.set_tones(w["f"], w["A"], w["th"], grid_log2=case.get("log2"))
    if w["chirps"]:
        _set_chirps(s, w["chirps"])
    if w["ramps"]:
        r = w["ramps"]
        s.set_amp_ramps(r["tone"], r["A1"], r["dur"], r["profile"], r["start"])
    if case.get("sine") == "rotator":
        s.set_sine_mode(awg.SINE_ROTATOR)
    return s, w


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "rearrange":
        st["synth"], st["w"] = awg.Synth(FS), _tones(case, seed)
        st["q"] = torch.empty(case["n"], dtype=torch.int16, pin_memory=True)
        return st
    if kind == "mux":
        st["synths"] = [_synth(case, seed * 16 + c)[0] for c in range(case["channels"])]
        st["q"] = torch.empty(case["n"] * case["channels"], dtype=torch.int16, device="cuda")
        return st
    s, _ = _synth(case, seed)
    st["synth"] = s
    if kind == "table":
        st["q"] = torch.empty(1 << case["log2"], dtype=torch.int16, device="cuda")
        st["x"] = torch.empty(1 << case["log2"], dtype=torch.float32, device="cuda")
        return st
    if kind == "engine":
        s.set_static_engine(awg.STATIC_GEMM_FP16 if case["prec"] == "fp16" else awg.STATIC_GEMM_BF16)
    if kind == "replay":
        s.set_periodic(case["log2"], awg.PERIODIC_DIRECT)
    st["q"] = torch.empty(case["n"], dtype=torch.int16, device="cuda")
    if case.get("f32"):
        st["x"] = torch.empty(case["n"], dtype=torch.float32, device="cuda")
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mux":
        for s in state["synths"]:
            s.seek(case["start"])
        awg.render_multiplexed(state["synths"], case["n"], state["q"])
        return {"q": state["q"]}
    s = state["synth"]
    if kind == "table":
        s.table_gemm(case["log2"], awg.PREC_FP16 if case["prec"] == "fp16" else awg.PREC_BF16, state["q"], state["x"])
        return {"q": state["q"], "x": state["x"]}
    s.seek(case["start"])
    if kind == "rearrange":
        w = state["w"]
        s.set_tones(w["f"], w["A"], w["th"])
        _set_chirps(s, w["chirps"])
        s.render_stream(case["n"], case["chunk"], state["q"])
    elif kind == "stream":
        s.render_stream(case["n"], case["chunk"], state["q"])
    elif case.get("f32"):
        s.render_f32(case["n"], state["x"], state["q"])
        return {"q": state["q"], "x": state["x"]}
    else:
        s.render(case["n"], state["q"])
    return {"q": state["q"]}


def work(case):
    """Tone parameters and chirps in, samples out; per tone-sample a sine, a multiply and an add."""
    ch = case.get("channels", 1)
    n = (1 << case["log2"]) if case["kind"] == "table" else case["n"]
    out = 2 * n * ch + (4 * n if case.get("f32") or case["kind"] == "table" else 0)
    if case["kind"] == "replay":   # the table is read once, the samples written
        return {"bytes": out + min(2 << case["log2"], 2 * n), "flops": 0}
    chirps = case["groups"] * case["group"] if case["kind"] == "engine" else case.get("chirps", 0)
    return {"bytes": out + ch * (24 * case["K"] + 40 * chirps + 32 * case.get("ramps", 0)), "flops": 3 * case["K"] * n * ch}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------
def _shape(profile, tau):
    """Phase of a frequency ramp by 1 over one unit of time, at time tau (its value at 1 is 1/2)."""
    return torch.where(profile == LINEAR, 0.5 * tau ** 2, tau ** 4 * (2.5 + tau * (tau - 3.0)))


def _sum64(w, start, n):
    """x[start .. start + n) in float64: phases in turns, tones in blocks."""
    dev = "cuda"
    K = len(w["f"])
    t = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=dev)  # noqa: E731
    f, A, turn = t(w["f"]) / FS, t(w["A"]), t(w["th"]) / (2 * math.pi)
    has = torch.zeros(K, dtype=torch.bool, device=dev)
    f0, f1, ns, L, prof = (torch.zeros(K, dtype=torch.float64, device=dev) for _ in range(5))
    L += 1
    if w["chirps"]:
        c = w["chirps"]
        at = torch.as_tensor(np.asarray(c["tone"], dtype=np.int64), device=dev)
        has[at] = True
        f0[at], f1[at], ns[at], prof[at] = t(c["f0"]) / FS, t(c["f1"]) / FS, t(c["start"]), t(c["profile"])
        L[at] = torch.round(t(c["dur"]) * FS)
    ramp = torch.zeros(K, dtype=torch.bool, device=dev)
    A1, rs, rL, rp = A.clone(), torch.zeros_like(A), torch.ones_like(A), torch.zeros_like(A)
    if w["ramps"]:
        r = w["ramps"]
        at = torch.as_tensor(np.asarray(r["tone"], dtype=np.int64), device=dev)
        ramp[at] = True
        A1[at], rs[at], rL[at], rp[at] = t(r["A1"]), t(r["start"]), torch.round(t(r["dur"]) * FS), t(r["profile"])
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    order = torch.argsort(has.to(torch.int8) * 2 + ramp.to(torch.int8), stable=True)
    rows, cols = 64, 1 << 17
    for j in range(0, n, cols):
        i = torch.arange(start + j, start + min(n, j + cols), dtype=torch.float64, device=dev)[None, :]
        for b in range(0, K, rows):
            k = order[b:b + rows]
            g = lambda v: v[k][:, None]  # noqa: E731
            ph = g(turn) + torch.frac(g(f) * i)
            if bool(has[k].any()):
                m = torch.minimum(torch.clamp(i - g(ns), min=0.0), g(L))
                tau = m / g(L)
                move = g(f0) * m + (g(f1) - g(f0)) * g(L) * _shape(g(prof), tau)
                if bool((prof[k] == EXPONENTIAL).any()):
                    lr = torch.log1p((g(f1) - g(f0)) / torch.where(g(f0) > 0, g(f0), 1.0))
                    e = torch.where(lr == 0, g(f0) * m, g(f0) * g(L) * torch.expm1(lr * tau) / torch.where(lr == 0, 1.0, lr))
                    move = torch.where(g(prof) == EXPONENTIAL, e, move)
                after = g(f1) * torch.clamp(i - g(ns) - g(L), min=0.0)
                ph = torch.where(g(has) & (i >= g(ns)), g(turn) + torch.frac(g(f) * g(ns)) + torch.frac(move) + torch.frac(after), ph)
            a = g(A)
            if bool(ramp[k].any()):
                tau = torch.clamp((i - g(rs)) / g(rL), 0.0, 1.0)
                s = torch.where(g(rp) == LINEAR, tau, tau ** 3 * (10.0 + tau * (6.0 * tau - 15.0)))
                a = torch.where(g(ramp), a + (g(A1) - a) * s, a)
            x[j:j + i.shape[1]] += (a * torch.sin(2 * math.pi * ph)).sum(0)
    return x


def _codes(x, full_scale):
    return torch.clamp(torch.round(x * (32767.0 / full_scale)), -32767, 32767).to(torch.int16)


def _period64(w, log2):
    """One period of tones snapped to the f_s / 2^log2 grid, by an inverse transform."""
    N = 1 << log2
    c = torch.zeros(N, dtype=torch.complex128, device="cuda")
    j = torch.as_tensor(np.rint(np.ldexp(w["f"] / FS, log2)).astype(np.int64) % N, device="cuda")
    a = torch.as_tensor(w["A"] * np.exp(1j * w["th"]), device="cuda")
    c.index_add_(0, j, a)
    return torch.fft.ifft(c).imag * N


def exact(case, seed):
    kind = case["kind"]
    if kind == "mux":
        qs = []
        for c in range(case["channels"]):
            w = _tones(case, seed * 16 + c)
            qs.append(_codes(_sum64(w, case["start"], case["n"]), float(np.abs(w["A"]).sum())))
        return {"q": torch.stack(qs, dim=1).reshape(-1)}
    w = _tones(case, seed)
    full = float(np.abs(w["A"]).sum())
    if kind == "table":
        x = _period64(w, case["log2"])
        return {"q": _codes(x, full), "x": x}
    if kind == "replay":
        tab = _codes(_period64(w, case["log2"]), full)
        i = torch.arange(case["start"], case["start"] + case["n"], device="cuda")
        return {"q": tab[i & ((1 << case["log2"]) - 1)]}
    x = _sum64(w, case["start"], case["n"])
    if case.get("f32"):
        return {"q": _codes(x, full), "x": x}
    return {"q": _codes(x, full)}
