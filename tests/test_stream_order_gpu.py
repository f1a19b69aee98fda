"""Calls issued back to back on one stream start while the one before still runs; what they write has to
be what synchronised calls write.  Random sequences of renders of several handles (chirping, static,
ramping, rotator, tensor-core engine, periodic hand-off, multiplexed, allocation-free, chunk sequences)
into one shared buffer, with copies and fills of that buffer between them, on the default and on another
stream, against the same sequence with a synchronisation after every call."""
import random

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6
N = 200001


@pytest.fixture(scope="module")
def handles(awglib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")

    def make(K, n_chirps, seed, ramps=0, mode=0, engine=0):
        r = np.random.default_rng(seed)
        s = awglib.Synth(FS)
        f = r.uniform(1e6, 139e6, K)
        s.set_tones(f, r.uniform(0.2, 1.0, K), r.uniform(0, 6, K))
        if n_chirps:
            s.set_chirps(np.arange(n_chirps), f[:n_chirps], r.uniform(1e6, 139e6, n_chirps), np.full(n_chirps, 2e-3),
                         np.arange(n_chirps) % 2, np.zeros(n_chirps, dtype=np.int64))
        if ramps:
            s.set_amp_ramps(np.arange(ramps), r.uniform(0, 1, ramps), np.full(ramps, 1e-3), np.arange(ramps) % 2,
                            np.zeros(ramps, dtype=np.int64))
        s.set_sine_mode(mode)
        s.set_static_engine(engine)
        return s

    hs = [make(5, 2, 1), make(100, 0, 2), make(300, 300, 3), make(700, 100, 4, ramps=50), make(150, 0, 5, mode=1),
          make(900, 20, 6, engine=1)]
    p = awglib.Synth(FS)
    p.set_tones(80e6 + 1e5 * np.arange(300), np.full(300, 1 / 300), np.arange(300.0), grid_log2=16)
    p.set_periodic(16, awglib.PERIODIC_DIRECT)
    return hs + [p]


def _run(awglib, hs, ops, stream, sync):
    outs = []
    with torch.cuda.stream(stream):
        buf = torch.zeros(3 * N, dtype=torch.int16, device="cuda")
        x = torch.zeros(N, dtype=torch.float32, device="cuda")
        for k, n, start, how, fill in ops:
            h = hs[k]
            h.seek(start)
            if how == "stream":
                h.render_stream(n, 1 << 15, buf)
            elif how == "f32":
                h.render_f32(n, x, buf)
            elif how == "noalloc":
                h.render_noalloc(n, buf)
            elif how == "mux":
                chs = [h, hs[(k + 1) % len(hs)], hs[(k + 2) % len(hs)]]
                for c in chs[1:]:
                    c.seek(start)
                awglib.render_multiplexed(chs, n, buf)
            else:
                h.render(n, buf)
            if sync:
                torch.cuda.synchronize()
            outs.append(buf.clone())
            if how == "f32":
                outs.append(x.clone())
            if fill:
                buf.zero_()
    torch.cuda.synchronize()
    return outs


@pytest.mark.parametrize("seed", range(4))
def test_unsynchronised_calls_write_the_same(awglib, handles, seed):
    rng = random.Random(seed)
    ops = [(rng.randrange(len(handles)), rng.choice([100, 5000, 70000, N]), rng.randrange(400000),
            rng.choice(["render", "render", "stream", "f32", "noalloc", "mux"]), rng.random() < 0.3) for _ in range(40)]
    ref = _run(awglib, handles, ops, torch.cuda.current_stream(), True)
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        got = _run(awglib, handles, ops, stream, False)
        for i, (a, b) in enumerate(zip(ref, got)):
            assert torch.equal(a, b), (i, ops)
    for h in handles:
        assert h.device_status() == 0
        assert 0 < h.last_render_ms() < 1000


def test_new_tones_and_chirps_behind_renders(awglib):
    """set_tones and set_chirps queue their uploads behind the renders issued so far: one handle that is
    given new tones, scattered chirps (few and many, short ones with phase tables too) and fewer or more
    tones again, without a synchronisation, against a fresh handle for every round."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 60001
    one = awglib.Synth(FS)
    got, want = [], []
    for rnd, K in enumerate([40, 700, 700, 30, 0, 650, 700, 1, 2000, 1900]):
        r = np.random.default_rng(rnd)
        f, a, th = r.uniform(1e6, 139e6, K), r.uniform(0.2, 1, K), r.uniform(0, 6, K)
        nc = [K // 2, 3, K // 7, K, 0, 100, 5, 1, 40, 1900][rnd]
        t = np.sort(r.choice(K, nc, replace=False)) if nc else np.zeros(0, dtype=int)
        dur = np.where(np.arange(nc) % 4 == 0, 3e-7, 1.5e-4)
        args = (t, f[t], r.uniform(1e6, 139e6, nc), dur, np.arange(nc) % 2, r.integers(0, 20000, nc))
        fresh = awglib.Synth(FS)
        for s, outs in ((one, got), (fresh, want)):
            s.seek(0)
            s.set_tones(f, a, th)
            if nc:
                s.set_chirps(*args)
            out = torch.empty(n, dtype=torch.int16, device="cuda")
            s.render(n, out)
            outs.append(out)
            out = torch.empty(n, dtype=torch.int16, device="cuda")
            s.seek(0)
            s.render_stream(n, 7000, out)
            outs.append(out)
        torch.cuda.synchronize() if rnd % 4 == 3 else None
        fresh.device_status() if rnd % 5 == 4 else None
    torch.cuda.synchronize()
    for i, (x, y) in enumerate(zip(got, want)):
        assert torch.equal(x, y), i
    assert one.device_status() == 0
