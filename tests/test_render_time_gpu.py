"""awg_last_render_ms spans a call from its first kernel to its last, against CUDA events around the call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


def _times(s, call):
    """(last_render_ms, event time) of the shortest of several calls, the device idle before each (a host that is
    held up between the first event and the call only adds to the latter)."""
    took = []
    for _ in range(6):
        s.seek(0)
        torch.cuda.synchronize()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        took.append((a.elapsed_time(b), s.last_render_ms()))
    assert s.device_status() == 0
    ev, ms = min(took)
    return ms, ev


def _grid_synth(awglib, K, log2):
    s = awglib.Synth(FS)
    s.set_tones(80e6 + 1e5 * np.arange(K), np.full(K, 1.0 / K), np.arange(float(K)), grid_log2=log2)
    return s


def test_replay_of_many_periods(awglib):
    s = _grid_synth(awglib, 50, 12)
    s.set_periodic(12, awglib.PERIODIC_DIRECT)
    n = 1 << 28
    out = torch.empty(n, dtype=torch.int16, device="cuda")
    ms, ev = _times(s, lambda: s.render(n, out))
    assert 0.7 * ev < ms < 1.1 * ev, (ms, ev)
    s.close()


def test_hand_off(awglib):
    """The rendered part before the periodic one counts."""
    s = _grid_synth(awglib, 1000, 16)
    f = FS / 65536 * (20000 + np.arange(1000))
    s.set_tones(f, np.full(1000, 1e-3), np.zeros(1000), grid_log2=16)
    s.set_chirps(np.arange(1000), f, f[::-1].copy(), np.full(1000, 5e-3), np.arange(1000) % 2, np.zeros(1000, dtype=np.int64))
    s.set_periodic(16, awglib.PERIODIC_DIRECT)
    n = s.periodic_start + 5000
    out = torch.empty(n, dtype=torch.int16, device="cuda")
    for call in (lambda: s.render(n, out), lambda: s.render_stream(n, 1 << 18, out), lambda: s.render_chunks(n // 5, 5, out)):
        ms, ev = _times(s, call)
        assert 0.7 * ev < ms < 1.1 * ev, (ms, ev)
    s.close()


@pytest.mark.parametrize("K,chirps,chunk", [(1000, 1000, 1 << 18), (60, 0, 1 << 16), (2000, 100, 1 << 17)])
def test_sequence(awglib, K, chirps, chunk):
    s = awglib.Synth(FS)
    f = np.linspace(80e6, 180e6, K)
    s.set_tones(f, np.full(K, 1.0 / K), np.zeros(K))
    if chirps:
        s.set_chirps(np.arange(chirps), f[:chirps], f[:chirps] + 1e6, np.full(chirps, 5e-3), np.zeros(chirps, dtype=np.int64),
                     np.zeros(chirps, dtype=np.int64))
    n = 12 * chunk + 777
    out = torch.empty(n, dtype=torch.int16, device="cuda")
    ms, ev = _times(s, lambda: s.render_stream(n, chunk, out))
    assert 0.6 * ev < ms < 1.1 * ev, (ms, ev)
    s.close()


@pytest.mark.parametrize("chirps", [0, 20])
def test_engine_pieces(awglib, chirps):
    """A window of more samples than the engine takes at a time."""
    K = 64
    f = np.linspace(80e6, 180e6, K)
    s = awglib.Synth(FS)
    s.set_tones(f, np.full(K, 1.0 / K), np.zeros(K))
    if chirps:
        s.set_chirps(np.arange(chirps), f[:chirps], f[:chirps] + 1e6, np.full(chirps, 1e-3), np.zeros(chirps, dtype=np.int64),
                     np.zeros(chirps, dtype=np.int64))
    s.set_static_engine(awglib.STATIC_GEMM_FP16)
    n = (1 << 26) + 5000
    out = torch.empty(n, dtype=torch.int16, device="cuda")
    ms, ev = _times(s, lambda: s.render(n, out))
    assert 0.7 * ev < ms < 1.1 * ev, (ms, ev)
    s.close()
