"""awg_last_render_ms spans a call from its first kernel to its last, against CUDA events around the call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


def _times(s, call):
    """(last_render_ms, event time) of the second of two calls, the device idle before each."""
    for _ in range(2):
        s.seek(0)
        torch.cuda.synchronize()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
    assert s.device_status() == 0
    return s.last_render_ms(), a.elapsed_time(b)


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
