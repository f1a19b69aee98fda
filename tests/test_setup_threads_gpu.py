"""A handful of chirps is set up on the calling thread: no slower per call than waking workers for them, next
to the time of one chirp."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


def _us(awglib, n):
    f = np.linspace(80e6, 180e6, 64)
    s = awglib.Synth(FS)
    s.set_tones(f, np.full(64, 1 / 64), np.zeros(64))
    took = []
    for _ in range(60):
        start = np.full(n, s.cursor, dtype=np.int64)
        torch.cuda.synchronize()
        time.sleep(0.002)   # the workers are asleep
        t = time.perf_counter()
        s.set_chirps(np.arange(n), f[:n], f[:n] + 1e6, np.full(n, 1e-5), np.zeros(n, dtype=np.int32), start)
        took.append(time.perf_counter() - t)
        s.seek(s.cursor + 8192)
    s.close()
    return 1e6 * min(took[10:])   # (other processes of the machine only add to a call)


def test_few_chirps(awglib):
    """Sixteen linear chirps take a few us more than one (0.4 us each); a wake-up takes 30 us and more."""
    one, sixteen = _us(awglib, 1), _us(awglib, 16)
    assert sixteen < one + 20, (one, sixteen)
