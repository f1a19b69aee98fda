"""Setting many tones again holds no pinned copy of them: pinned memory shows in the process's shared pages."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _shared_mb():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) for line in f if line.startswith("RssShmem")) / 1024


@pytest.mark.parametrize("K", [170000, 180000, 1000000])
def test_pinned_memory_is_bounded(awglib, K):
    torch.cuda.init()
    s = awglib.Synth(280e6)
    f, A, th = np.linspace(80e6, 130e6, K), np.full(K, 1.0 / K), np.linspace(0, 6, K)
    out = torch.empty(1000, dtype=torch.int16, device="cuda")
    s.set_tones(f, A, np.zeros(K))
    s.render(1000, out)
    torch.cuda.synchronize()
    before = _shared_mb()
    for k in range(3):   # behind renders still under way
        s.set_tones(f, A, th)
        s.seek(0)
        s.render(1000, out)
    torch.cuda.synchronize()
    assert _shared_mb() - before < 24
    fresh, want = awglib.Synth(280e6), torch.empty_like(out)
    fresh.set_tones(f, A, th)
    fresh.render(1000, want)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    for h in (s, fresh):
        assert h.device_status() == 0
        h.close()
