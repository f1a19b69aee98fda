"""The tensor-core engine renders a call's chirping tones on a stream of its own beside the GEMM; that stream
has the caller's priority, so a call on a high-priority stream does not queue behind other work."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


def test_high_priority_call_passes_other_work(awglib):
    K, n = 600, 1 << 16
    f = np.linspace(80e6, 180e6, K)
    s = awglib.Synth(FS)
    s.set_tones(f, np.full(K, 1.0 / K), np.zeros(K))
    s.set_chirps(np.arange(50), f[:50], f[:50] + 1e6, np.full(50, 5e-3), np.zeros(50, dtype=np.int64), np.zeros(50, dtype=np.int64))
    s.set_static_engine(awglib.STATIC_GEMM_FP16)
    out, want = (torch.empty(n, dtype=torch.int16, device="cuda") for _ in range(2))
    low, high = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)
    # one kernel of tens of ms, of many more blocks than the device holds
    work = torch.full((1 << 26,), 5.0, dtype=torch.float64, device="cuda")
    result = torch.empty_like(work)

    def events(k):
        return [torch.cuda.Event(enable_timing=True) for _ in range(k)]

    s.render(n, want, stream=low)   # the engine's stream exists, at the other priority
    torch.cuda.synchronize()
    for _ in range(2):
        s.seek(0)
        w0, w1, r0, r1 = events(4)
        with torch.cuda.stream(low):
            w0.record()
            torch.special.gammainc(work, work, out=result)
            w1.record()
        r0.record(high)
        s.render(n, out, stream=high)
        r1.record(high)
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    assert s.device_status() == 0
    assert r0.elapsed_time(r1) < 0.25 * w0.elapsed_time(w1)
    # and back at the default priority
    s.seek(0)
    out.zero_()
    torch.cuda.synchronize()
    s.render(n, out, stream=low)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    s.close()
