"""What a set-up call uploads synchronously (the first tones, a larger chirp pool, amplitude ramps) is on the
device before the next render reads it, on a stream that waits for nothing else."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


@pytest.mark.parametrize("K", [100, 1000, 20000])
def test_render_right_after_setup(awglib, K):
    rng = np.random.default_rng(K)
    f = rng.uniform(80e6, 180e6, K)
    th = rng.uniform(0, 6.28, K)
    ns = np.zeros(K, dtype=np.int64)
    n = 20000
    stream = torch.cuda.Stream()

    def steps(s, after):
        s.set_tones(f, np.full(K, 1.0 / K), th)
        after()
        s.set_chirps(np.arange(K), f, f[::-1].copy(), np.full(K, 1e-3), np.arange(K) % 2, ns)
        after()
        s.set_amp_ramps(np.arange(0, K, 2), np.zeros((K + 1) // 2), np.full((K + 1) // 2, 5e-5), np.arange(0, K, 2) % 2,
                        ns[:(K + 1) // 2] + s.cursor)
        after()

    got, want = [], []
    s = awglib.Synth(FS)

    def at_once():
        out = torch.empty(n, dtype=torch.int16, device="cuda")
        stream.wait_stream(torch.cuda.current_stream())
        s.seek(0)
        s.render(n, out, stream=stream)
        got.append(out)
        s.seek(0)

    def settled():
        torch.cuda.synchronize()
        out = torch.empty(n, dtype=torch.int16, device="cuda")
        s.seek(0)
        s.render(n, out)
        torch.cuda.synchronize()
        want.append(out)
        s.seek(0)

    steps(s, at_once)
    torch.cuda.synchronize()
    assert s.device_status() == 0
    s.close()
    s = awglib.Synth(FS)
    steps(s, settled)
    assert s.device_status() == 0
    s.close()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
