"""Windows on either side of the length from which a single render has its chirp records formed by the set-up
kernel again (many tiles, few tones per CTA): the same samples as short windows over them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6
TILE = 4096


@pytest.mark.parametrize("K,chirps,tiles", [(97, 97, 900), (100, 100, 903), (100, 100, 904), (128, 100, 1200), (128, 30, 1200), (193, 193, 1175)])
def test_long_windows(awglib, K, chirps, tiles):
    rng = np.random.default_rng(K + tiles)
    s = awglib.Synth(FS)
    f = rng.uniform(80e6, 180e6, K)
    s.set_tones(f, np.full(K, 1.0 / K), rng.uniform(0, 6.28, K))
    s.set_chirps(np.arange(chirps), f[:chirps], rng.uniform(80e6, 180e6, chirps), rng.uniform(1e-3, 20e-3, chirps),
                 np.arange(chirps) % 3, rng.integers(0, 1 << 20, chirps))
    n = tiles * TILE
    a, b = (torch.empty(n, dtype=torch.int16, device="cuda") for _ in range(2))
    s.render(n, a)
    s.seek(0)
    for at in range(0, n, 333333):
        s.render(min(333333, n - at), b[at:])
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert s.device_status() == 0
    s.close()


def test_no_memory_for_the_records(awglib):
    """A long window whose records do not fit the device forms them in the CTAs."""
    K, n = 100, 1 << 28
    rng = np.random.default_rng(3)
    s = awglib.Synth(FS)
    f = rng.uniform(80e6, 180e6, K)
    s.set_tones(f, np.full(K, 1.0 / K), rng.uniform(0, 6.28, K))
    s.set_chirps(np.arange(K), f, rng.uniform(80e6, 180e6, K), np.full(K, 0.9), np.arange(K) % 2, np.zeros(K, dtype=np.int64))
    out, want = torch.empty(n, dtype=torch.int16, device="cuda"), torch.empty(1 << 20, dtype=torch.int16, device="cuda")
    s.render(1 << 20, want)
    s.seek(0)
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")   # records: 1.15 GB
    try:
        s.render(n, out)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(out[:1 << 20], want)
    s.seek(n - (1 << 20))
    s.render(1 << 20, want)
    torch.cuda.synchronize()
    assert torch.equal(out[n - (1 << 20):], want)
    assert s.device_status() == 0
    s.close()
