"""With the tensor-core engine and every tone chirping or ramping, a sample does not depend on how the
stream is cut into calls: a long window, in which every tone is live somewhere, against short ones over the
same samples, in which only some are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6
TILE = 4096


@pytest.mark.parametrize("K,ramps", [(33, False), (100, True), (700, False)])
def test_every_tone_chirps(awglib, K, ramps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(K)
    f = rng.uniform(80e6, 180e6, K)
    s = awglib.Synth(FS)
    s.set_tones(f, rng.uniform(0.2, 1.0, K), rng.uniform(0, 2 * np.pi, K))
    # linear, minimum-jerk and exponential chirps of 50 to 120 tiles that begin one after another in
    # the first 40 tiles: some live at first, all in tiles 40 to 50, some again after that
    start = rng.permutation(K) * (40 * TILE // K)
    dur = rng.integers(50 * TILE, 120 * TILE, K) / FS
    s.set_chirps(np.arange(K), f, rng.uniform(80e6, 180e6, K), dur, np.arange(K) % 3, start)
    if ramps:
        r = np.arange(0, K, 3)
        s.set_amp_ramps(r, rng.uniform(0, 1, len(r)), np.full(len(r), 7 * TILE / FS), np.arange(len(r)) % 2,
                        rng.integers(0, 40 * TILE, len(r)))
    s.set_static_engine(awglib.STATIC_GEMM_FP16)
    n = 80 * TILE + 99
    x, y = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    q, p = (torch.empty(n, dtype=torch.int16, device="cuda") for _ in range(2))
    s.render_f32(n, x, q)
    s.seek(0)
    at = 0
    while at < n:
        m = int(min(n - at, rng.integers(1, 4 * TILE)))
        s.render_f32(m, y[at:], p[at:])
        at += m
    torch.cuda.synchronize()
    assert s.device_status() == 0
    assert torch.equal(x, y)
    assert torch.equal(q, p)
    s.close()
