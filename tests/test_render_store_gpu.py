"""The stores of a render: outputs off the 16-byte alignment, windows that start and end inside a tile,
FP32 sums with and without the codes.  The same samples, bit for bit, as an aligned render of whole tiles,
and nothing outside the window."""
import numpy as np
import pytest
import torch

import paper_2403_15582_gb300 as awg

pytestmark = pytest.mark.gpu
TILE = 4096


# one CTA per part (40 tones) and three (250); chirps: the CTA forms its records; rotator: whole tiles
@pytest.mark.parametrize("K,chirps,sine", [(40, 0, awg.SINE_SFU), (40, 40, awg.SINE_SFU), (250, 0, awg.SINE_SFU),
                                           (250, 9, awg.SINE_SFU), (250, 0, awg.SINE_ROTATOR)])
# tiles: quarters of a tile, halves and whole tiles
@pytest.mark.parametrize("tiles", [2, 60, 700])
def test_unaligned_windows(K, chirps, sine, tiles):
    rng = np.random.default_rng(K + tiles)
    s = awg.Synth(280e6)
    f = rng.uniform(80e6, 180e6, K)
    s.set_tones(f, rng.uniform(0.1, 1.0, K) / K, rng.uniform(0, 6.28, K))
    if chirps:
        s.set_chirps(np.arange(chirps), f[:chirps], rng.uniform(80e6, 180e6, chirps), np.full(chirps, 1e-3),
                     np.arange(chirps) % 2, np.full(chirps, 10))
    s.set_sine_mode(sine)
    total = tiles * TILE
    x0 = torch.empty(total, dtype=torch.float32, device="cuda")
    q0 = torch.empty(total, dtype=torch.int16, device="cuda")
    s.seek(0)
    s.render_f32(total, x0, q0)
    for start, n, off in [(0, total, 1), (1, total - 1, 0), (5, total - 9, 3), (TILE - 1, total - TILE + 1, 7), (TILE, total - TILE, 8),
                          (8, 1, 0), (TILE - 1, 2, 5), (12, total - 24, 4)]:
        x = torch.full((total + 16,), 3.0, dtype=torch.float32, device="cuda")
        q = torch.full((total + 16,), 77, dtype=torch.int16, device="cuda")
        q1 = q.clone()
        x1 = x.clone()
        s.seek(start)
        s.render_f32(n, x[off:], q[off:])
        s.seek(start)
        s.render(n, q1[off:])
        s.seek(start)
        s.render_f32(n, x1[off:])
        for got, want, rest in ((x, x0, 3.0), (x1, x0, 3.0), (q, q0, 77), (q1, q0, 77)):
            assert torch.equal(got[off:off + n], want[start:start + n])
            assert bool((got[:off] == rest).all()) and bool((got[off + n:] == rest).all())
