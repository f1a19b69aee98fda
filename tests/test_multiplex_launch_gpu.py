"""Multiplexed channels share their launches: every channel's samples are those of its own render, bit
for bit, whatever the other channels are (no tones, more tones than a CTA forms records for, the
rotator sine, ramps, another cursor, another tile count, windows of several launches)."""
import numpy as np
import pytest
import torch

import paper_2403_15582_gb300 as awg

pytestmark = pytest.mark.gpu
FS = 280e6


def _channel(K, chirps, ramps, sine, seed):
    rng = np.random.default_rng(seed)
    s = awg.Synth(FS)
    f = rng.uniform(80e6, 180e6, K)
    s.set_tones(f, rng.uniform(0.1, 1.0, K) / max(K, 1), rng.uniform(0, 6.28, K))
    if chirps:
        s.set_chirps(np.arange(chirps), f[:chirps], rng.uniform(80e6, 180e6, chirps), np.full(chirps, 1e-4),
                     np.arange(chirps) % 3, rng.integers(0, 9000, chirps))
    if ramps:
        s.set_amp_ramps(np.arange(ramps), rng.uniform(0, 1, ramps) / K, np.full(ramps, 3e-5), np.arange(ramps) % 2,
                        rng.integers(0, 9000, ramps))
    s.set_sine_mode(sine)
    return s


# (tones, chirps, ramps, sine) of each channel
ONCE = [(250, 250, 0, awg.SINE_SFU), (0, 0, 0, awg.SINE_SFU), (97, 97, 40, awg.SINE_SFU)]
STATIC = [(1, 0, 0, awg.SINE_SFU), (777, 0, 300, awg.SINE_SFU)]
ROTATOR = [(33, 5, 0, awg.SINE_SFU), (300, 0, 0, awg.SINE_ROTATOR)]
SETUP = [(1537, 1537, 0, awg.SINE_SFU), (20, 0, 0, awg.SINE_SFU), (200, 200, 7, awg.SINE_SFU)]
EIGHT = [(k, k // 2, 0, awg.SINE_SFU) for k in range(1, 65, 8)]


@pytest.mark.parametrize("offsets", [0, 4095])
@pytest.mark.parametrize("n", [1, 4096, 4097, 50001])
@pytest.mark.parametrize("channels", [ONCE, STATIC, ROTATOR, SETUP, EIGHT], ids=["once", "static", "rotator", "setup", "eight"])
def test_channels_equal_their_own_renders(channels, n, offsets):
    _compare(channels, n, offsets)


@pytest.mark.parametrize("channels", [[(20, 20, 0, awg.SINE_SFU), (200, 3, 0, awg.SINE_SFU)], [(1537, 4, 0, awg.SINE_SFU), (5, 0, 0, awg.SINE_SFU)]],
                         ids=["once", "setup"])
def test_windows_of_several_launches(channels):
    _compare(channels, (1 << 21) + 5000, 4095)


def _compare(channels, n, offsets):
    synths = [_channel(*c, seed=i) for i, c in enumerate(channels)]
    start = [100 + offsets * (i % 2) for i in range(len(channels))]
    out = torch.full((n * len(channels),), 77, dtype=torch.int16, device="cuda")
    q = torch.empty(n, dtype=torch.int16, device="cuda")
    for _ in range(2):   # again on the same scratch
        for s, c in zip(synths, start):
            s.seek(c)
        awg.render_multiplexed(synths, n, out)
    assert [s.cursor for s in synths] == [c + n for c in start]
    for i, s in enumerate(synths):
        s.seek(start[i])
        s.render(n, q)
        assert torch.equal(out[i::len(channels)], q), i
        assert s.device_status() == 0
