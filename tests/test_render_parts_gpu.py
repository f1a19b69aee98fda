"""The render cuts a tile's samples over 1, 2 or 4 CTAs by the size of the launch: the sums are the same
bits in every form.  A record large enough for whole tiles is rendered in one call, then again in
windows small enough for halves and quarters (ragged starts and lengths, single samples); every sample
has to match bit for bit.  The tones hold every form a tile can take: static (SFU and rotator), linear
and minimum-jerk chirps that cover the tile (shared and own set-ups, with an odd tone left over), chirp
boundaries, a per-sample phase table, amplitude ramps on static and on chirping tones, inside and at
their ends.  Windows are checked against the oracle too (bounds as in test_amp_ramps_gpu)."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NTHREADS = os.cpu_count() or 1
FS = 280e6
TILE = 4096


@pytest.fixture(scope="module")
def awg(awglib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return awglib


def _case(seed, K, span):
    rng = np.random.default_rng(seed)
    f = rng.uniform(1e6, 139e6, K)
    a = rng.uniform(0.2, 1.0, K)
    th = rng.uniform(0, 2 * np.pi, K)
    chirps, ramps = [], []
    for k in range(K):
        if k % 4 == 3:
            continue                                    # static
        if k % 8 == 0:
            L, start = int(rng.integers(60, 400)), int(rng.integers(0, 3 * TILE))      # boundary or table
        elif k % 8 == 1:
            L, start = int(rng.integers(2 * TILE, 9 * TILE)), int(rng.integers(0, 5 * TILE))
        else:
            L, start = span, 0                          # covers the record
        chirps.append(dict(tone=k, f_start=float(f[k]), f_end=float(rng.uniform(1e6, 139e6)), duration=L / FS,
                           profile=int(k // 2 % 2), start_sample=start))
    for k in range(0, K, 5):
        ramps.append(dict(tone=k, amp_end=0.0 if k % 2 else float(rng.uniform(0.1, 1.5)), profile=int(k % 2),
                          duration=float(rng.integers(40, 12 * TILE)) / FS, start_sample=int(rng.integers(0, 6 * TILE))))
    return f, a, th, chirps, ramps


def _bound(a, ramps, split):
    amax = np.abs(np.asarray(a)).copy()
    dA = np.zeros_like(amax)
    for r in ramps:
        dA[r["tone"]] = abs(r["amp_end"] - a[r["tone"]])
        amax[r["tone"]] = max(amax[r["tone"]], abs(r["amp_end"]))
    K = len(a)
    return float(np.sum(5e-6 * amax + 6e-7 * dA) + np.sum(amax) * (K / split + split + 2) * 2.0**-24)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("K,tiles", [(1, 400), (11, 400), (97, 260), (500, 90)])
def test_parts_give_the_same_bits(awg, oracle, K, tiles, mode):
    n = tiles * TILE
    f, a, th, chirps, ramps = _case(K, K, n + 5000)
    s = awg.Synth(FS)
    s.set_tones(f, a, th)
    s.set_chirp_list(chirps)
    s.set_ramp_list(ramps)
    s.set_sine_mode(mode)
    x = torch.empty(n, dtype=torch.float32, device="cuda")
    q = torch.empty(n, dtype=torch.int16, device="cuda")
    s.render_f32(n, x, q)
    w = oracle.add_ramps(oracle.make_waveform(FS, f, a, th, chirps), ramps)
    for start, m in ((0, 1), (TILE - 1, 2), (3, 5 * TILE + 1), (2 * TILE, 8 * TILE), (777, 40 * TILE), (TILE, 70 * TILE)):
        xs = torch.empty(m, dtype=torch.float32, device="cuda")
        qs = torch.empty(m, dtype=torch.int16, device="cuda")
        s.seek(start)
        s.render_f32(m, xs, qs)
        assert torch.equal(qs, q[start:start + m]), (start, m)
        assert torch.equal(xs, x[start:start + m]), (start, m)
    if mode == 0:
        m = 9 * TILE + 17
        ref = oracle.render(w, 0, m, nthreads=NTHREADS)
        assert np.max(np.abs(x[:m].cpu().numpy().astype(np.float64) - ref)) <= _bound(a, ramps, s.tone_split)
        dq = np.abs(q[:m].cpu().numpy().astype(np.int32) - oracle.quantize(ref, s.full_scale).astype(np.int32))
        assert dq.max() <= 1
    assert s.device_status() == 0
    s.close()
