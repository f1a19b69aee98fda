"""Renders that form their chirp records in the CTA (at most 96 tones per CTA, chirps in the window) against
renders that take them from the set-up kernel (the allocation-free render, chunk sequences): the same
bits.  Tone counts around one and sixteen full CTAs, all chirp profiles, chirps that cover the window in
every form (linear, LOW3, LOW6, FLAT3, general), boundaries, tables, ramps over chirps, windows inside a
tile and over many tiles; samples against the oracle within 1 LSB."""
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


@pytest.mark.parametrize("K", [1, 2, 95, 96, 97, 193, 1535, 1536, 1537])
def test_same_bits_as_the_set_up_kernel(awg, oracle, K):
    rng = np.random.default_rng(K)
    f = rng.uniform(1e6, 139e6, K)
    a = rng.uniform(0.2, 1.0, K)
    th = rng.uniform(0, 2 * np.pi, K)
    lengths = [100, 3000, 9 * TILE, 30 * TILE, 200 * TILE, 2000 * TILE]
    chirps = [dict(tone=k, f_start=float(f[k]), f_end=float(rng.uniform(1e6, 139e6)), duration=lengths[k % 6] / FS,
                   profile=k % 3, start_sample=int(rng.integers(0, 3 * TILE))) for k in range(K) if k % 5 != 4]
    ramps = [dict(tone=k, amp_end=float(rng.uniform(0, 1)), duration=2.5 * TILE / FS, profile=k % 2,
                  start_sample=int(rng.integers(0, 4 * TILE))) for k in range(0, K, 7)]
    s = awg.Synth(FS)
    s.set_tones(f, a, th)
    s.set_chirp_list(chirps)
    s.set_ramp_list(ramps)
    for start, n in ((0, 12 * TILE + 3), (TILE + 77, 1), (5000, 3000), (2 * TILE, 25 * TILE)):
        got = torch.zeros(n, dtype=torch.int16, device="cuda")
        ref = torch.zeros(n, dtype=torch.int16, device="cuda")
        s.seek(start)
        s.render(n, got)
        s.seek(start)
        s.render_stream(n, max(1, n // 2), ref)
        assert torch.equal(got, ref), (start, n)
        if K <= 193:
            s.seek(start)
            s.render_noalloc(n, ref)
            assert torch.equal(got, ref), (start, n)
    assert s.device_status() == 0
    w = oracle.add_ramps(oracle.make_waveform(FS, f, a, th, chirps), ramps)
    idx = np.unique(rng.integers(2 * TILE, 27 * TILE, 300))
    q_ref = oracle.quantize(oracle.render_at(w, idx, nthreads=NTHREADS), s.full_scale)
    assert np.max(np.abs(got.cpu().numpy()[idx - 2 * TILE].astype(np.int32) - q_ref)) <= 1
    s.close()
