"""The tensor-core engine's A operand at the edges of its tiles: tone counts around the 16 tones of a
stage, chirps and amplitude ramps that begin and end at a 4096-sample tile boundary and one sample
beside it, windows that start inside a tile (rows not aligned to a tile) and inside a row of 256
samples, and tiles of 128 rows that hold every combination of segments.

FP32 bound, in LSB of the full scale sum max|A|: per unit amplitude 5e-6 for the tones the render
sums, and for the GEMM 2 x 2^-22 (FP16 hi + lo residual of both operands), 4.6e-7 and 5e-8 (operand
sines), 1e-6 for the FP32 accumulation of up to 4 x 40 columns; together below 7e-6, 0.23 LSB."""
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


@pytest.mark.parametrize("K", [1, 15, 16, 17, 40])
@pytest.mark.parametrize("start", [0, 256 * 3 + 5, 37 * TILE + 256 * 7])
def test_segments_at_tile_edges(awg, oracle, K, start):
    rng = np.random.default_rng(100 * K + start)
    f = rng.uniform(1e6, 139e6, K)
    a = rng.uniform(0.2, 1.0, K)
    th = rng.uniform(0, 2 * np.pi, K)
    t0 = start // TILE
    chirps, ramps = [], []
    for k in range(K):
        edge = (t0 + 2 + k % 5) * TILE + (k % 3) - 1
        if k % 4 < 2:
            L = (1 + k % 7) * TILE + (k // 4 % 3) - 1
            chirps.append(dict(tone=k, f_start=float(f[k]), f_end=float(rng.uniform(1e6, 139e6)), duration=L / FS,
                               profile=k % 2, start_sample=edge))
        if k % 5 < 2:
            ramps.append(dict(tone=k, amp_end=float(rng.uniform(0, 1)), duration=(TILE * (1 + k % 3) + k % 2) / FS,
                              profile=k % 2, start_sample=(t0 + 1 + k % 6) * TILE + (k // 5 % 3) - 1))
    n = 150 * TILE + 77 if K == 17 else 20 * TILE + 77
    s = awg.Synth(FS)
    s.set_tones(f, a, th)
    if start:
        s.seek(0)
    s.set_chirp_list(chirps)
    s.set_ramp_list(ramps)
    amax = np.abs(a).copy()
    for r in ramps:
        amax[r["tone"]] = max(amax[r["tone"]], r["amp_end"])
    full = float(np.sum(amax))
    s.set_full_scale(full)
    s.set_static_engine(awg.STATIC_GEMM_FP16)
    x = torch.empty(n, dtype=torch.float32, device="cuda")
    q = torch.empty(n, dtype=torch.int16, device="cuda")
    s.seek(start)
    s.render_f32(n, x, q)
    torch.cuda.synchronize()
    assert s.device_status() == 0
    w = oracle.add_ramps(oracle.make_waveform(FS, f, a, th, chirps), ramps)
    ref = oracle.render(w, start, n, nthreads=NTHREADS)
    err = float(np.max(np.abs(x.cpu().numpy().astype(np.float64) - ref))) / (full / 32767.0)
    assert err <= 0.23, err
    dq = np.abs(q.cpu().numpy().astype(np.int32) - oracle.quantize(ref, full).astype(np.int32))
    assert dq.max() <= 1
    s.close()


@pytest.mark.parametrize("K,groups,aligned", [(600, 10, True), (600, 10, False), (97, 3, True), (3000, 40, False)])
def test_groups_that_chirp_in_turn(awg, oracle, K, groups, aligned):
    """Groups of interleaved tones (tone k in group k mod groups) that chirp for about two tiles in turn:
    the tile's live tones are spread over the list, their records over the window's; also into an
    unaligned buffer and as two interleaved channels."""
    rng = np.random.default_rng(K)
    f = rng.uniform(1e6, 139e6, K)
    a = rng.uniform(0.2, 1.0, K)
    th = rng.uniform(0, 2 * np.pi, K)
    L = 2 * TILE - 100
    chirps = [dict(tone=k, f_start=float(f[k]), f_end=float(rng.uniform(1e6, 139e6)), duration=L / FS, profile=k % 2,
                   start_sample=1000 + (k % groups) * L) for k in range(K) if k % 7]
    n = 1000 + groups * L + 3 * TILE + 5
    handles = []
    for _ in range(2):
        s = awg.Synth(FS)
        s.set_tones(f, a, th)
        s.set_chirp_list(chirps)
        s.set_static_engine(awg.STATIC_GEMM_FP16)
        handles.append(s)
    s = handles[0]
    off = 0 if aligned else 3
    q = torch.zeros(n + 8, dtype=torch.int16, device="cuda")
    x = torch.zeros(n + 8, dtype=torch.float32, device="cuda")
    s.render_f32(n, x[off:], q[off:])
    w = oracle.make_waveform(FS, f, a, th, chirps)
    ref = oracle.render(w, 0, n, nthreads=NTHREADS)
    err = float(np.max(np.abs(x[off:off + n].cpu().numpy().astype(np.float64) - ref))) / (s.full_scale / 32767.0)
    assert err <= 0.23, err
    dq = np.abs(q[off:off + n].cpu().numpy().astype(np.int32) - oracle.quantize(ref, s.full_scale).astype(np.int32))
    assert dq.max() <= 1
    both = torch.zeros(2 * n, dtype=torch.int16, device="cuda")
    for h in handles:
        h.seek(0)
    awg.render_multiplexed(handles, n, both)
    torch.cuda.synchronize()
    for c in range(2):
        assert torch.equal(both[c::2], q[off:off + n])
    for h in handles:
        assert h.device_status() == 0
        h.close()


def test_first_call_of_a_handle_on_used_memory(awg):
    """The split sums' counters are zero before the engine's side stream counts on them, also when the
    memory held another split's counts and the caller's stream is busy."""
    K, n = 700, 12000
    rng = np.random.default_rng(5)
    f, th = rng.uniform(80e6, 180e6, K), rng.uniform(0, 6.28, K)
    busy = torch.empty(1 << 28, dtype=torch.float32, device="cuda")
    for split_tones in (480, 200, 900):
        old = awg.Synth(280e6)
        old.set_tones(f[:split_tones] if split_tones < K else np.resize(f, split_tones), np.full(split_tones, 1e-3), np.zeros(split_tones))
        x = torch.empty(n, dtype=torch.float32, device="cuda")
        old.render_f32(n, x)
        torch.cuda.synchronize()
        old.close()
        s = awg.Synth(280e6)
        s.set_tones(f, np.full(K, 1.0 / K), th)
        s.set_amp_ramps(np.arange(K), np.zeros(K), np.full(K, 1e-5), np.arange(K) % 2, rng.integers(0, n, K))
        s.set_static_engine(awg.STATIC_GEMM_FP16)
        first, again = torch.empty_like(x), torch.empty_like(x)
        for _ in range(8):
            busy.zero_()
        s.render_f32(n, first)
        torch.cuda.synchronize()
        s.seek(0)
        s.render_f32(n, again)
        torch.cuda.synchronize()
        assert torch.equal(first, again)
        s.close()
