"""The periodic replay against the table it copies, sample by sample: cursors at every offset from a
16-byte vector, outputs at every alignment, lengths below one vector up to many periods (repeats beyond
one thread's share), nothing written outside, and interleaved channels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


@pytest.fixture(scope="module")
def awg(awglib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return awglib


def _handle(awg, log2, seed=0):
    rng = np.random.default_rng(seed)
    s = awg.Synth(FS)
    s.set_tones(rng.uniform(1e6, 139e6, 20), rng.uniform(0.1, 1, 20), rng.uniform(0, 6, 20), grid_log2=log2)
    N = 1 << log2
    table = torch.empty(N, dtype=torch.int16, device="cuda")
    s.render(N, table)      # rendered: one period of the static state
    s.seek(0)
    s.set_periodic(log2, awg.PERIODIC_DIRECT)
    return s, table


@pytest.mark.parametrize("log2", [12, 15])
@pytest.mark.parametrize("shift", range(8))
def test_replay_copies_the_table(awg, log2, shift):
    s, table = _handle(awg, log2)
    N = 1 << log2
    for n in (1, 7, 8, 9, 15, 16, 17, 4095, N - 1, N, N + 9, 9 * N + 13, 21 * N + 5):
        for off in (0, 1, 3, 7):
            start = 3 * N - 8 + shift
            out = torch.full((n + 24,), 12345, dtype=torch.int16, device="cuda")
            s.seek(start)
            s.render(n, out[8 + off:])
            idx = (start + torch.arange(n, device="cuda")) % N
            assert torch.equal(out[8 + off:8 + off + n], table[idx]), (n, off)
            assert bool((out[:8 + off] == 12345).all()) and bool((out[8 + off + n:] == 12345).all()), (n, off)
    s.close()


def test_replay_of_interleaved_channels(awg):
    a, ta = _handle(awg, 13, 1)
    b, tb = _handle(awg, 13, 2)
    n = 50001
    out = torch.zeros(2 * n, dtype=torch.int16, device="cuda")
    for h in (a, b):
        h.seek(777)
    awg.render_multiplexed([a, b], n, out)
    idx = (777 + torch.arange(n, device="cuda")) % (1 << 13)
    assert torch.equal(out[0::2], ta[idx]) and torch.equal(out[1::2], tb[idx])
