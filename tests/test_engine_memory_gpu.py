"""The tensor-core engine in little device memory: it renders in shorter pieces, the same samples."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 280e6


@pytest.mark.parametrize("left_mb", [400, 150])
def test_sums_that_do_not_fit(awglib, left_mb):
    K, n = 64, 1 << 26   # two FP32 sums of 256 MiB
    f = np.linspace(80e6, 180e6, K)

    def make():
        s = awglib.Synth(FS)
        s.set_tones(f, np.full(K, 1.0 / K), np.zeros(K))
        s.set_chirps(np.arange(5), f[:5], f[:5] + 1e6, np.full(5, 0.1), np.arange(5) % 2, np.arange(5) * 100000)
        s.set_static_engine(awglib.STATIC_GEMM_FP16)
        return s

    want, out = (torch.empty(n, dtype=torch.int16, device="cuda") for _ in range(2))
    s = make()
    s.render(n, want)
    torch.cuda.synchronize()
    s.close()
    s = make()
    s.render(1000, out)   # the handle's small buffers
    s.seek(0)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (left_mb << 20), dtype=torch.uint8, device="cuda")
    try:
        s.render(n, out)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert s.device_status() == 0
    assert torch.equal(out, want)
    s.close()
