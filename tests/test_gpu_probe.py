"""The throughput probes measure the pipes: this GPU has 64 times fewer FP64 than FP32 lanes, so the
two rates have that ratio at any clock."""
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _rate(B, precision, iters):
    import torch
    blocks = 152 * 16
    out = torch.empty(blocks * 256, dtype=torch.float64 if precision == 0 else torch.float32, device="cuda")
    best = 1e30
    for _ in range(4):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        B.lasto_probe_fma(precision, blocks, iters, out)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    assert bool(torch.isfinite(out).all())
    return iters / best


def test_fp64_rate_is_a_64th_of_fp32():
    B = need_gpu()
    ratio = 64 * _rate(B, 0, 100) / _rate(B, 1, 4000)
    assert 0.93 < ratio < 1.07, ratio      # (clock steps between the two: a few per cent)
