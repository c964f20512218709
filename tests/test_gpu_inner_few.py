"""The radial solve of few atoms (a block per harmonic) and of more (five harmonics per block): the
same values bit for bit, on both sides of the line."""
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rad", [5, 64, 429, 4096])
def test_both_forms(n_rad):
    import torch
    B = need_gpu()
    g = torch.Generator(device="cuda").manual_seed(n_rad)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    R, Z, rho, v = 1.0 + rand(41), 50 * rand(41), rand(41, 25, n_rad), rand(41, 25)
    many = B.lasto_op_inner_solve(R, Z, rho, v)
    for na in (1, 40):
        few = B.lasto_op_inner_solve(R[:na].contiguous(), Z[:na].contiguous(), rho[:na].contiguous(), v[:na].contiguous())
        torch.cuda.synchronize()
        assert bool(torch.isfinite(few).all()) and torch.equal(few, many[:na]), na
