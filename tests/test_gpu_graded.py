"""Mixed-precision solves on strongly graded axes, whose coarse operators have eigenvalues that FP32
cannot tell from zero beside their largest elements: the exactly solved level has to stay definite."""
import numpy as np
import pytest

import synth
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _axis(n, half, w):
    """Spacings w from the centre outwards, scaled to the half width."""
    x = np.concatenate([[0.0], np.cumsum(w)])
    x *= half / x[-1]
    return np.concatenate([-x[::-1], x[1:]])


def _fine_cells(n, half, ratio, k):
    """Uniform but for 2 k cells at the centre, `ratio` times finer."""
    w = np.ones((n - 1) // 2)
    w[:k] = 1.0 / ratio
    return _axis(n, half, w)


def _power(n, half, ratio, power):
    """Spacings that grow by `ratio` from the centre, fast at first."""
    m = (n - 1) // 2
    return _axis(n, half, ratio ** (((np.arange(m) + 0.5) / m) ** power))


# (the smoothed hierarchy without the exact level took 148, 155, 196 and 179 iterations)
@pytest.mark.parametrize("n,axis", [(129, lambda n: _fine_cells(n, 40.0, 1000, 2)), (129, lambda n: _power(n, 40.0, 64000, 0.25)),
                                    (193, lambda n: _power(n, 40.0, 64000, 0.25)), (193, lambda n: _fine_cells(n, 40.0, 1000, 2))])
def test_one_strongly_graded_axis(n, axis):
    import torch
    B = need_gpu()
    cl = synth.workloads.make_cluster("pair", np.array([[-2.6, 0.1, 0.0], [2.6, 0.0, -0.2]]), np.random.default_rng(3), n=33,
                                      half_width=12.0, h_min=0.75, h_max=0.75)
    u = np.linspace(-40.0, 40.0, n)
    dc = B.DeviceCluster(cl, axes=[axis(n), u, u])
    dc.n = (n, n, n)
    solver = B.Poisson(n_max=n, max_atoms=2, precision=B.LASTO_PREC_MIXED, max_cycles=250)
    v = torch.empty((2, 25), dtype=torch.float64, device="cuda")
    st = solver.solve(dc, v)[0]
    torch.cuda.synchronize()
    assert st.status == 0 and st.rel_resid <= 1e-10, (st.status, st.cycles, st.rel_resid)
