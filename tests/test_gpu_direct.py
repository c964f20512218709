"""Solves whose coarse levels are solved exactly by fast diagonalisation: every plan (which level,
which tile, both precisions), unequal axes, and an axis with two refined regions, whose operator
has nearly equal eigenvalue pairs."""
import numpy as np
import pytest

import synth
from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu


def _axis(n, half, two=False):
    t = np.linspace(-1, 1, n)
    if not two:
        return half * (0.6 * t + 0.4 * t ** 3)
    w = 0.15 + np.minimum(np.abs(t[:-1] + t[1:]) / 2 - 0.5, 0.5) ** 2      # dense at +-0.5
    x = np.concatenate([[0.0], np.cumsum(w)])
    return half * (2 * x / x[-1] - 1)


def _solve(B, axes, **kw):
    import torch
    cl = synth.workloads.make_cluster("pair", np.array([[-2.6, 0.1, 0.0], [2.6, 0.0, -0.2]]), np.random.default_rng(3), n=33,
                                      half_width=12.0, h_min=0.75, h_max=0.75)
    dc = B.DeviceCluster(cl, axes=axes)
    dc.n = tuple(len(a) for a in axes)
    solver = B.Poisson(n_max=max(dc.n), max_atoms=2, **kw)
    v = torch.empty((2, 25), dtype=torch.float64, device="cuda")
    u = torch.empty(dc.n[::-1], dtype=torch.float64, device="cuda")
    st = solver.solve(dc, v, potential=u)[0]
    torch.cuda.synchronize()
    assert st.status == 0 and st.rel_resid <= 1e-10, (st.status, st.cycles, st.rel_resid)
    b, _, _ = B.lasto_op_deposit(dc, precision=kw["precision"])
    ub = u.clone()
    ub[1:-1, 1:-1, 1:-1] = 0
    r, rb = B.lasto_op_residual(dc.x, dc.y, dc.z, u, b), B.lasto_op_residual(dc.x, dc.y, dc.z, ub, b)
    # the solve's own bound, on the operator that callers use (FP64 rounding of the operator's
    # terms, eps |A| |u| / |b|, is 1e-12 here)
    assert float(r.norm()) <= 1.1e-10 * float(rb.norm())
    return host(v).copy(), st.cycles


@pytest.mark.parametrize("n", [(65, 65, 65), (81, 81, 81), (113, 97, 65), (129, 113, 129), (161, 161, 161), (193, 129, 97),
                               (225, 65, 65), (49, 41, 33)])
def test_levels(n):
    B = need_gpu()
    axes = [_axis(m, 12.0) for m in n]
    v64, _ = _solve(B, axes, precision=B.LASTO_PREC_FP64)
    v32, _ = _solve(B, axes, precision=B.LASTO_PREC_MIXED)
    # two answers to a residual of 1e-10: their distance is that bound times the solution's
    # smoothness constant, below 1e-8 in every parity test here
    assert np.abs(v64 - v32).max() <= 1e-8 * np.abs(v64).max()


@pytest.mark.parametrize("precision", [0, 1])
def test_two_refined_regions(precision):
    B = need_gpu()
    x = _axis(129, 12.0, two=True)
    _solve(B, [x, x, x], precision=precision)


@pytest.mark.parametrize("cycle", [0, 1])
def test_stationary_cycles(cycle):
    B = need_gpu()
    x = np.linspace(-12, 12, 65)
    _solve(B, [x, x, x], precision=B.LASTO_PREC_FP64, cycle=cycle, max_cycles=120)
