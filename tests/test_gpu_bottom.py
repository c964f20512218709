"""The FP32 cycle's one-block coarse levels (grids of at most 33 nodes per axis have them): their
sweep count changes the iteration, not the answer, alone and in a lockstep batch."""
import numpy as np
import pytest

import synth
from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu


def _solve(B, cls, nu_coarse, launch):
    import torch
    dcs = [B.DeviceCluster(c) for c in cls]
    solver = B.Poisson(n_max=33, max_atoms=13, max_batch=len(cls), precision=B.LASTO_PREC_MIXED, nu_coarse=nu_coarse,
                       launch=launch)
    v = torch.empty((13 * len(cls), 25), dtype=torch.float64, device="cuda")
    st = solver.solve(dcs, v)
    torch.cuda.synchronize()
    out = host(v).copy(), [(s.status, s.cycles, s.rel_resid) for s in st]
    solver.close()
    return out


def test_coarse_sweeps(orc):
    B = need_gpu()
    cls = [synth.pd13_small(n=33, seed=s) for s in (21, 22, 23)]
    ref = np.concatenate([orc.poisson_solve(c, tol=1e-13, max_cycles=200)["vlm"] for c in cls])
    residuals = set()
    for nu in (0, 1, 4):
        v, st = _solve(B, cls, nu, 0)
        assert all(s[0] == 0 and s[2] <= 1e-10 for s in st), st
        assert np.abs(v - ref).max() < 1e-8 * np.abs(ref).max()
        residuals.add(tuple(st))
        vl, stl = _solve(B, cls, nu, 2)
        assert stl == st and np.array_equal(v, vl), nu      # the group's levels in one launch: bitwise
    assert len(residuals) == 3, residuals                   # the sweeps are not left out
