"""The deposits of clusters up to the largest that they admit: their lists of atoms in shared memory."""
import numpy as np
import pytest

import synth
from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu


def _lattice(na, k):
    return np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:na].astype(float)


# around the atoms whose lists fit beside the kernels' static memory in the default 48 KiB, and the most
@pytest.mark.parametrize("precision,na,tol", [(1, 1276, 1e-11), (1, 1277, 1e-11), (1, 2431, 1e-11), (1, 2432, 1e-11), (0, 1277, 1e-12),
                                              (0, 1828, 1e-12)])
def test_deposit(precision, na, tol):
    """Owners everywhere and the values outside the spheres, which are the Slater sums themselves,
    against 64 bits."""
    import torch
    B = need_gpu()
    cl = synth.workloads.make_cluster("lattice", 1.5 * _lattice(na, 14) - 9.75, np.random.default_rng(na), n=33, half_width=12.0,
                                      h_min=0.75, h_max=0.75)
    cl.R[:] = 0.7
    x = np.linspace(-12.0, 12.0, 33)
    b, owner, status = B.lasto_op_deposit(B.DeviceCluster(cl, axes=(x, x, x)), precision=precision)
    assert host(status)[0] == 0 and bool(torch.isfinite(b).all())
    t = torch.as_tensor(x, device="cuda")
    ref, own = torch.zeros(33 ** 3, dtype=torch.float64, device="cuda"), torch.full((33 ** 3,), -1, dtype=torch.int32, device="cuda")
    for a in range(na):
        p = cl.pos[a]
        r = ((t[None, None, :] - p[0]) ** 2 + (t[None, :, None] - p[1]) ** 2 + (t[:, None, None] - p[2]) ** 2).sqrt().view(-1)
        own[r < cl.R[a]] = a
        for w, z in zip(cl.slater_w[a], cl.slater_zeta[a]):
            ref += 4 * np.pi * w * z ** 3 / (8 * np.pi) * torch.exp(-z * r)
    assert torch.equal(owner.view(-1), own)
    out = own < 0
    # the bound of the deposit's own tests
    assert float((b.view(-1)[out] - ref[out]).abs().max()) < tol * float(ref[out].max())


@pytest.mark.parametrize("precision,na", [(0, 1829), (1, 2433)])
def test_deposit_refuses_more(precision, na):
    B = need_gpu()
    cl = synth.workloads.make_cluster("lattice", 1.5 * _lattice(na, 14) - 9.75, np.random.default_rng(na), n=33, half_width=12.0,
                                      h_min=0.75, h_max=0.75)
    with pytest.raises(RuntimeError):
        B.lasto_op_deposit(B.DeviceCluster(cl, axes=(np.linspace(-12.0, 12.0, 33),) * 3), precision=precision)


# around the list that fits beside the static memory in the default 48 KiB and the one that fits alone
@pytest.mark.parametrize("na", [10240, 11300, 12288, 12800])
def test_raw_deposit(orc, na):
    B = need_gpu()
    rng = np.random.default_rng(na)
    pos, Z, R = _lattice(na, 24) + 0.5, rng.uniform(1, 50, size=na), np.full(na, 0.4)
    x = np.concatenate([[-0.3, -0.2], np.linspace(0.0, 24.0, 17), [24.2, 24.3]])
    r = 0.4 * np.exp(np.linspace(np.log(1e-5 / 0.4), 0.0, 16))
    rho00 = rng.uniform(1, 9, size=(na, 1)) * np.exp(-3.0 * r)[None]
    ne = rng.uniform(0, 2, size=(21, 21, 21))
    ref, rowner = orc.raw_deposit(pos, Z, R, x, x, x, ne, rho00)
    b, owner, status = B.lasto_op_raw_deposit(B.RawCluster(pos, Z, R, x, x, x, (0, 0, 0), ne, rho00))
    assert int(host(status)[0]) == 0
    assert np.array_equal(host(owner).reshape(rowner.shape), rowner)
    assert np.abs(host(b).reshape(ref.shape) - ref).max() < 1e-12 * np.abs(ref).max()   # the bound of the kernel's own test


def test_raw_deposit_refuses_more():
    B = need_gpu()
    x = np.linspace(0.0, 24.0, 9)
    rc = B.RawCluster(_lattice(12801, 24) + 0.5, np.ones(12801), np.full(12801, 0.4), x, x, x, (0, 0, 0), np.ones((9, 9, 9)),
                      np.ones((12801, 16)))
    with pytest.raises(RuntimeError):
        B.lasto_op_raw_deposit(rc)


def test_exact_faces_of_many_atoms_on_a_small_grid():
    """A solve whose atoms' five moments need more room than the grid's multipole tables."""
    import torch
    B = need_gpu()
    na, n = 600, 17
    cl = synth.workloads.make_cluster("lattice", 2.0 * _lattice(na, 9) - 8.0, np.random.default_rng(na), n=n, half_width=12.0,
                                      h_min=1.5, h_max=1.5)
    cl.R[:] = 0.6
    dc = B.DeviceCluster(cl, axes=(np.linspace(-12.0, 12.0, n),) * 3)
    u = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    B.lasto_op_boundary_exact(dc, u)
    for precision in (B.LASTO_PREC_FP64, B.LASTO_PREC_MIXED):
        solver = B.Poisson(n_max=n, max_atoms=na, precision=precision, boundary=B.LASTO_BC_EXACT)
        v, pot = torch.empty((na, 25), dtype=torch.float64, device="cuda"), torch.empty_like(u)
        st = solver.solve(dc, v, potential=pot)[0]
        torch.cuda.synchronize()
        assert st.status == 0 and st.rel_resid <= 1e-10, (st.status, st.rel_resid)
        face = torch.ones_like(u, dtype=torch.bool)
        face[1:-1, 1:-1, 1:-1] = False
        assert torch.equal(pot[face], u[face])
