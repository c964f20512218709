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
