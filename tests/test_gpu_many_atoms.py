"""The deposits of clusters up to the largest that they admit: their lists of atoms in shared memory."""
import numpy as np
import pytest

import synth
from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu


def _lattice(na, k):
    return np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:na].astype(float)


# around the atoms whose lists fit beside the kernels' static memory in the default 48 KiB, and the most
@pytest.mark.parametrize("precision,na,tol", [(1, 1276, 1e-11), (1, 1277, 1e-11), (1, 2431, 1e-11), (0, 1277, 1e-12),
                                              (0, 1828, 1e-12)])
def test_deposit(orc, precision, na, tol):
    B = need_gpu()
    cl = synth.workloads.make_cluster("lattice", 1.25 * _lattice(na, 14) - 8.125, np.random.default_rng(na), n=17, half_width=12.0,
                                      h_min=1.5, h_max=1.5)
    cl.R[:] = 0.6
    x = np.linspace(-12.0, 12.0, 17)
    ref, rowner = orc.deposit(cl, x, x, x)
    b, owner, status = B.lasto_op_deposit(B.DeviceCluster(cl, axes=(x, x, x)), precision=precision)
    assert host(status)[0] == 0
    assert np.array_equal(host(owner), rowner)
    assert np.abs(host(b) - ref).max() < tol * np.abs(ref).max()   # the bound of the deposit's own tests
