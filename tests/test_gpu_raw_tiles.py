"""The raw deposit's lists of spheres per box of 32 x 8 x 4 nodes: ragged boxes, more atoms than one
pass of the block, spheres smaller than a box and larger, against the oracle."""
import numpy as np
import pytest

from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells,radius", [((33, 9, 7), (2, 2, 1), 0.45), ((35, 17, 7), (10, 9, 3), 0.4),
                                            ((65, 33, 21), (8, 8, 5), 0.49), ((97, 7, 9), (1, 1, 1), 0.45),
                                            ((31, 41, 33), (7, 7, 7), 0.05)])
def test_raw_deposit(orc, n, cells, radius):
    B = need_gpu()
    rng = np.random.default_rng(n[0])
    grid = np.stack(np.meshgrid(*[np.arange(c) for c in cells], indexing="ij"), -1).reshape(-1, 3)
    pos = grid + 0.5 + rng.uniform(-0.005, 0.005, size=grid.shape)   # disjoint spheres, in no spatial order
    pos = pos[rng.permutation(len(pos))]
    na = len(pos)
    Z, R = rng.uniform(1, 50, size=na), np.full(na, radius)
    # (two nodes outside the spheres at each end of an axis)
    x, y, z = [np.sort(np.concatenate([[-0.3, -0.2, 0.0, c, c + 0.2, c + 0.3], rng.uniform(0, c, size=v - 6)]))
               for v, c in zip(n, cells)]
    r = radius * np.exp(np.linspace(np.log(1e-5 / radius), 0.0, 64))
    rho00 = rng.uniform(1, 9, size=(na, 1)) * np.exp(-3.0 * r)[None]
    ne = rng.uniform(0, 2, size=n[::-1])
    b, owner, status = B.lasto_op_raw_deposit(B.RawCluster(pos, Z, R, x, y, z, (0, 0, 0), ne, rho00))
    ref, rowner = orc.raw_deposit(pos, Z, R, x, y, z, ne, rho00)
    assert int(host(status)[0]) == 0
    assert np.array_equal(host(owner).reshape(rowner.shape), rowner)
    # sums of a few terms of the quartic's size: the bound of the kernel's own test
    assert np.abs(host(b).reshape(ref.shape) - ref).max() < 1e-12 * np.abs(ref).max()
