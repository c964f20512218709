"""The deposit at the edges of its plans: atoms in each distance class of a tile, ragged tiles,
spheres larger than the near distance, and exponents in every order and ratio."""
import numpy as np
import pytest

import synth
from gpu_common import host, need_gpu

pytestmark = pytest.mark.gpu

ZETAS = [(1.5, 3.0, 8.0), (3.0, 1.5, 8.0), (8.0, 3.0, 1.5), (1.5, 3.0, 3.0), (1.0, 1.3, 2.0), (2.0, 2.0, 2.0), (0.4, 0.8, 9.0)]


def _check(orc, B, cl, axes, precision, tol):
    x, y, z = axes
    dc = B.DeviceCluster(cl, axes=axes)
    dc.n = (len(x), len(y), len(z))
    ref, rowner = orc.deposit(cl, x, y, z)
    b, owner, status = B.lasto_op_deposit(dc, precision=precision)
    assert host(status)[0] == 0
    assert np.array_equal(host(owner), rowner)
    err = np.abs(host(b) - ref)
    # the bounds of the deposit's own test: of the largest value, and node by node where the
    # density matters
    assert err.max() < tol * np.abs(ref).max()
    big = np.abs(ref) > 1e-3 * np.abs(ref).max()
    assert (err[big] / np.abs(ref[big])).max() < 1e-10


@pytest.mark.parametrize("zeta", ZETAS)
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-11)])
def test_exponents(orc, zeta, precision, tol):
    """A row of seven atoms over 45 bohr: every tile sees near, mid, far and dropped atoms."""
    B = need_gpu()
    pos = np.stack([np.linspace(-22, 22, 7), 0.3 * np.arange(7), -0.2 * np.arange(7)], -1)
    cl = synth.workloads.make_cluster("row", pos, np.random.default_rng(5), n=49, half_width=32.0, h_min=4 / 3, h_max=4 / 3)
    cl.slater_zeta[:] = zeta
    x, y, z = orc.mesh(cl)
    _check(orc, B, cl, (x, y[8:-8].copy(), z[10:-10].copy()), precision, tol)


@pytest.mark.parametrize("n", [(33, 35, 37), (65, 9, 17), (17, 41, 11)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-11)])
def test_ragged_tiles(orc, n, precision, tol):
    B = need_gpu()
    cl = synth.pd2_dimer(n=33)
    axes = [np.linspace(-9.0, 9.0, m) for m in n]
    _check(orc, B, cl, axes, precision, tol)


@pytest.mark.parametrize("precision", [0, 1])
def test_spheres_beyond_the_near_distance(orc, precision):
    """Spheres of 7 and 15 bohr (the near distance is 6, the far one 13.3): nodes inside a sphere
    belong to it however far the atom is.  (Owners only: at these radii the neighbours' average
    cancels cosh(zeta R) against sinh(zeta R), in either precision and in the oracle.)"""
    B = need_gpu()
    cl = synth.workloads.make_cluster("large", np.array([[-11.0, 0, 0], [11.5, 0, 0]]), np.random.default_rng(6), n=49,
                                      half_width=30.0, h_min=1.25, h_max=1.25)
    cl.R[:] = (7.0, 15.0)
    cl.slater_zeta[:] = (1.5, 3.0, 4.0)
    axes = orc.mesh(cl)
    _, rowner = orc.deposit(cl, *axes)
    _, owner, status = B.lasto_op_deposit(B.DeviceCluster(cl, axes=axes), precision=precision)
    assert host(status)[0] == 0
    assert np.array_equal(host(owner), rowner)
