"""The sphere quadrature's users at the sizes where their plans change: the projection split over
one to eight blocks per sphere, its axes staged in shared memory or not, and the density's
harmonics from Chebyshev points or from every radius, with rules that are not exact."""
import numpy as np
import pytest

import synth
from gpu_common import dev, host, need_gpu

pytestmark = pytest.mark.gpu


def _axis(n, half):
    return np.linspace(-half, half, n)


@pytest.mark.parametrize("na,n,rule", [(1, (9, 11, 13), (16, 32)), (13, (65, 33, 17), (16, 32)), (120, (33, 33, 33), (16, 32)),
                                       (310, (17, 17, 17), (16, 32)), (5, (2801, 5, 9), (16, 32)), (7, (33, 35, 37), (1, 1)),
                                       (7, (33, 35, 37), (3, 5)), (7, (33, 35, 37), (13, 9)), (3, (33, 35, 37), (32, 64))])
def test_projection_plans(orc, na, n, rule):
    B = need_gpu()
    rng = np.random.default_rng(na)
    x, y, z = _axis(n[0], 9.0), _axis(n[1], 8.0), _axis(n[2], 7.0)
    pos, R = rng.uniform(-3, 3, (na, 3)), rng.uniform(0.3, 3.5, na)
    u = rng.normal(size=n[::-1])
    vlm, status = B.lasto_op_project(dev(x), dev(y), dev(z), dev(u), dev(pos), dev(R), n_theta=rule[0], n_phi=rule[1])
    ref = orc.project(x, y, z, u, pos, R, *rule)
    assert host(status)[0] == 0
    # sums of at most 2048 FP64 products: n eps of their absolute sum, well below 1e-13 of the largest
    assert np.abs(host(vlm) - ref).max() < 1e-13 * max(np.abs(ref).max(), 1.0)


def test_projection_reports_points_outside(orc):
    B = need_gpu()
    x = _axis(17, 4.0)
    u = np.ones((17, 17, 17))
    pos, R = np.array([[0.0, 0.0, 0.0], [2.0, 0.0, 0.0]]), np.array([4.0, 2.5])
    _, status = B.lasto_op_project(dev(x), dev(x), dev(x), dev(u), dev(pos[:1]), dev(R[:1]))
    assert host(status)[0] == 0                       # the surface touches the faces
    _, status = B.lasto_op_project(dev(x), dev(x), dev(x), dev(u), dev(pos), dev(R))
    assert host(status)[0] == B.LASTO_ERR_GEOMETRY


def _pair(rng, R, d):
    cl = synth.workloads.make_cluster("pair", np.array([[0.0, 0.0, 0.0], [0.6 * d, 0.0, 0.8 * d]]), rng, n=33,
                                      half_width=14.0, h_min=0.875, h_max=0.875)
    cl.R[:] = R
    return cl


# r_min = 3: radii outside the sphere.  (2.4, 0.01): the small sphere all but touches the large
# one, so every radius is evaluated; the small sphere keeps its few points.
@pytest.mark.parametrize("R,d,n_rad,r_min,rule", [
    ((2.4, 2.4), 4.85, 429, 1e-5, (16, 32)), ((2.4, 0.01), 2.42, 429, 1e-5, (16, 32)), ((2.0, 1.0), 3.1, 60, 1e-3, (16, 32)),
    ((2.4, 2.4), 4.85, 20, 1e-5, (16, 32)), ((2.4, 2.4), 4.85, 4, 1e-5, (8, 16)), ((2.4, 2.4), 5.2, 64, 3.0, (16, 32)),
    ((2.4, 2.4), 4.85, 100, 1e-5, (4, 32)), ((2.4, 2.4), 4.85, 100, 1e-5, (16, 8)), ((2.4, 2.4), 4.85, 100, 1e-5, (5, 9)),
    ((2.4, 2.4), 4.85, 50, 1e-5, (1, 1))])
def test_sphere_density_plans(orc, R, d, n_rad, r_min, rule):
    B = need_gpu()
    cl = _pair(np.random.default_rng(n_rad), np.array(R), d)
    rho, _ = B.lasto_op_sphere_density(B.DeviceCluster(cl), n_rad=n_rad, r_min=r_min, n_theta=rule[0], n_phi=rule[1])
    # the entry point's density: every atom's Slater shells and the sphere's own nonspherical part
    # (the oracle's density holds a neighbour's part too where a radius reaches into its sphere)
    ref = np.empty(rho.shape)
    for a in range(2):
        own = synth.workloads.replace(cl, c_lm=np.where(np.arange(2)[:, None] == a, cl.c_lm, 0.0))
        ref[a] = orc.sphere_density(own, n_rad=n_rad, r_min=r_min, n_theta=rule[0], n_phi=rule[1])[a]
    # FP32-pair sums (~44 bits); the interpolation adds 2^-66 of the weights
    assert np.abs(host(rho) - ref).max() < 1e-12 * np.abs(ref).max()


def test_sphere_density_of_a_single_atom(orc):
    B = need_gpu()
    cl = synth.workloads.make_cluster("one", np.zeros((1, 3)), np.random.default_rng(3), n=33, half_width=12.0, h_min=0.75,
                                      h_max=0.75)
    rho, _ = B.lasto_op_sphere_density(B.DeviceCluster(cl))
    ref = orc.sphere_density(cl)
    assert np.abs(host(rho) - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("n_rad", [5, 6, 8, 129, 430])
def test_raw_sphere_charge(orc, n_rad):
    """The composite cubic weights of the raw path's charge integral, from the shortest table on:
    the deposit inside the spheres against the oracle's interval-by-interval rule."""
    B = need_gpu()
    cl = _pair(np.random.default_rng(n_rad), 2.4, 4.9)
    x, y, z = orc.mesh(cl)
    r = np.stack([orc.radial_mesh(n_rad, 1e-2, R) for R in cl.R])
    rho00 = np.exp(-r) * (1.0 + 0.1 * np.arange(2)[:, None])
    ne = np.random.default_rng(1).uniform(0.1, 0.2, (33, 33, 33))
    b, owner, status = B.lasto_op_raw_deposit(B.RawCluster(cl.pos, cl.Z, cl.R, x, y, z, cl.centre, ne, rho00, r_min=1e-2))
    ref, rowner = orc.raw_deposit(cl.pos, cl.Z, cl.R, x, y, z, ne, rho00, r_min=1e-2)
    assert int(host(status)[0]) == 0
    assert np.array_equal(host(owner).reshape(rowner.shape), rowner)
    assert np.abs(host(b).reshape(ref.shape) - ref).max() < 1e-12 * np.abs(ref).max()
