"""Boundary multipoles and faces where the plane kernel's split changes (few columns and many ranges,
one range, columns beyond one tile), and the learned guess's copies on nested grids."""
import numpy as np
import pytest

from gpu_common import dev, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(5, 7, 9), (9, 5, 33), (33, 129, 5), (129, 33, 17), (257, 9, 5), (1023, 5, 5),
                               (1031, 7, 3), (2053, 5, 3)])
def test_multipoles_and_faces(orc, n):
    B = need_gpu()
    rng = np.random.default_rng(n[0])
    x, y, z = [np.cumsum(rng.uniform(0.5, 1.5, size=v)) / v for v in n]
    b = rng.uniform(0.5, 1.5, size=n[::-1])   # one sign: no cancellation in the sums below degree 1
    centre = (0.3, 0.4, 0.6)
    Q = host(B.lasto_op_multipoles(dev(x), dev(y), dev(z), dev(b), centre))
    ref = orc.multipoles(x, y, z, b, centre)
    # products of three table entries and sums of at most 2053 + 7 + 33 terms, added in another
    # order: 1e-12 leaves a factor of four
    assert np.abs(Q - ref).max() < 1e-12 * np.abs(ref).max()
    import torch
    u = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    far = (centre[0] + 5.0, centre[1] - 4.0, centre[2] + 6.0)   # outside the box: no face near it
    B.lasto_op_boundary_fill(dev(x), dev(y), dev(z), dev(ref), u, far)
    uref = orc.boundary_fill(x, y, z, ref, np.zeros(n[::-1]), far)
    assert np.abs(host(u) - uref).max() < 1e-13 * np.abs(uref).max()
