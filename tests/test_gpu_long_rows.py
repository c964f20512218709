"""The FP64 grid operations on very long rows (split over blocks: one node on either side of 512, several
pieces) and very short ones (several rows per warp, narrow blocks of columns)."""
import numpy as np
import pytest

from gpu_common import dev, host, need_gpu

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53
SIZES = [(511, 5, 7), (513, 7, 5), (1023, 5, 5), (1025, 5, 9), (2049, 5, 5), (5, 67, 65), (7, 33, 67), (9, 65, 35), (15, 35, 33),
         (17, 65, 33), (19, 37, 35), (31, 35, 33), (33, 65, 35), (35, 33, 37)]


@pytest.mark.parametrize("n", SIZES)
def test_residual(orc, n):
    B = need_gpu()
    rng = np.random.default_rng(n[0])
    x, y, z = [np.cumsum(rng.uniform(0.5, 1.5, size=v)) for v in n]
    u, b = rng.normal(size=n[::-1]), rng.normal(size=n[::-1])
    r = host(B.lasto_op_residual(dev(x), dev(y), dev(z), dev(u), dev(b)))
    # eight terms; the coefficients are the same numbers up to four roundings of their own
    h = min(np.diff(a).min() for a in (x, y, z))
    assert np.abs(r - orc.residual(x, y, z, u, b)).max() <= 2 * 12 * EPS * 12.0 / (h * h) * np.abs(u).max()
    assert (r[0] == 0).all() and (r[:, -1] == 0).all() and (r[:, :, 0] == 0).all() and (r[:, :, -1] == 0).all()


@pytest.mark.parametrize("n", SIZES)
def test_transfers(orc, n):
    B = need_gpu()
    rng = np.random.default_rng(n[0])
    x, y, z = [np.cumsum(rng.uniform(0.5, 1.5, size=v)) for v in n]
    r = rng.normal(size=n[::-1])
    # 27 weighted terms: at most 27 roundings of the sum of their sizes on each side
    size = orc.restrict(x, y, z, np.abs(r))
    bc = host(B.lasto_op_restrict(dev(x), dev(y), dev(z), dev(r)))
    assert (np.abs(bc - orc.restrict(x, y, z, r)) <= 2 * 27 * EPS * np.abs(size)).all()
    ec, u = rng.normal(size=tuple((v + 1) // 2 for v in n[::-1])), rng.normal(size=n[::-1])
    size = orc.prolong_add(x, y, z, np.abs(ec), np.abs(u))
    got = host(B.lasto_op_prolong_add(dev(x), dev(y), dev(z), dev(ec), dev(u)))
    assert (np.abs(got - orc.prolong_add(x, y, z, ec, u.copy())) <= 2 * 12 * EPS * np.abs(size)).all()


@pytest.mark.parametrize("n", [(513, 7, 5), (1025, 5, 9)])
def test_smooth(orc, n):
    """The inverse diagonal of long rows: one red half sweep from zero with b = 1 returns its negative."""
    import torch
    B = need_gpu()
    rng = np.random.default_rng(n[0])
    ax = [np.cumsum(rng.uniform(0.5, 1.5, size=v)) for v in n]
    u = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    B.lasto_op_smooth(*[dev(a) for a in ax], u, torch.ones(n[::-1], dtype=torch.float64, device="cuda"), 1)
    dg = []
    for a in ax:
        h = np.diff(a)
        dg.append(2 / ((h[:-1] + h[1:]) * h[:-1]) + 2 / ((h[:-1] + h[1:]) * h[1:]))
    ref = -1 / (dg[2][:, None, None] + dg[1][None, :, None] + dg[0][None, None, :])
    k, j, i = np.indices(ref.shape) + 1
    red = (i + j + k) % 2 == 0
    # the diagonal's six terms up to 4 roundings each and two additions, the reciprocal one, on both sides
    assert (np.abs(host(u)[1:-1, 1:-1, 1:-1] - ref)[red] <= 2 * 8 * 2 * EPS * np.abs(ref)[red]).all()
