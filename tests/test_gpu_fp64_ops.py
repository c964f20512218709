"""The FP64 grid transfers and residual against the oracle where their thread layouts end:
rows of one warp step and one node more, column blocks of 32 x 4, marches of four planes."""
import numpy as np
import pytest

from gpu_common import dev, host, need_gpu

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53
SIZES = [(5, 5, 5), (7, 5, 9), (65, 9, 11), (67, 11, 7), (129, 13, 19), (131, 5, 17), (9, 67, 21), (63, 65, 67)]


def _grid(n, seed):
    rng = np.random.default_rng(seed)
    return [np.cumsum(rng.uniform(0.5, 1.5, size=v)) for v in n]


@pytest.mark.parametrize("n", SIZES)
def test_transfers(orc, n):
    B = need_gpu()
    x, y, z = _grid(n, 1)
    rng = np.random.default_rng(2)
    r = rng.normal(size=n[::-1])
    # 27 weighted terms: at most 27 roundings of the sum of their sizes on each side
    size = orc.restrict(x, y, z, np.abs(r))
    bc = host(B.lasto_op_restrict(dev(x), dev(y), dev(z), dev(r)))
    assert (np.abs(bc - orc.restrict(x, y, z, r)) <= 2 * 27 * EPS * np.abs(size)).all()
    nc = tuple((v + 1) // 2 for v in n)
    ec, u = rng.normal(size=nc[::-1]), rng.normal(size=n[::-1])
    size = orc.prolong_add(x, y, z, np.abs(ec), np.abs(u))
    got = host(B.lasto_op_prolong_add(dev(x), dev(y), dev(z), dev(ec), dev(u)))
    ref = orc.prolong_add(x, y, z, ec, u.copy())
    assert (np.abs(got - ref) <= 2 * 12 * EPS * np.abs(size)).all()


@pytest.mark.parametrize("n", SIZES)
def test_residual(orc, n):
    B = need_gpu()
    x, y, z = _grid(n, 3)
    rng = np.random.default_rng(4)
    u, b = rng.normal(size=n[::-1]), rng.normal(size=n[::-1])
    r = host(B.lasto_op_residual(dev(x), dev(y), dev(z), dev(u), dev(b)))
    ref = orc.residual(x, y, z, u, b)
    # eight terms; the coefficients are the same numbers up to four roundings of their own
    h = min(np.diff(a).min() for a in (x, y, z))
    assert np.abs(r - ref).max() <= 2 * 12 * EPS * 12.0 / (h * h) * np.abs(u).max()
    assert (r[0] == 0).all() and (r[:, -1] == 0).all() and (r[:, :, 0] == 0).all()


@pytest.mark.parametrize("n,scale", [((5, 5, 5), 1.0), ((65, 9, 11), 1e-3), ((33, 37, 29), 1e4), ((5, 9, 5), 1e-153),
                                     ((5, 9, 5), 1e152)])
def test_inverse_diagonal(n, scale):
    """One red half sweep from zero with b = 1 returns the negated reciprocal of the diagonal."""
    import torch
    B = need_gpu()
    x, y, z = [a * scale for a in _grid(n, 5)]
    u = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    b = torch.ones(n[::-1], dtype=torch.float64, device="cuda")
    B.lasto_op_smooth(dev(x), dev(y), dev(z), u, b, 1)
    got = host(u)

    def dg(a):
        h = np.diff(a).astype(np.longdouble)
        s = h[:-1] + h[1:]
        return 2 / (s * h[:-1]) + 2 / (s * h[1:])

    d = dg(z)[:, None, None] + dg(y)[None, :, None] + dg(x)[None, None, :]
    k, j, i = np.indices(d.shape) + 1
    red = (i + j + k) % 2 == 0
    ref = -1 / d
    # the diagonal's own six terms carry up to 4 roundings each and two additions, the reciprocal one
    assert (np.abs(got[1:-1, 1:-1, 1:-1] - ref)[red] <= 8 * 2 * EPS * np.abs(ref)[red]).all()
