"""The weight gradient where one sum is long: its error must not grow with the number of nodes that
a block takes (the tensor core's FP32 accumulation truncates)."""
import ctypes

import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def wgrad(B, x, dy, nb, dims, cin, cout):
    import torch
    dw = torch.zeros(27, cin, cout, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert B.load().lasto_nn_conv3d_wgrad_tc(nb, (ctypes.c_int * 3)(*dims), cin, cout, B._ptr(x), B._ptr(dy), None, B._ptr(dw),
                                             None, B._ptr(err), B._stream()) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    return dw


def wgrad_ref(x, dy, nb, dims):
    """The same in 64 bits: per tap, the rows of x at the neighbour against the rows of dy."""
    import torch
    W, H, D = dims
    X, Y = x.double().view(nb, D, H, W, -1), dy.double().view(nb, D, H, W, -1)
    here = lambda d, n: slice(max(0, -d), n - max(0, d))
    there = lambda d, n: slice(max(0, d), n + min(0, d))
    out = []
    for dz in (-1, 0, 1):
        for dy_ in (-1, 0, 1):
            for dx in (-1, 0, 1):
                a = X[:, there(dz, D), there(dy_, H), there(dx, W)].reshape(-1, X.shape[-1])
                b = Y[:, here(dz, D), here(dy_, H), here(dx, W)].reshape(-1, Y.shape[-1])
                out.append(a.T @ b)
    return torch.stack(out)


@pytest.mark.parametrize("cin,cout,nb,dims", [(64, 64, 8, (33, 33, 33)), (128, 128, 4, (33, 33, 33)), (128, 64, 6, (65, 17, 31)),
                                              (96, 32, 12, (33, 33, 33))])
def test_long_sums(cin, cout, nb, dims):
    import torch
    B = need_gpu()
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    N = nb * dims[0] * dims[1] * dims[2]
    # (positive values: truncation then always errs to the same side)
    x = torch.randn(N, cin, generator=g, device="cuda").abs().bfloat16()
    dy = torch.randn(N, cout, generator=g, device="cuda").abs().bfloat16()
    got, ref = wgrad(B, x, dy, nb, dims, cin, cout).double(), wgrad_ref(x, dy, nb, dims)
    # sums of at most 2048 nodes, 16 per MMA, each truncated by up to 2^-23 of a partial sum that is
    # half the whole on average; then one rounded FP32 addition (2^-24) per such sum
    tol = 2.0 ** -24 * (2048 / 16 + N / 2048 + 1)
    assert float(((got - ref) / ref).abs().max()) <= tol


@pytest.mark.parametrize("cin,cout,nb,dims", [(16, 16, 2, (7, 8, 9)), (48, 16, 2, (7, 8, 9)), (32, 32, 2, (7, 8, 9)),
                                              (128, 64, 1, (5, 3, 4)), (32, 96, 1, (9, 5, 6)), (64, 64, 4, (33, 33, 33))])
@pytest.mark.parametrize("where", ["x", "dy"])
def test_infinities_at_the_edges(cin, cout, nb, dims, where):
    """An infinity at a corner, an edge and a face of a grid reaches the taps that have a partner for it
    inside the grid, and no others."""
    import torch
    B = need_gpu()
    W, H, D = dims
    g = torch.Generator(device="cuda").manual_seed(cin)
    x = torch.randn(nb, D, H, W, cin, generator=g, device="cuda").bfloat16()
    dy = torch.randn(nb, D, H, W, cout, generator=g, device="cuda").bfloat16()
    t = x if where == "x" else dy
    t[0, 0, 0, 0, 1] = float("inf")
    t[nb - 1, D - 1, 1, W - 1, 2] = -float("inf")
    t[0, 1, H - 1, 2, 3] = float("inf")
    x, dy = x.view(-1, cin), dy.view(-1, cout)
    got, ref = wgrad(B, x, dy, nb, dims, cin, cout).double(), wgrad_ref(x, dy, nb, dims)
    assert bool(ref.isinf().any()) and bool(ref.isfinite().any())
    assert torch.equal(got.isnan(), ref.isnan()) and torch.equal(got.isinf(), ref.isinf())
    assert torch.equal(got[ref.isinf()], ref[ref.isinf()])
    ok = ref.isfinite()
    assert float((got[ok] - ref[ok]).abs().max()) <= 2e-5 * float(ref[ok].abs().max())


def test_bias_gradient_sums_pairwise():
    """64 rows of a block whose serial FP32 sum would round down by almost half a last place each time."""
    import numpy as np
    import torch
    B = need_gpu()
    v = [1.5]
    s = np.float32(1.5)
    for _ in range(63):
        ulp = float(np.spacing(s + np.float32(1.25)))
        x = 1.25
        if ulp > 2.0 ** -22:
            x += (ulp / 2 - 2.0 ** -23 - (float(s) + x) % ulp) % ulp
        v.append(x)
        s = np.float32(s + np.float32(x))
    dy = torch.as_tensor(np.repeat(np.array(v, dtype=np.float32)[:, None], 16, 1)).cuda()
    x16, dy16 = torch.zeros(64, 16, dtype=torch.bfloat16, device="cuda"), dy.bfloat16()
    dw, db = torch.zeros(27, 16, 16, device="cuda"), torch.zeros(16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert B.load().lasto_nn_conv3d_wgrad_tc(1, (ctypes.c_int * 3)(4, 4, 4), 16, 16, B._ptr(x16), B._ptr(dy16), B._ptr(dy),
                                             B._ptr(dw), B._ptr(db), B._ptr(err), B._stream()) == 0
    torch.cuda.synchronize()
    exact = sum(v)
    # eight sums of eight rows and their three levels: ten roundings
    assert float((db.double() - exact).abs().max()) <= 10 * 2.0 ** -24 * exact


@pytest.mark.parametrize("cin,cout,nb,dims", [(16, 16, 3, (1000, 1, 9)), (32, 48, 2, (1000, 9, 1)), (64, 32, 2, (900, 1, 1)),
                                              (16, 16, 3, (1, 7, 18)), (64, 96, 1, (7, 1, 18)), (48, 16, 2, (7, 18, 1)),
                                              (32, 32, 4, (1, 1, 1))])
def test_axes_of_one_node(cin, cout, nb, dims):
    """Gathered rows (beyond about 450 nodes) and the padded sequence."""
    import torch
    B = need_gpu()
    g = torch.Generator(device="cuda").manual_seed(dims[0])
    N = nb * dims[0] * dims[1] * dims[2]
    x = torch.randn(N, cin, generator=g, device="cuda").bfloat16()
    dy = torch.randn(N, cout, generator=g, device="cuda").bfloat16()
    got, ref = wgrad(B, x, dy, nb, dims, cin, cout).double(), wgrad_ref(x, dy, nb, dims)
    # FP32 sums: the bound of the kernels' own tests
    assert float((got - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
