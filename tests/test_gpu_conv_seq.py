"""The convolution and its weight gradient over the padded sequence of grids, at sizes where the
plan changes: enough tiles for it, one channel chunk or several, ragged grids, strided and
unaligned outputs, rows so long that the channel groups shrink, and rows beyond it."""
import ctypes

import numpy as np
import pytest

from gpu_common import need_gpu
from oracle import unet_oracle as U

pytestmark = pytest.mark.gpu


def _bf16(a):
    import torch
    return torch.as_tensor(np.asarray(a, dtype=np.float32)).to(torch.bfloat16)


def _f64(t):
    return t.float().double().cpu().numpy()


@pytest.mark.parametrize("cin,cout,nb,dims,ldy,off", [
    (16, 16, 1, (33, 29, 21), 16, 0), (48, 16, 2, (17, 23, 31), 24, 4), (32, 48, 3, (9, 31, 29), 53, 3),
    (16, 96, 40, (5, 8, 9), 96, 0), (64, 64, 1, (27, 30, 25), 64, 0), (16, 128, 1, (700, 5, 4), 128, 0),
    (32, 32, 2, (1, 120, 80), 32, 0), (128, 64, 1, (28, 28, 25), 64, 0), (32, 96, 2, (17, 23, 31), 101, 2),
    (48, 128, 1, (20, 20, 20), 128, 0)])
def test_forward(cin, cout, nb, dims, ldy, off):
    import torch
    B = need_gpu()
    L = B.load()
    rng = np.random.default_rng(cin + 7 * cout)
    W, H, D = dims
    N = nb * D * H * W
    x = _bf16(rng.normal(size=(nb, D, H, W, cin))).cuda()
    w = _bf16(rng.normal(size=(27, cin, cout)) * 0.1).cuda()
    wpk = torch.empty_like(w)
    bias = torch.as_tensor(rng.normal(size=cout), dtype=torch.float32).cuda()
    y = torch.full((N, ldy), -7.0, dtype=torch.float32, device="cuda")
    y16 = torch.full((N, ldy), -7.0, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert L.lasto_nn_pack_weights(cin, cout, B._ptr(w), B._ptr(wpk), B._stream()) == 0
    assert L.lasto_nn_conv3d_fwd_tc(nb, (ctypes.c_int * 3)(*dims), cin, cout, B._ptr(x), B._ptr(wpk), B._ptr(bias), 1,
                                    B._ptr(y), ldy, off, B._ptr(y16), ldy, off, B._ptr(err), B._stream()) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = np.maximum(U.conv3d(_f64(x), _f64(w), bias.double().cpu().numpy()), 0).reshape(N, cout)
    got = y[:, off:off + cout].double().cpu().numpy()
    # FP32 sums of 27 cin products: the bound of the kernel's own tests
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()
    assert torch.equal(y16[:, off:off + cout], y[:, off:off + cout].to(torch.bfloat16))
    rest = torch.ones(ldy, dtype=torch.bool, device="cuda")
    rest[off:off + cout] = False
    assert bool((y[:, rest] == -7).all()) and bool((y16[:, rest] == -7).all())


@pytest.mark.parametrize("cin,cout,nb,dims", [(48, 16, 2, (33, 12, 10)), (16, 16, 1, (3, 2, 1)), (128, 64, 1, (9, 9, 9)),
                                              (96, 32, 3, (17, 5, 6)), (64, 64, 1, (201, 3, 3)), (32, 16, 1, (440, 3, 2)),
                                              (16, 32, 1, (1000, 2, 2)), (32, 96, 1, (20, 11, 8)), (16, 48, 5, (33, 7, 9))])
def test_weight_gradient(cin, cout, nb, dims):
    import torch
    B = need_gpu()
    L = B.load()
    rng = np.random.default_rng(3 * cin + cout)
    W, H, D = dims
    x = _bf16(rng.normal(size=(nb, D, H, W, cin))).cuda()
    dy16 = _bf16(rng.normal(size=(nb * D * H * W, cout))).cuda()
    dy32 = dy16.float()
    w = _bf16(np.zeros((27, cin, cout)))
    _, rdw, _ = U.conv3d_backward(_f64(x), _f64(w), _f64(dy16).reshape(nb, D, H, W, cout))
    for shift in (0, 1):                     # dw on 16 bytes, and not
        buf = torch.zeros(27 * cin * cout + 4, dtype=torch.float32, device="cuda")
        dw = buf[shift:shift + 27 * cin * cout]
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert L.lasto_nn_conv3d_wgrad_tc(nb, (ctypes.c_int * 3)(*dims), cin, cout, B._ptr(x), B._ptr(dy16), B._ptr(dy32),
                                          B._ptr(dw), None, B._ptr(err), B._stream()) == 0
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        got = dw.double().cpu().numpy().reshape(27, cin, cout)
        assert np.abs(got - rdw).max() <= 2e-5 * np.abs(rdw).max()


@pytest.mark.parametrize("n,shift", [(4096, 0), (4099, 0), (1024, 1), (8, 0), (1, 0)])
def test_relu_gradient(n, shift):
    import torch
    B = need_gpu()
    L = B.load()
    g = torch.Generator(device="cuda").manual_seed(n)
    y = torch.randn(n + 4, generator=g, device="cuda")[shift:shift + n]
    y[0], y[-1] = 0.0, float("nan")
    for inplace in (False, True):
        dy = torch.randn(n + 4, generator=g, device="cuda")[shift:shift + n]
        dx = dy if inplace else torch.empty_like(dy)
        dx16 = torch.empty(n, dtype=torch.bfloat16, device="cuda")
        ref = torch.where(y > 0, dy, torch.zeros_like(dy))
        assert L.lasto_nn_relu_grad(n, B._ptr(y), B._ptr(dy), B._ptr(dx), B._ptr(dx16), B._stream()) == 0
        assert torch.equal(dx, ref) and torch.equal(dx16, ref.to(torch.bfloat16))


@pytest.mark.parametrize("cout,nb,dims,shift", [(16, 2, (33, 9, 11), 0), (16, 1, (5, 3, 2), 0), (48, 1, (13, 7, 9), 1),
                                                (128, 1, (17, 5, 7), 0), (96, 3, (9, 9, 9), 0)])
def test_bias_gradient(cout, nb, dims, shift):
    import torch
    B = need_gpu()
    L = B.load()
    W, H, D = dims
    N = nb * D * H * W
    g = torch.Generator(device="cuda").manual_seed(N)
    dy = torch.randn(N * cout + 4, generator=g, device="cuda")[shift:shift + N * cout].view(N, cout)
    x, dy16 = torch.zeros(N, 16, dtype=torch.bfloat16, device="cuda"), dy.to(torch.bfloat16)
    dw, db = torch.zeros(27 * 16 * cout, device="cuda"), torch.ones(cout, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert L.lasto_nn_conv3d_wgrad_tc(nb, (ctypes.c_int * 3)(*dims), 16, cout, B._ptr(x), B._ptr(dy16), B._ptr(dy),
                                      B._ptr(dw), B._ptr(db), B._ptr(err), B._stream()) == 0
    ref = 1.0 + dy.double().sum(0)
    # FP32 sums: at most 64 terms per thread, 256 threads and N / 512 + 1 blocks one after another
    tol = (64 + 256 + N / 128 + 2) * 2.0 ** -24 * (1.0 + dy.double().abs().sum(0))
    assert bool(((db.double() - ref).abs() <= tol).all())
