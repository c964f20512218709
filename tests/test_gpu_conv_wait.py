"""A convolution block whose bounded wait runs out: it leaves the result alone, waits for its own
copies and matrix instructions, gives its tensor memory back and sets the error word; the calls that
follow find all of the tensor memory and give the right sums."""
import ctypes

import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


# rows that the padded sequence takes, and rows beyond it
@pytest.mark.parametrize("which,cin,cout,dims", [(0, 64, 64, (33, 33, 33)), (0, 48, 16, (33, 33, 33)), (0, 48, 32, (1000, 9, 9)),
                                                 (1, 64, 64, (33, 33, 33)), (1, 48, 16, (33, 33, 33)), (1, 32, 32, (1000, 9, 9))])
def test_wait_that_runs_out(which, cin, cout, dims):
    import torch
    B = need_gpu()
    L = B.load()
    d3 = (ctypes.c_int * 3)(*dims)
    N = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cuda").manual_seed(which)
    x = torch.randn(N, cin, generator=g, device="cuda").bfloat16()
    m = torch.randn(*((27, cin, cout) if which == 0 else (N, cout)), generator=g, device="cuda").bfloat16()
    size = (N, cout) if which == 0 else (27, cin, cout)

    def call():
        out, err = torch.zeros(size, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        if which == 0:
            st = L.lasto_nn_conv3d_fwd_tc(1, d3, cin, cout, B._ptr(x), B._ptr(m), None, 0, B._ptr(out), cout, 0, None, 0, 0,
                                          B._ptr(err), B._stream())
        else:
            st = L.lasto_nn_conv3d_wgrad_tc(1, d3, cin, cout, B._ptr(x), B._ptr(m), None, B._ptr(out), None, B._ptr(err),
                                            B._stream())
        assert st == 0
        return out, err

    before, e0 = call()
    out, err = torch.full(size, 3.0, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(20):      # (tensor memory that was not given back would stop the second round of blocks)
        assert L.lasto_selftest_conv_wait(which, 1, d3, cin, cout, B._ptr(x), B._ptr(m), B._ptr(out), B._ptr(err),
                                          B._stream()) == 0
    after, e1 = call()
    torch.cuda.synchronize()
    assert int(err.item()) == 1 and bool((out == 3.0).all())
    assert int(e0.item()) == 0 and int(e1.item()) == 0
    if which == 0:
        assert torch.equal(before, after)
    else:                    # (FP32 atomics: the order of the blocks' sums; 2^-24 for each of some 40)
        assert float((before - after).abs().max()) <= 40 * 2.0 ** -24 * float(before.abs().max())
