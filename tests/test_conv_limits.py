"""What lbm_nn_conv3d_bf16 and lbm_nn_conv3d_wgrad_bf16 refuse before they launch anything (the
operands of those calls are addresses that nothing may read), and that unaligned bases which the
kernels write element by element are still taken."""
import ctypes

import pytest

from paper_1710_04751_gb300 import lbm as binding
from paper_1710_04751_gb300 import net

BASE = 1 << 40


def conv(batch=1, n=16, cin=32, cout=32, X=BASE, W=BASE, bias=BASE, out=BASE, mode=net.CONV_F32):
    p = [ctypes.c_void_p(v) for v in (X, W, bias, out)]
    return net._lib().lbm_nn_conv3d_bf16(p[0], batch, n, cin, p[1], 27 * cin, cout, p[2], p[3], mode, None)


# rows = batch n^3 in 32 bits, up to the end of the last tile: at 2^31 and beyond the start of a tile,
# and with it the address of a store, would wrap
@pytest.mark.parametrize("batch,n", [(1 << 19, 16), ((1 << 19) + 1, 16), (1 << 16, 32), (1 << 13, 64), (8193, 64),
                                     (1 << 10, 128), (1025, 128), (2049, 128), (128, 256), (1 << 28, 2),
                                     ((1 << 28) - 1, 2), ((1 << 31) - 1, 256)])
@pytest.mark.parametrize("mode", [net.CONV_F32, net.CONV_BIAS_RELU_BF16])
def test_more_rows_than_32_bits_hold_are_refused(batch, n, mode):
    assert conv(batch=batch, n=n, mode=mode) == binding.LBM_EINVAL


def wgrad(cout=32, n=64, X=BASE, dZ=BASE, ws=BASE, dWT=BASE):
    p = [ctypes.c_void_p(v) for v in (X, dZ, ws, dWT)]
    return net._lib().lbm_nn_conv3d_wgrad_bf16(p[0], 1, n, 32, p[1], cout, 896, p[2], 8 * 896 * cout, 8, p[3], None)


# the kernels store 16 bytes at a time where the rows hold a multiple of 8 values
@pytest.mark.parametrize("n", [8, 16, 64])
@pytest.mark.parametrize("mode,cout,bases", [
    (net.CONV_F32, 32, dict(out=BASE + 4)), (net.CONV_F32, 8, dict(out=BASE + 8)), (net.CONV_F32, 17, dict(out=BASE + 2)),
    (net.CONV_BIAS_RELU_BF16, 32, dict(out=BASE + 2)), (net.CONV_BIAS_RELU_BF16, 24, dict(out=BASE + 8)),
    (net.CONV_BIAS_RELU_BF16, 17, dict(out=BASE + 1)), (net.CONV_BIAS_RELU_BF16, 32, dict(bias=BASE + 2)),
    (net.CONV_F32, 32, dict(X=BASE + 8)), (net.CONV_F32, 32, dict(W=BASE + 8))])
def test_unaligned_bases_of_a_convolution_are_refused(n, mode, cout, bases):
    assert conv(n=n, mode=mode, cout=cout, **bases) == binding.LBM_EINVAL


@pytest.mark.parametrize("n", [8, 64])
@pytest.mark.parametrize("cout,bases", [(32, dict(ws=BASE + 4)), (16, dict(ws=BASE + 8)), (24, dict(ws=BASE + 4)),
                                        (256, dict(ws=BASE + 8)), (8, dict(ws=BASE + 2)), (32, dict(dWT=BASE + 2)),
                                        (32, dict(X=BASE + 8)), (32, dict(dZ=BASE + 8))])
def test_unaligned_bases_of_a_weight_gradient_are_refused(n, cout, bases):
    assert wgrad(n=n, cout=cout, **bases) == binding.LBM_EINVAL


# operands of -1, 0 and 1: every sum is exact, whatever its order
@pytest.mark.gpu
@pytest.mark.parametrize("n", [8, 16, 64])
@pytest.mark.parametrize("mode", [net.CONV_F32, net.CONV_BIAS_RELU_BF16])
def test_output_on_an_element_boundary(n, mode):
    import torch
    cin, cout = 32, 17
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randint(-1, 2, (1, n ** 3, cin), generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randint(-1, 2, (cout, 27 * cin), generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randint(-3, 4, (cout,), generator=g, device="cuda").float()
    outs = []
    for first in (0, 1):
        buf = torch.full((n ** 3 * cout + 16,), -7.0, device="cuda",
                         dtype=torch.float32 if mode == net.CONV_F32 else torch.bfloat16)
        out = buf[first:first + n ** 3 * cout].view(n ** 3, cout)
        net.conv3d_bf16(X, n, W, out, mode=mode, bias=bias)
        assert (buf[:first] == -7).all() and (buf[first + n ** 3 * cout:] == -7).all()
        outs.append(out.clone())
    assert torch.equal(*outs)


@pytest.mark.gpu
def test_workspace_on_an_element_boundary():
    import torch
    n, cin, cout, Kp, splits = 64, 32, 8, 896, 8
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randint(-1, 2, (1, n ** 3, cin), generator=g, device="cuda").to(torch.bfloat16)
    dZ = torch.randint(-1, 2, (n ** 3, cout), generator=g, device="cuda").to(torch.bfloat16)
    grads = []
    for first in (0, 1):
        ws = torch.empty(splits * Kp * cout + 4, device="cuda")[first:]
        dWT = torch.zeros(Kp * cout + 4, device="cuda")[first:first + Kp * cout]
        net._check(net._lib().lbm_nn_conv3d_wgrad_bf16(X.data_ptr(), 1, n, cin, dZ.data_ptr(), cout, Kp, ws.data_ptr(),
                                                       splits * Kp * cout, splits, dWT.data_ptr(), net._stream(dWT)))
        grads.append(dWT.clone())
    assert torch.equal(*grads)
