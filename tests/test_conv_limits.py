"""What lbm_nn_conv3d_bf16 and lbm_nn_conv3d_wgrad_bf16 refuse before they launch anything: the
operands here are addresses that nothing may read."""
import ctypes

import pytest

from paper_1710_04751_gb300 import lbm as binding
from paper_1710_04751_gb300 import net

BASE = 1 << 40


def conv(batch=1, n=16, cin=32, cout=32, X=BASE, W=BASE, out=BASE, mode=net.CONV_F32):
    p = [ctypes.c_void_p(v) for v in (X, W, BASE, out)]
    return net._lib().lbm_nn_conv3d_bf16(p[0], batch, n, cin, p[1], 27 * cin, cout, p[2], p[3], mode, None)


# rows = batch n^3 in 32 bits, up to the end of the last tile: at 2^31 and beyond the start of a tile,
# and with it the address of a store, would wrap
@pytest.mark.parametrize("batch,n", [(1 << 19, 16), ((1 << 19) + 1, 16), (1 << 16, 32), (1 << 13, 64), (8193, 64),
                                     (1 << 10, 128), (1025, 128), (2049, 128), (128, 256), (1 << 28, 2),
                                     ((1 << 28) - 1, 2), ((1 << 31) - 1, 256)])
@pytest.mark.parametrize("mode", [net.CONV_F32, net.CONV_BIAS_RELU_BF16])
def test_more_rows_than_32_bits_hold_are_refused(batch, n, mode):
    assert conv(batch=batch, n=n, mode=mode) == binding.LBM_EINVAL
