"""The weight-gradient kernel that puts nine taps side by side in the tensor cores' N (grids from
16^3, up to 64 output channels, voxels x input channels >= 2^23), at the edges of its tiles: blocks
of four, two and one x-rows and of half an x-row, 8 to 64 output channels, the last M tile with
one, two and four of its channel groups in use, ranges that start inside a plane, one range and
several, single CTAs and pairs.

Each element against the FP64 sum.  A chain adds L/16 partial products to an FP32 sum that its
tensor core truncates: an error of at most 2^-22 of the running sum each, which for random
operands of unit and 1/64 variance stays below 6 sqrt(L)/64."""
import pytest

from tests.test_gpu_conv_taps import _shifted

pytestmark = pytest.mark.gpu

CASES = [(16, 16, 128, 64, 5), (17, 16, 128, 8, 3), (2, 32, 128, 40, 3), (3, 32, 96, 64, 7), (1, 32, 256, 24, 1),
         (1, 64, 32, 24, 4), (1, 64, 96, 48, 11), (1, 128, 32, 8, 9)]


@pytest.mark.parametrize("B,n,cin,cout,splits", CASES)
def test_nine_tap_weight_gradient(B, n, cin, cout, splits):
    import torch
    from paper_1710_04751_gb300 import net
    g = torch.Generator(device="cuda").manual_seed(B + n + cin + cout)
    M = B * n ** 3
    X = torch.randn((B, n ** 3, cin), generator=g, device="cuda").to(torch.bfloat16)
    dZ = (torch.randn((M, cout), generator=g, device="cuda") / 64).to(torch.bfloat16)
    Kp = (27 * cin + 63) // 64 * 64
    dWT = torch.zeros((Kp, cout), device="cuda")
    net.conv3d_wgrad_bf16(X, n, dZ, dWT, splits=splits)
    ref = torch.zeros((27 * cin, cout), dtype=torch.float64, device="cuda")
    for tap, S in _shifted(X, B, n, cin):
        ref[tap * cin:(tap + 1) * cin] = S.T @ dZ.double()
    L = 1.15 * M / splits + 64
    bound = splits * L / 16 * 2.0 ** -22 * 6 * L ** 0.5 / 64 + splits * 2.0 ** -23 * ref.abs()
    assert ((dWT[:27 * cin].double() - ref).abs() <= bound).all()
    assert (dWT[27 * cin:] == 0).all()
