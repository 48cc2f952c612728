"""The convolutions and the weight gradient on operands of -1, 0 and 1: every partial sum is a whole
number far below 2^24, so the FP32 result is exact whatever the order, the split or the
truncation of the sums, and is compared for equality.  A tap, a block of channels, a row at a
tile's halo or a voxel at the seam of two ranges that is lost or taken twice shows, however
long the sum is."""
import pytest

pytestmark = pytest.mark.gpu


def _operand(g, *shape):
    import torch
    return torch.randint(-1, 2, shape, generator=g, device="cuda").to(torch.bfloat16)


def _shifted(X, B, n, cin):
    import torch
    P = torch.zeros((B, n + 2, n + 2, n + 2, cin), device="cuda")
    P[:, 1:-1, 1:-1, 1:-1] = X.reshape(B, n, n, n, cin)
    for tap in range(27):
        kz, ky, kx = tap // 9, tap // 3 % 3, tap % 3
        yield tap, P[:, kz:kz + n, ky:ky + n, kx:kx + n].reshape(-1, cin)


CONV = [(3, 2, 32, 8), (2, 4, 64, 40), (3, 8, 96, 130), (1, 16, 256, 72), (3, 16, 96, 16), (2, 16, 64, 80), (5, 16, 32, 256),
        (1, 32, 32, 48), (2, 32, 96, 24), (1, 32, 64, 200), (2, 64, 96, 32), (1, 64, 32, 96), (2, 64, 32, 17),
        (1, 128, 32, 32), (1, 128, 64, 96), (1, 256, 32, 8)]


@pytest.mark.parametrize("B,n,cin,cout", CONV)
def test_convolution_of_whole_numbers(B, n, cin, cout):
    import torch
    from paper_1710_04751_gb300 import net
    g = torch.Generator(device="cuda").manual_seed(n + cin + cout)
    X, W = _operand(g, B, n ** 3, cin), _operand(g, cout, (27 * cin + 7) // 8 * 8)
    bias = torch.randint(-9, 10, (cout,), generator=g, device="cuda").float()
    y = torch.zeros((B * n ** 3, cout), device="cuda")
    for tap, S in _shifted(X, B, n, cin):
        y += S @ W[:, tap * cin:(tap + 1) * cin].float().T
    out = torch.full_like(y, float("nan"))
    net.conv3d_bf16(X, n, W, out, mode=net.CONV_F32)
    assert torch.equal(out, y)
    outb = torch.full_like(y, float("nan"), dtype=torch.bfloat16)
    net.conv3d_bf16(X, n, W, outb, mode=net.CONV_BIAS_RELU_BF16, bias=bias)
    assert torch.equal(outb, torch.relu(y + bias).to(torch.bfloat16))


WGRAD = [(3, 2, 32, 8, 1), (2, 8, 64, 48, 3), (4, 16, 64, 48, 5), (16, 16, 128, 64, 5), (17, 16, 128, 8, 3), (2, 32, 128, 40, 3),
         (3, 32, 96, 64, 7), (1, 32, 256, 24, 1), (2, 32, 64, 128, 9), (1, 64, 32, 24, 4), (2, 64, 96, 32, 14), (1, 64, 96, 48, 11),
         (1, 64, 32, 32, 43), (1, 128, 32, 8, 9), (1, 128, 32, 32, 43), (1, 256, 32, 8, 8), (1, 256, 32, 32, 43), (16, 16, 128, 64, 26), (3, 32, 96, 64, 14), (1, 64, 32, 24, 43),
         (1, 64, 96, 48, 14), (1, 128, 32, 8, 43), (1, 256, 32, 8, 43)]


@pytest.mark.parametrize("B,n,cin,cout,splits", WGRAD)
def test_weight_gradient_of_whole_numbers(B, n, cin, cout, splits):
    import torch
    from paper_1710_04751_gb300 import net
    g = torch.Generator(device="cuda").manual_seed(B + n + cin + cout)
    X, dZ = _operand(g, B, n ** 3, cin), _operand(g, B * n ** 3, cout)
    Kp = (27 * cin + 63) // 64 * 64
    dWT = torch.full((Kp, cout), 3.0, device="cuda")
    net.conv3d_wgrad_bf16(X, n, dZ, dWT, splits=splits)
    Z = dZ.float()
    for tap, S in _shifted(X, B, n, cin):
        assert torch.equal(dWT[tap * cin:(tap + 1) * cin], 3 + S.T @ Z), tap
    assert (dWT[27 * cin:] == 3).all()
