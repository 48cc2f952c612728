"""The convolution kernels that put several taps side by side in the tensor cores' N, at the
edges of their tiles: grids 16 to 128 (x-rows of half a warp to four warps, whose neighbours
cross warps from 64 on), one to four tiles per block, output channels around the tile widths
16, 32, 48, 64 and over several tiles, one to eight input-channel chunks.

Forward and input gradient (lbm_nn_conv3d_bf16): every element within 1e-6 K sum |x w| of the
FP64 sum (FP32 accumulation of K = 27 cin BF16 products), plus 2^-8 of the value for the BF16
output; the bounds of test_gpu_nn.py."""
import pytest

pytestmark = pytest.mark.gpu


def _shifted(X, B, n, cin):
    import torch
    P = torch.zeros((B, n + 2, n + 2, n + 2, cin), dtype=torch.float64, device="cuda")
    P[:, 1:-1, 1:-1, 1:-1] = X.double().reshape(B, n, n, n, cin)
    for tap in range(27):
        kz, ky, kx = tap // 9, tap // 3 % 3, tap % 3
        yield tap, P[:, kz:kz + n, ky:ky + n, kx:kx + n].reshape(-1, cin)


CONV = [(1, 16, 32, 8), (3, 16, 96, 16), (1, 16, 256, 72), (2, 16, 64, 80), (1, 32, 32, 48), (2, 32, 96, 24),
        (1, 32, 64, 200), (1, 64, 64, 56), (2, 64, 32, 17), (1, 128, 32, 32), (1, 128, 32, 96)]


@pytest.mark.parametrize("B,n,cin,cout", CONV)
def test_convolution_at_the_edges_of_its_tiles(B, n, cin, cout):
    import torch
    from paper_1710_04751_gb300 import net
    g = torch.Generator(device="cuda").manual_seed(n + cin + cout)
    X = torch.randn((B, n ** 3, cin), generator=g, device="cuda").to(torch.bfloat16)
    ldw = (27 * cin + 7) // 8 * 8 + 8
    W = torch.full((cout, ldw), 3.0, device="cuda", dtype=torch.bfloat16)  # past 27 cin: not read
    W[:, :27 * cin] = torch.randn((cout, 27 * cin), generator=g, device="cuda") / (27 * cin) ** 0.5
    bias = 0.1 * torch.randn(cout, generator=g, device="cuda")
    y = torch.zeros((B * n ** 3, cout), dtype=torch.float64, device="cuda")
    mag = torch.zeros_like(y)
    for tap, S in _shifted(X, B, n, cin):
        w = W[:, tap * cin:(tap + 1) * cin].double().T
        y += S @ w
        mag += S.abs() @ w.abs()
    e = 1e-6 * 27 * cin * mag + 1e-30
    out = torch.full((B * n ** 3, cout), float("nan"), device="cuda")
    net.conv3d_bf16(X, n, W, out, mode=net.CONV_F32)
    assert ((out.double() - y).abs() <= e).all()
    outb = torch.full((B * n ** 3, cout), float("nan"), dtype=torch.bfloat16, device="cuda")
    net.conv3d_bf16(X, n, W, outb, mode=net.CONV_BIAS_RELU_BF16, bias=bias)
    ref = torch.relu(y + bias.double())
    assert ((outb.double() - ref).abs() <= 2.0 ** -8 * (ref + e) + e).all()
