"""Weight gradient of wide layers over many voxels.  A tensor-core FP32 accumulator that takes more of
them is further off, so the voxels of one split are bounded whatever the channels.  Tolerance as for the
other shapes, 1e-5 of the largest value: at the bound of 4096 voxels (256 products of 16, each at most
2^-23 of the accumulator) a sum that grows evenly is off by 128 x 2^-23 = 1.5e-5 of itself at most, by half
of that on average, and these gradients, of output gradients of both signs, grow more slowly than evenly."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch, g, cin, cout", [(4, (64, 64, 64), 64, 64), (2, (40, 72, 96), 48, 64),
                                                 (1, (96, 80, 96), 64, 32)])
def test_against_64_bits(batch, g, cin, cout):
    import torch
    from paper_2110_00733_gb300 import build, net
    build.build()
    net.load_library()
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((batch,) + g + (cin,), generator=gen, device="cuda").relu().bfloat16()
    G = torch.randn((batch,) + g + (cout,), generator=gen, device="cuda").bfloat16()
    dW = torch.empty(27, cout, cin, device="cuda")
    net.conv3d_wgrad(g, G, x, dW)
    Gd = G.double().reshape(-1, cout)
    for t in range(27):
        d = (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)
        ref = Gd.T @ torch.roll(x, tuple(-v for v in d), (1, 2, 3)).double().reshape(-1, cin)
        assert float((dW[t] - ref).abs().max()) <= 1e-5 * float(ref.abs().max())
