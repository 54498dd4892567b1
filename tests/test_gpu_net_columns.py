"""The column-march convolution and weight gradient at the edges of their
tiling, against the FP64 network oracle: ragged x, y and z, planes fewer than a
column's, several columns per CTA with the weights resident and reloaded chunk
by chunk (one and two weight buffers), an upsampled second source.

Tolerances as for the other convolution shapes: both sides use the same BF16
values, so an FP32 output differs by FP32 accumulation only (1e-5 of the
largest value), a BF16 output by one BF16 rounding more (2^-8)."""
import numpy as np
import pytest

from oracle import net_oracle as no

pytestmark = pytest.mark.gpu

CASES = [  # (batch, grid, c0, c1, cout)
    (1, (1, 2, 3), 16, 0, 16),       # smaller than a halo
    (1, (9, 20, 12), 32, 0, 16),     # last column one plane deep, ragged x and y
    (2, (5, 17, 9), 16, 0, 32),
    (3, (22, 32, 64), 48, 32, 48),   # several columns per CTA, two weight buffers
    (2, (17, 16, 24), 64, 0, 64),    # column of one plane at the end
    (1, (10, 16, 16), 112, 0, 80),   # the widest output of the march
    (1, (8, 16, 8), 16, 0, 96),      # beyond it: the brick kernels
    (12, (16, 32, 32), 16, 32, 16),  # more columns than CTAs, weights resident
]


@pytest.mark.parametrize("case", CASES)
def test_columns(case):
    import torch
    from paper_2110_00733_gb300 import build, net
    build.build()
    net.load_library()
    B, g, c0, c1, cout = case
    rng = np.random.default_rng(sum(g) + c0 + cout)
    rnd = lambda shape, s=1.0: no.bf16(rng.standard_normal(shape) * s)  # noqa: E731
    dev = lambda a: torch.tensor(np.asarray(a, dtype=np.float32), device="cuda").to(torch.bfloat16).contiguous()  # noqa: E731
    x0, W, G = rnd((B,) + g + (c0,)), rnd((27, cout, c0 + c1), 0.1), rnd((B,) + g + (cout,))
    x1 = rnd((B,) + tuple(v // 2 for v in g) + (c1,)) if c1 else None
    bias = rng.standard_normal(cout).astype(np.float32)
    xin = x0 if x1 is None else np.concatenate([x0, no.upsample2(x1)], axis=-1)
    # the oracle's convolution, one voxel sum per tap (27 matrix products)
    ref = np.broadcast_to(bias.astype(np.float64), (B,) + g + (cout,)).copy()
    dref = np.zeros((27, cout, c0 + c1))
    for t in range(27):
        d = (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)
        xs = np.roll(xin, tuple(-v for v in d), (1, 2, 3)).reshape(-1, c0 + c1)
        ref += (xs @ W[t].T).reshape(ref.shape)
        dref[t] = G.reshape(-1, cout).T @ xs
    s0, s1, Wt, bt = dev(x0), dev(x1) if c1 else None, dev(W), torch.tensor(bias, device="cuda")
    o = torch.empty((B,) + g + (cout,), dtype=torch.float32, device="cuda")
    net.conv3d(g, s0, Wt, cout, src1=s1, bias=bt, out=o)
    assert np.abs(o.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    h = torch.empty((B,) + g + (cout,), dtype=torch.bfloat16, device="cuda")
    net.conv3d(g, s0, Wt, cout, src1=s1, bias=bt, relu=True, out=h)
    r = np.maximum(ref, 0)
    assert np.abs(h.float().cpu().numpy() - r).max() <= 2.0 ** -8 * r.max()
    if cout <= 64:
        dW = torch.empty(27, cout, c0 + c1, device="cuda")
        net.conv3d_wgrad(g, dev(G), s0, dW, src1=s1)
        assert np.abs(dW.cpu().numpy() - dref).max() <= 1e-5 * np.abs(dref).max()
