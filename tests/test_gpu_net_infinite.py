"""Weight gradient of activations or output gradients that overflowed, on grids that the kernel's tiles
(8 planes, 16 rows, 8 columns) do not fill: positions beyond the grid add nothing, not 0 times infinity.
Everything is 1 except one infinite value, so dW is +infinity over that channel's 27 taps times 16 and
the number of voxels elsewhere (exact in FP32)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [(8, 16, 8), (8, 8, 16), (1, 1, 1), (5, 6, 9), (5, 17, 12), (9, 20, 12), (2, 3, 7)])
@pytest.mark.parametrize("where", ["x", "G"])
def test_one_infinite_value(g, where):
    import torch
    from paper_2110_00733_gb300 import build, net
    build.build()
    net.load_library()
    x, G = (torch.ones((2,) + g + (16,), device="cuda").bfloat16() for _ in range(2))
    (x if where == "x" else G)[1, 0, g[1] - 1, 0, 3] = float("inf")
    dW = torch.empty(27, 16, 16, device="cuda")
    net.conv3d_wgrad(g, G, x, dW)
    ref = np.full((27, 16, 16), 2.0 * np.prod(g))
    if where == "x":
        ref[:, :, 3] = np.inf
    else:
        ref[:, 3, :] = np.inf
    assert np.array_equal(dW.cpu().numpy(), ref)
