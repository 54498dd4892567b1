"""The network's step-level entry points refuse shapes before they touch a device or
any of the arrays (no compute calls: this runs without a GPU)."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def net():
    from paper_2110_00733_gb300 import build, net
    build.build()
    net.load_library()
    return net


@pytest.mark.parametrize("grid, cout, c0, c1", [
    ((5, 4, 4), 16, 16, 16), ((4, 7, 8), 32, 16, 32), ((6, 8, 9), 64, 0, 16),   # an odd size with a second source
    ((4, 4, 4), 0, 16, 0), ((4, 4, 4), -16, 16, 0), ((4, 4, 4), 80, 16, 0), ((4, 4, 4), 24, 16, 0),
    ((4, 4, 4), 16, 8, 0), ((4, 4, 4), 16, 16, 24), ((4, 4, 4), 16, 0, 0), ((4, 4, 4), 16, -16, 32),
])
def test_weight_gradient_refuses(net, grid, cout, c0, c1):
    buf = np.zeros(64, np.float32)
    p = ctypes.c_void_p(buf.ctypes.data)
    lib = net.load_library()
    rc = lib.hom_net_conv3d_wgrad(1, (ctypes.c_int * 3)(*grid), p, cout, p, c0, p, c1, p, None)
    from paper_2110_00733_gb300 import hom
    assert rc == hom.HOM_EINVAL, lib.hom_net_last_error()
    assert b"even with a second source" in lib.hom_net_last_error()


def test_convolution_without_a_device_does_not_blame_the_shape(net):
    """Without a device there is no error word for the kernel's waits: HOM_ENOMEM, and before any launch."""
    import torch
    if torch.cuda.is_available():
        pytest.skip("host buffers stand in for device ones")
    from paper_2110_00733_gb300 import hom
    buf = np.zeros(4096, np.float32)
    p = ctypes.c_void_p(buf.ctypes.data)
    lib = net.load_library()
    rc = lib.hom_net_conv3d(1, (ctypes.c_int * 3)(1, 1, 1), p, 16, None, 0, p, None, 0, 16, p, 1, None)
    assert rc == hom.HOM_ENOMEM and b"error word" in lib.hom_net_last_error()
