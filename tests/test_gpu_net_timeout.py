"""A tensor-core kernel whose bounded wait gave up has set the error word; the call that ran it says
so and clears it.  The word is set from the host here, as the kernel would: nothing waits."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2110_00733_gb300 import build, hom, net
    build.build()
    lib = net.load_library()
    word = getattr(lib, "_ZN4hnet19conv3_tc_error_wordEv")   # int *hnet::conv3_tc_error_word()
    word.restype = ctypes.POINTER(ctypes.c_int)
    word.argtypes = []
    return torch, hom, net, word


def calls(torch, net):
    g = (4, 16, 8)
    x = torch.ones((1,) + g + (16,), device="cuda").bfloat16()
    W = torch.ones(27, 16, 16, device="cuda").bfloat16()
    y, dW = torch.empty_like(x), torch.empty(27, 16, 16, device="cuda")
    return {"conv3d": lambda: net.conv3d(g, x, W, 16, out=y), "conv3d_wgrad": lambda: net.conv3d_wgrad(g, x, x, dW)}


@pytest.mark.parametrize("name", ["conv3d", "conv3d_wgrad"])
def test_the_call_reports_its_timeout(env, name):
    torch, hom, net, word = env
    call = calls(torch, net)[name]
    call()
    word()[0] = 1
    with pytest.raises(Exception) as e:
        call()
    assert e.value.code == hom.HOM_ETIMEOUT
    assert word()[0] == 0
    call()


def test_another_devices_timeout_is_left_to_it(env):
    """Each device has its own word (host memory: no second device is needed to hold one)."""
    torch, hom, net, word = env
    of = getattr(net.load_library(), "_ZN4hnet22conv3_tc_error_word_ofEi")   # int *hnet::conv3_tc_error_word_of(int)
    of.restype, of.argtypes = ctypes.POINTER(ctypes.c_int), [ctypes.c_int]
    here = torch.cuda.current_device()
    assert ctypes.addressof(of(here).contents) == ctypes.addressof(word().contents)
    other = of(here + 1)
    other[0] = 1
    for call in calls(torch, net).values():
        call()
    assert other[0] == 1
    other[0] = 0
