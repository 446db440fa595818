"""Launch shapes chosen on the host by size (no GPU is needed to ask)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def block():
    from paper_2204_01133_gb300 import api, build
    build.build()
    f = api.lib()._Z15atk_stage_blockii  # int atk_stage_block(int pde, int Tw)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int, ctypes.c_int]
    return f


EULER, ADV_WENO = 2, 3


@pytest.mark.parametrize("tw,threads", [(16, 96), (60, 256), (63, 256), (64, 128), (128, 128), (191, 128), (192, 256),
                                        (251, 256), (509, 256), (1021, 256)])
def test_threads_of_a_detonation_window(block, tw, threads):
    assert block(EULER, tw) == threads


@pytest.mark.parametrize("tw,threads", [(16, 32), (128, 160), (255, 256), (1021, 256)])
def test_threads_of_a_scalar_weno_window(block, tw, threads):
    assert block(ADV_WENO, tw) == threads


@pytest.mark.parametrize("tw,windows,threads", [(64, 1, 256), (64, 608, 256), (64, 609, 64), (16, 608, 128), (16, 609, 32),
                                                (32, 100, 128), (48, 608, 256), (128, 300, 256), (256, 40, 256),
                                                (256, 5000, 256), (1021, 4, 256)])
def test_threads_of_a_flame_window(tw, windows, threads):
    """On 152 SMs."""
    from paper_2204_01133_gb300 import api, build
    build.build()
    f = api.lib()._Z17atk_flame_threadsili  # int atk_flame_threads(int Tw, int64_t windows, int sms)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    assert f(tw, windows, 152) == threads
