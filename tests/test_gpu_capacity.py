"""How many PEs the resident kernels hold on a GB300 (152 SMs), at the edges of
what each variant of them takes.  All give the bits of the per-stage path."""
import numpy as np
import pytest

from paper_2204_01133_gb300 import workloads as W

pytestmark = pytest.mark.gpu
OPT_ARRIVAL = 3


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the counts are those of 152 SMs")
    from paper_2204_01133_gb300 import build
    build.build()


def _run(pb, u0, steps, path):
    from paper_2204_01133_gb300.api import Solver
    s = Solver(pb, u0, path=path)
    s.run(steps)
    out = s.read_state(), s.read_delays(), s.stats()
    s.close()
    return out


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("pe_size,pes", [(16, 1368), (24, 1064), (32, 760), (48, 608), (64, 304), (64, 305), (64, 456),
                                         (65, 152), (96, 152), (96, 153), (97, 152), (128, 152), (128, 153), (129, 152), (223, 100), (224, 152),
                                         (224, 153), (256, 1), (280, 456), (320, 456), (421, 304), (488, 304), (749, 152), (750, 152),
                                         (850, 152), (872, 152)])
def test_flames_on_the_persistent_path(order, pe_size, pes):
    pb, u0 = W.rns(case="flame", n=pe_size * pes, pe_size=pe_size, order=order, mode="at", k_max=3, seed=2)
    a, b = _run(pb, u0, 3, "persistent"), _run(pb, u0, 3, "stage")
    assert a[2].path == 2
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("pe_size,pes", [(64, 456), (320, 456), (872, 20)])
def test_delays_by_arrival(pe_size, pes):
    """They have no other path."""
    from paper_2204_01133_gb300.api import Solver
    pb, u0 = W.rns(case="flame", n=pe_size * pes, pe_size=pe_size, mode="at", k_max=3, seed=2)
    s = Solver(pb, u0)
    s.set_option(OPT_ARRIVAL, 1)
    s.run(5)
    assert s.stats().path == 2 and np.isfinite(s.read_state()).all()
    s.close()


@pytest.mark.parametrize("pe_size,pes", [(32, 760), (64, 384), (64, 456), (200, 456), (800, 100)])
def test_the_automatic_rule_keeps_them_resident(pe_size, pes):
    pb, u0 = W.rns(case="flame", n=pe_size * pes, pe_size=pe_size, mode="at", k_max=3, seed=2)
    assert _run(pb, u0, 2, "auto")[2].path == 2


@pytest.mark.parametrize("pe_size", [873, 900])
def test_larger_pes_are_refused(pe_size):
    from paper_2204_01133_gb300.api import AtError
    pb, u0 = W.rns(case="flame", n=pe_size * 4, pe_size=pe_size, mode="at", k_max=3, seed=2)
    with pytest.raises(AtError):
        _run(pb, u0, 1, "persistent")


@pytest.mark.parametrize("order,rk,pe_size,pes", [
    (2, "rk4", 32, 4864), (2, "rk4", 64, 4864), (2, "rk4", 128, 3648), (4, "rk4", 32, 4864), (4, "rk4", 64, 4096),
    (4, "rk4", 64, 4864), (4, "rk4", 128, 3648), (6, "rk4", 32, 4864), (6, "rk4", 64, 3648), (6, "rk4", 128, 3648),
    (2, "rk3tvd", 64, 4864), (2, "rk3tvd", 128, 3648), (2, "rk3tvd", 256, 3648), (4, "rk3tvd", 64, 4864),
    (4, "rk3tvd", 128, 3648), (6, "rk3tvd", 64, 4864), (6, "rk3tvd", 128, 3648), (2, "rk2", 128, 4864),
    (2, "rk2", 256, 3648), (4, "rk2", 64, 4864), (4, "rk2", 128, 3648), (6, "rk2", 64, 4864), (6, "rk2", 128, 2432),
    (4, "rk4", 256, 1824), (6, "rk4", 256, 1824)])
def test_advection_diffusion_in_one_launch(order, rk, pe_size, pes):
    pb, u0 = W.advdiff(n=pe_size * pes, pe_size=pe_size, order=order, rk=rk, mode="at", k_max=3, seed=3, cfl=0.01)
    a, b = _run(pb, u0, 7, "fused"), _run(pb, u0, 7, "stage")
    assert a[2].kernels_launched == 2  # the counters' reset and the kernel
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("pe_size", [96, 160, 192, 224])
@pytest.mark.parametrize("pes,order,rk", [(1, 4, "rk4"), (2, 6, "rk3tvd"), (3, 2, "rk2"), (101, 6, "rk4"), (305, 4, "rk4"),
                                          (1216, 6, "rk2"), (2500, 4, "rk4"), (6001, 6, "rk3tvd")])
def test_pes_of_any_multiple_of_32(pe_size, pes, order, rk):
    """By the automatic rule, in one launch or one a step; asked for by name the
    path takes the powers of two, as ever."""
    from paper_2204_01133_gb300.api import AtError
    pb, u0 = W.advdiff(n=pe_size * pes, pe_size=pe_size, order=order, rk=rk, mode="at", k_max=3, seed=3, cfl=0.01)
    a, b = _run(pb, u0, 7, "auto"), _run(pb, u0, 7, "stage")
    assert a[2].path == 3
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    with pytest.raises(AtError):
        _run(pb, u0, 1, "fused")


@pytest.mark.parametrize("variant", [7, 8], ids=["advection", "burgers"])
def test_batched_scalar_weno_solves_hold_the_ctas_a_batch_asks_for(variant):
    import ctypes
    from paper_2204_01133_gb300 import api
    L = api.lib()
    smem = L._Z20atk_stage_smem_bytesiii  # size_t atk_stage_smem_bytes(int pde, int Tw, int H)
    smem.restype, smem.argtypes = ctypes.c_size_t, [ctypes.c_int] * 3
    ctas = L._Z25atk_batch_max_ctas_per_smiim  # int atk_batch_max_ctas_per_sm(int variant, int block, size_t smem)
    ctas.restype, ctas.argtypes = ctypes.c_int, [ctypes.c_int, ctypes.c_int, ctypes.c_size_t]
    assert ctas(variant, 256, smem({7: 3, 8: 4}[variant], 64, 3)) >= 3


@pytest.mark.parametrize("variant,halo", [(3, 1), (4, 2)], ids=["order 2", "order 4"])
def test_batched_flames_hold_the_ctas_a_batch_asks_for(variant, halo):
    import ctypes
    from paper_2204_01133_gb300 import api
    L = api.lib()
    smem, ctas = L._Z20atk_stage_smem_bytesiii, L._Z25atk_batch_max_ctas_per_smiim
    smem.restype, smem.argtypes = ctypes.c_size_t, [ctypes.c_int] * 3
    ctas.restype, ctas.argtypes = ctypes.c_int, [ctypes.c_int, ctypes.c_int, ctypes.c_size_t]
    assert ctas(variant, 256, smem(1, 64, halo)) >= 3
