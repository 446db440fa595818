"""The choices the library makes by size: PEs per CTA of the multi-step
advection-diffusion kernel, window lengths of the per-stage WENO kernels,
windows per CTA of the flame, batched stages with one and with several RK
schemes.  None of them may change a bit."""
import numpy as np
import pytest

from paper_2204_01133_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2204_01133_gb300 import build
    build.build()


def _run(pb, u0, steps, path):
    from paper_2204_01133_gb300.api import Solver
    s = Solver(pb, u0, path=path)
    s.run(steps)
    out = s.read_state(), s.read_delays()
    s.close()
    return out


def _same(a, b):
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("pe_size,pes", [(64, 303), (64, 305), (32, 609), (128, 2431), (256, 152), (64, 2500)])
def test_pes_per_cta_of_the_multi_step_kernel(pe_size, pes):
    pb, u0 = W.advdiff(n=pe_size * pes, pe_size=pe_size, mode="at", k_max=3, seed=3, cfl=0.05)
    _same(_run(pb, u0, 25, "stage"), _run(pb, u0, 25, "fused"))


@pytest.mark.parametrize("pes,order,rk", [(1, 4, "rk4"), (2, 6, "rk3tvd"), (101, 6, "rk3tvd"), (305, 4, "rk4"),
                                          (2500, 4, "rk4"), (6001, 6, "rk4")])
def test_pes_of_96_points(pes, order, rk):
    """By the automatic rule (resident and one launch per step); the path asked
    for by name still takes the sizes it took."""
    from paper_2204_01133_gb300.api import AtError
    pb, u0 = W.advdiff(n=96 * pes, pe_size=96, order=order, rk=rk, mode="at", k_max=3, seed=3, cfl=0.01)
    _same(_run(pb, u0, 25, "stage"), _run(pb, u0, 25, "auto"))
    with pytest.raises(AtError):
        _run(pb, u0, 1, "fused")


@pytest.mark.parametrize("pe_size,pes", [(512, 2), (480, 7), (480, 128), (96, 3), (1024, 60), (720, 300), (16, 5),
                                         (1021, 2), (22, 9)])
def test_window_lengths_of_the_weno_kernels(pe_size, pes):
    pb, u0 = W.adv_weno(n=pe_size * pes, pe_size=pe_size, mode="at", k_max=3, seed=4)
    _same(_run(pb, u0, 12, "stage"), _run(pb, u0, 12, "fused"))
    if pe_size * pes >= 960:
        pb, u0 = W.detonation(n=pe_size * pes, pe_size=pe_size, mode="at", k_max=4, seed=4)
        _same(_run(pb, u0, 6, "stage"), _run(pb, u0, 6, "fused"))


@pytest.mark.parametrize("pe_size,pes", [(64, 13), (64, 1300), (64, 1301), (32, 2432), (48, 1218), (256, 700)])
def test_windows_per_cta_of_the_flame(pe_size, pes):
    pb, u0 = W.rns(case="flame", n=pe_size * pes, pe_size=pe_size, mode="at", k_max=4, seed=5)
    _same(_run(pb, u0, 6, "stage"), _run(pb, u0, 6, "fused"))


@pytest.mark.parametrize("rks", [("rk4", "rk4"), ("rk4", "rk3tvd"), ("rk3tvd", "rk3tvd")])
def test_batched_stages_with_one_and_two_schemes(rks):
    from paper_2204_01133_gb300 import batch
    inst = []
    for i, rk in enumerate(rks):
        pb, u0 = W.rns(case="flame", n=64 * (9 + i), pe_size=64, mode="at", k_max=3, seed=i, instance=i)
        inst.append((dict(pb, rk=rk), u0))
        pb, u0 = W.detonation(n=2048, pe_size=512, mode="at", k_max=4, seed=i)
        inst.append((dict(pb, rk=rk, instance=7 + i), u0))
    b = batch.Batch(len(inst))
    b.set_config(batch.FLAT, 128, 1, True)
    for i, (pb, u0) in enumerate(inst):
        b.bind(i, pb, u0, 14)
    b.run(14)
    for i, (pb, u0) in enumerate(inst):
        assert np.array_equal(b.state(i).cpu().numpy(), _run(pb, u0, 14, "stage")[0])
    b.close()
