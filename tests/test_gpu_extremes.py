"""Inputs at the ends of what the kernels' integer arithmetic takes, against
the oracle with the per-variable bounds of parity.py."""
import numpy as np
import pytest

from paper_2204_01133_gb300 import workloads as W
from parity import TOL_STEP, check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2204_01133_gb300 import build
    build.build()


@pytest.mark.parametrize("amp,eps", [(1e7, 1e-30), (1e12, 1e-20), (1e20, 1e-6)])
def test_weno_front_beside_a_uniform_state(amp, eps):
    """Zero smoothness indicators: eps alone is their denominators.  One step
    against the oracle; later ones would compare rounding (the oracle moves by
    4e-7 in 20 steps when its input moves by 1e-15), so they are held to be
    finite and the same on both paths."""
    import oracle
    from paper_2204_01133_gb300.api import Solver
    pb, u0 = W.adv_weno(n=1024, pe_size=64, eps=eps, mode="at", k_max=3, seed=2)
    u0 = amp * (np.arange(1024) // 100 % 2 == 1).astype(np.float64)[None, :]
    o = oracle.Oracle(pb, u0)
    assert o.run(1) == 0
    out = []
    for path in ("stage", "fused"):
        s = Solver(pb, u0, path=path)
        s.run(1)
        check(pb, s.read_state(), o.state(), TOL_STEP, "front of %g, eps %g, %s" % (amp, eps, path))
        s.run(19)
        out.append(s.read_state())
        s.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("which", [5, 6], ids=["reciprocal", "root"])
def test_reciprocal_and_root_outside_the_normal_range(which):
    """Each by itself: no wrong finite value, and the signs of zeros and of
    infinities as in IEEE arithmetic where a value is defined (the probe test of
    the normal range checks only part of them)."""
    import ctypes
    import os
    import torch
    from paper_2204_01133_gb300 import build
    L = ctypes.CDLL(os.path.join(os.path.dirname(build.__file__), "libat_probe.so"))
    L.at_probe_fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int]
    x = np.array([0.0, np.inf, np.nan, -1.0, 1e-310, 5e-324, 2.0 ** -1022, 1.7e308, 2.0 ** 1022])
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    assert L.at_probe_fn(xd.data_ptr(), yd.data_ptr(), xd.numel(), which) == 0
    zero, inf, nan, neg, sub, least, normal, most, big = yd.cpu().numpy().tolist()
    assert np.isnan(nan)
    if which == 5:
        assert not np.isfinite(zero)
        assert inf == 0.0 or np.isnan(inf)
        assert neg == -1.0
        assert not np.isfinite(sub) and not np.isfinite(least)  # above the largest number
        assert normal == 2.0 ** 1022 and big == 2.0 ** -1022
        assert abs(most - 1 / 1.7e308) <= 2.0 ** -1022 * 2.0 ** -50 or most == 0.0 or np.isnan(most)
    else:
        assert zero == 0.0 and inf == np.inf and np.isnan(neg)
        assert sub == np.sqrt(1e-310) and least == np.sqrt(5e-324) and normal == 2.0 ** -511
        assert abs(most - np.sqrt(1.7e308)) <= np.spacing(most) and big == 2.0 ** 511
