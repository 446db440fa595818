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
