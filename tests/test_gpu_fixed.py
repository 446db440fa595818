"""The kernels' integer reciprocal and root on the GPU (libat_probe.so), whose
seeds come from the hardware's FP32 approximations."""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [5, 6], ids=["reciprocal", "root"])
def test_within_0_52_ulp(which):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2204_01133_gb300 import build
    build.build()
    L = ctypes.CDLL(os.path.join(os.path.dirname(build.__file__), "libat_probe.so"))
    L.at_probe_fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int]
    rng = np.random.default_rng(4)
    # every FP32 seed argument of a binade and its neighbours in FP64, both parities, and the whole range
    m = 1.0 + np.arange(1 << 20) * 2.0 ** -20
    x = np.concatenate([m, 2.0 * m, np.nextafter(m, 0.0), 4.0 - np.arange(1, 4097) * 2.0 ** -51,
                        np.ldexp(rng.uniform(1.0, 2.0, 1 << 18), rng.integers(-1000, 1000, 1 << 18)),
                        [0.0, np.inf, 1e-310]])
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    assert L.at_probe_fn(xd.data_ptr(), yd.data_ptr(), xd.numel(), which) == 0
    got = yd.cpu().numpy()
    with np.errstate(divide="ignore"):
        ref = 1.0 / x if which == 5 else np.sqrt(x)
    n = len(x) - 3
    # the reference is itself within half an ulp: two values within 0.52 of the exact one are at most one apart
    assert (np.abs(got[:n] - ref[:n]) <= np.spacing(np.abs(ref[:n]))).all()
    assert (got[:n] != ref[:n]).mean() < 0.04  # they differ only next to a rounding boundary
    if which == 6:
        np.testing.assert_array_equal(got[n:], ref[n:])
    else:
        assert not np.isfinite(got[n]) and got[n + 1] in (0.0,) or np.isnan(got[n + 1])
