"""The bound that ms-CLEAN's tile update takes from the cleaned peak
(clean_bound.cuh, compiled for the host) against the loop's own arithmetic, in
both precisions, with and without a fused multiply-add, over the accepted gains:
never above the value the peak keeps."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")


@pytest.fixture(scope="module")
def keep(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("bound")
    (d / "b.cpp").write_text('#include "clean_bound.cuh"\nextern "C" void keep(const float* v, double g, float* o, int n) '
                             "{ for (int i = 0; i < n; ++i) o[i] = rix::clean_keep(v[i], g); }\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "b.so"), str(d / "b.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "b.so"))

    def f(v, gain):
        v = np.ascontiguousarray(v, np.float32)
        out = np.empty_like(v)
        lib.keep(v.ctypes.data_as(ctypes.c_void_p), ctypes.c_double(gain), out.ctypes.data_as(ctypes.c_void_p), v.size)
        return out
    return f


@pytest.mark.parametrize("real", [np.float32, np.float64])
@pytest.mark.parametrize("gain", [1e-3, 0.1, 0.5, 0.9, 0.99, 0.999, 0.9995, 0.9999, 0.99999, 0.999999, 1.0])
def test_never_above_the_remainder(keep, real, gain):
    rng = np.random.default_rng(3)
    n = 50000
    r = rng.normal(size=n).astype(real)
    peak = rng.uniform(0.1, 5.0, n).astype(real)
    scale = (rng.uniform(0.4, 1.0, n).astype(real) / peak).astype(real)
    amp = (real(gain) * r / peak).astype(real)
    wide = np.longdouble
    fused = (r.astype(wide) - amp.astype(wide) * peak.astype(wide)).astype(real)
    rounded = r - (amp * peak).astype(real)
    bound = keep((np.abs(r) * scale).astype(real), gain).astype(np.float64)
    for left in (fused, rounded):
        assert (bound <= (np.abs(left) * scale).astype(np.float64)).all()
    if gain <= 0.9:      # and close to it where that is what leaves tiles alone
        assert (bound >= 0.999 * (1.0 - gain) * (np.abs(r) * scale)).all()


def test_values_that_are_not_finite(keep):
    inf = np.array([np.inf, np.nan], np.float32)
    assert keep(inf, 0.1)[0] == np.inf and np.isnan(keep(inf, 0.1)[1]) and keep(inf, 1.0)[0] == -np.inf
