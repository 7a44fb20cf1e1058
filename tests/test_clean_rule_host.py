"""Which ms-CLEAN loop a call takes (clean_bound.cuh, compiled for the host) against
the measured times of both: never one that is slower by more than the runs differ."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")

# (FP64, image side, scales): microseconds per iteration of the lazy form, of a sweep on
# two CTAs per SM and on four (None: not measured)
MEASURED = {
    (0, 64, 1): (5.4, 3.6, 3.6), (0, 64, 4): (6.1, 3.9, 3.9), (0, 128, 1): (5.8, 3.4, 3.4), (0, 128, 8): (7.6, 4.4, 4.4),
    (0, 512, 1): (7.4, 5.1, 6.3), (0, 512, 4): (9.4, 6.6, 7.3), (0, 512, 8): (12.3, 9.2, 9.1),
    (0, 1024, 1): (11.0, 8.0, 8.4), (0, 1024, 3): (13.4, 11.8, 10.7), (0, 1024, 4): (15.7, None, 12.8),
    (0, 1024, 8): (22.1, None, 19.9), (0, 2048, 1): (18.3, 22.3, 15.5), (0, 2048, 2): (21.5, None, 25.3),
    (0, 2048, 4): (29.3, None, 42.5), (0, 4096, 1): (48.0, None, 79.0), (0, 4096, 4): (84.5, None, 200.6),
    (1, 64, 1): (6.7, 4.6, 4.6), (1, 128, 8): (10.6, 6.1, 6.3), (1, 256, 1): (9.2, 6.0, 6.0), (1, 512, 1): (11.0, 7.8, 10.7),
    (1, 512, 3): (14.8, 10.3, 13.1), (1, 512, 8): (27.6, 17.3, 18.6), (1, 1024, 1): (17.8, 13.4, 15.6),
    (1, 1024, 4): (29.4, 28.2, 28.9), (1, 1024, 6): (38.6, 46.1, 37.3), (1, 2048, 1): (28.0, None, 35.2),
    (1, 2048, 4): (60.1, None, 87.6),
}


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text('#include "clean_bound.cuh"\nextern "C" int lazy(int d, int n, int s) { return '
                             "rix::clean_lazy(d, n, s); }\nextern \"C\" int ctas(int d, int n, int s, int l) { return "
                             "rix::clean_ctas_per_sm(d, n, s, l); }\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "r.so"), str(d / "r.cpp")], check=True)
    return ctypes.CDLL(str(d / "r.so"))


@pytest.mark.parametrize("case", sorted(MEASURED))
def test_the_faster_loop(rules, case):
    lazy, two, four = MEASURED[case]
    if rules.lazy(*case):
        taken = lazy
    else:
        taken = two if rules.ctas(*case, 0) == 2 else four
    assert taken is not None and taken <= 1.05 * min(t for t in (lazy, two, four) if t is not None)
