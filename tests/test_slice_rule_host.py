"""The cut of the gridders' work items (slice_rule.cuh, compiled for the host): its
bounds, and that FP32 sums in the pieces it chooses are no less accurate than in
whole work items."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")
ITEM = 2048


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("slices")
    (d / "s.cpp").write_text('#include "slice_rule.cuh"\nextern "C" int f(int64_t e, int64_t n, int64_t c) '
                             "{ return rix::slice_entries(e, n, c); }\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "s.so"), str(d / "s.cpp")], check=True)
    f = ctypes.CDLL(str(d / "s.so")).f
    f.argtypes = [ctypes.c_int64] * 3
    return f


@pytest.mark.parametrize("slots", [0, 1, 304, 1216])
@pytest.mark.parametrize("entries", [1, 63, 4999, 16639, 16641, 92681, 92683, 311296, 10 ** 7, 2 ** 31 - 1])
def test_bounds(rule, entries, slots):
    for crowded in sorted({0, 1, entries // 7, entries}):
        s = rule(entries, slots, crowded)
        assert 64 <= s <= ITEM and ITEM % s == 0
        assert s == ITEM or crowded ** 2 <= s * ITEM * (s + ITEM)
        assert s == 64 or s < 2 * (entries // (4 * max(slots, 1))) or crowded ** 2 > s // 2 * ITEM * (s // 2 + ITEM)


def _rounding(pieces, m, runs):
    """rms relative error of FP32 sums of m positive values added in pieces"""
    rng = np.random.default_rng(m)
    err = []
    for _ in range(runs):
        x = rng.uniform(0.5, 1.5, m).astype(np.float32)
        part = [np.add.accumulate(x[k:k + pieces])[-1] for k in range(0, m, pieces)]
        total = np.add.accumulate(np.array(part, np.float32))[-1]
        err.append(float(total) / float(x.astype(np.float64).sum()) - 1.0)
    return float(np.sqrt(np.mean(np.square(err))))


@pytest.mark.parametrize("m", [3000, 12000, 16600, 17000, 40000, 92000, 93000, 300000])
def test_sums_as_accurate_as_in_whole_items(rule, m):
    """Both are estimated from 64 sums: 9 % of standard error each, so within 1.3."""
    s = rule(m, 1216, m)
    assert _rounding(s, m, 64) <= 1.3 * _rounding(ITEM, m, 64), s
