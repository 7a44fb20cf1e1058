"""How the gridders' CTAs share the slices of the work items (slice_rule.cuh, compiled
for the host): every entry is in one slice of one CTA, and no CTA has much more than
its share, whether the entries are spread thinly, crowded in one tile, or both."""
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
    d = tmp_path_factory.mktemp("walk")
    (d / "s.cpp").write_text('#include "slice_rule.cuh"\nextern "C" { int e(int64_t n, int64_t s, int64_t c) { return '
                             "rix::slice_entries(n, s, c); }\nint l(int64_t f, int s) { return rix::slices_log2(f, s); }\n"
                             "int64_t b(int64_t t, int64_t s) { return rix::slice_blocks(t, s); } }\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "s.so"), str(d / "s.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "s.so"))
    lib.e.argtypes, lib.l.argtypes, lib.b.argtypes = [ctypes.c_int64] * 3, [ctypes.c_int64, ctypes.c_int], [ctypes.c_int64] * 2
    lib.b.restype = ctypes.c_int64
    return lib


def _tiles(kind):
    rng = np.random.default_rng(7)
    thin = rng.integers(1, 60, 16000)
    return {"thin": thin, "one": np.array([1]), "crowded": np.array([30000, 20000, 7]), "edges": np.array(
        [5, 2049, 4096, 1, 2047, 64, 65, 6000]), "both": np.concatenate([thin[:5000], [100000], thin[5000:9000]]),
        "as many as CTAs": np.full(1217, 3), "long": rng.integers(1, 300, 700)}[kind]


@pytest.mark.parametrize("slots", [152, 304, 1216])
@pytest.mark.parametrize("kind", ["thin", "one", "crowded", "edges", "both", "as many as CTAs", "long"])
def test_every_entry_once_and_evenly(rule, kind, slots):
    tiles = _tiles(kind)
    cuts = [min(ITEM, n - k) for n in tiles for k in range(0, n, ITEM)]
    items = np.concatenate([[0], np.cumsum(cuts)])
    for crowded in (0, int(tiles.max())):
        s = rule.e(int(items[-1]), slots, crowded)
        l = rule.l(int(tiles.max()), s)
        total = len(cuts) << l
        grid = rule.b(total, slots)
        assert 1 <= grid <= slots and (grid == total or grid % 2 == 1)
        it = np.arange(total)
        lo = items[it >> l] + (it & ((1 << l) - 1)) * s
        hi = np.minimum(items[(it >> l) + 1], lo + s)
        full = lo < hi
        assert (hi - lo)[full].sum() == items[-1] and (hi - lo)[full].max() <= s
        assert np.array_equal(lo[full][1:], hi[full][:-1]) and lo[full][0] == 0
        load = np.bincount(it[full] % grid, minlength=grid)
        assert load.max() <= 2.0 * load.mean() + 2
