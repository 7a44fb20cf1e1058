"""The row passes refuse a geometry without the factor tables that they would
read, in the form they read it in: n - 1 is kept as doubles or, for the FP32 inverse
rows of padded planes, as pairs of floats.  The check is host code, compiled
and run without a GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "fft_engine.cuh"
namespace rix {
int set_error(int code, const char*, ...) { return code; }
void note_launch(long long) {}
void timing_mark(int, cudaStream_t, bool) {}
}
using namespace rix;
template <typename R> void row(const char* name, int L, int mode, bool screen, bool corr, bool nm1, bool nm1f) {
  XformGeom g{};
  g.M = 64; g.L = L; g.logL = ilog2(L); g.S = 64; g.nplanes = 2; g.mode = mode;
  g.screen = screen ? &g : nullptr;
  g.corr = corr ? &g : nullptr;
  g.nm1 = nm1 ? (const double*)&g : nullptr;
  g.nm1f = nm1f ? (const float2*)&g : nullptr;
  std::printf("%s %d %d\n", name, check_rows<R>(g, false) == RIX_OK, check_rows<R>(g, true) == RIX_OK);
}
int main() {
  row<float>("none", 128, kFacNone, 0, 0, 0, 0);
  row<float>("screen", 128, kFacPhase, 1, 0, 0, 0);
  row<float>("real", 128, kFacReal, 0, 1, 0, 0);
  row<float>("real-without", 128, kFacReal, 0, 0, 0, 0);
  row<float>("doubles", 128, kFacPhase, 0, 1, 1, 0);
  row<float>("pairs", 128, kFacPhase, 0, 1, 0, 1);
  row<float>("full-length-pairs", 64, kFacPhase, 0, 1, 0, 1);
  row<float>("phase-without", 128, kFacPhase, 0, 1, 0, 0);
  row<double>("fp64-doubles", 128, kFacPhase, 0, 1, 1, 0);
  row<double>("fp64-pairs", 128, kFacPhase, 0, 1, 0, 1);
}
"""


def test_row_passes_refuse_missing_tables(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    got = {r.split()[0]: tuple(int(v) for v in r.split()[1:]) for r in out if r}
    # (forward accepted, inverse accepted)
    assert got == {"none": (1, 1), "screen": (1, 1), "real": (1, 1), "real-without": (0, 0), "doubles": (1, 0),
                   "pairs": (0, 1), "full-length-pairs": (0, 0), "phase-without": (0, 0), "fp64-doubles": (1, 1),
                   "fp64-pairs": (0, 0)}
