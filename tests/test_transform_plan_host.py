"""The plans of the row and column passes (fft_engine.cuh): the radices of every length
multiply to it and fit a thread's values, a CTA holds whole rows, its shared memory
fits an SM, and a short FP64 transform is spread over at least a warp's threads per
eight rows with few values each (a thread with 16 took longer than the whole pass).
Host code, compiled and run without a GPU."""
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
template <typename R, int LOGF, int E> void row() {
  using X = Xf<R, LOGF, E, false>;
  std::printf("%d %d %d %d %d %d %d", (int)sizeof(R), LOGF, E, X::V, X::T, X::NB, (int)X::kSmem);
  for (int p = 0; p < X::NP; ++p) std::printf(" %d", 1 << ct_lr(LOGF, p, X::MLR));
  std::printf("\n");
}
template <typename R, int LO, int HI> void rows() {
  if constexpr (LO <= HI) {
    row<R, LO, 1>();
    if constexpr (LO < HI) row<R, LO, 2>();
    rows<R, LO + 1, HI>();
  }
}
int main() {
  rows<float, kMinLogF, kMaxLogL<float>>();
  rows<double, kMinLogF, kMaxLogL<double>>();
}
"""


def test_plans(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    rows = [[int(v) for v in r.split()] for r in out if r]
    assert len(rows) == 2 * (9 + 8) - 2
    for size, logf, e, v, t, nb, smem, *radices in rows:
        length = 1
        for r in radices:
            assert 2 <= r <= v and v % r == 0
            length *= r
        assert length == 1 << logf and nb >= 1 and nb * length == t * v and t % 32 == 0
        assert smem <= 227 * 1024
        if size == 8 and logf <= 9:
            assert v <= 8 and t * 8 >= 32 * nb
