"""The cluster that a small FISTA loop runs on: 16 CTAs, or the largest power of two
that the device takes, down to one; a launch that none helps returns its error.
Host code, compiled and run without a GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "k_fista.cuh"
namespace rix {
int set_error(int code, const char*, ...) { return code; }
void note_launch(long long) {}
void timing_mark(int, cudaStream_t, bool) {}
}
int main() {
  for (int most : {64, 16, 15, 8, 7, 4, 2, 1, 0}) {
    int tried = 0, ran = 0;
    const cudaError_t e = rix::launch_clusters([&](int c) {
      ++tried;
      if (c > most) return cudaErrorInvalidConfiguration;
      ran = c;
      return cudaSuccess;
    });
    std::printf("%d %d %d %d\n", most, ran, tried, (int)(e == cudaSuccess));
  }
}
"""


def test_largest_cluster_that_fits(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    got = {most: (ran, tried, ok) for most, ran, tried, ok in zip(*[iter(map(int, out))] * 4)}
    assert got == {64: (16, 1, 1), 16: (16, 1, 1), 15: (8, 2, 1), 8: (8, 2, 1), 7: (4, 3, 1), 4: (4, 3, 1), 2: (2, 4, 1),
                   1: (1, 5, 1), 0: (0, 5, 0)}


GRID_PROGRAM = r"""
#include <cstdio>
#include "k_fista.cuh"
namespace rix {
int set_error(int code, const char*, ...) { return code; }
void note_launch(long long) {}
void timing_mark(int, cudaStream_t, bool) {}
}
int main() {
  for (int dict : {RIX_DICT_DB4, RIX_DICT_DB1_8})
    for (int n : {256, 512, 1024, 4096})
      for (int nb : {1, 2})
        for (int solo : {0, 1})
          if (nb == 1 || !solo) std::printf("%d ", rix::loop_ctas_per_sm(nb, solo, dict, n));
}
"""


def test_a_single_loop_leaves_room_for_another(tmp_path):
    """CTAs per SM of one loop of a partitioned job, of an unpartitioned job's loop
    and of a batch: the second is given the room of two only where it is faster with
    other jobs in flight too."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(GRID_PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "1", "2"] * 6 + ["1", "2", "2"] * 2
