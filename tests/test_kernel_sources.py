"""Rules of the kernels' sources that no run can be relied on to break: an order
of memory that the hardware happens to give today, or a state that two host
threads share.  Each is read from the source, comments removed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_22128_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_flush_locks_order_the_whole_warp():
    """k_tiles_fp: lane 0 takes and gives back a lock of the shared grid tile for
    its warp.  A shuffle orders no memory, so the other lanes' accesses lie
    between two __syncwarp: one after lane 0's acquiring fence, one before its
    releasing fence."""
    src = _source("k_tiles_fp.cu")
    take = src.index("atomicCAS(lock")
    give = src.index("atomicExch(lock")
    section = src[take:give]
    first, last = section.index("flush_half("), section.rindex("flush_half(")
    acquire, release = section[:first], section[last:]
    assert "__syncwarp()" in acquire[acquire.index("__threadfence_block()"):]
    assert "__threadfence_block()" in release[release.index("__syncwarp()"):]


def test_clean_kernel_sets_no_attribute():
    """A kernel's attributes belong to the process, and the shared memory of
    k_msclean is sized by the job: a value set for one thread's launch would
    bound another's."""
    assert "cudaFuncSetAttribute" not in _source("k_minor.cu")


def test_one_size_of_a_work_item():
    """The partition cuts work items, and the gridders walk, order and slice them,
    by the same number."""
    found = [(f, line.strip()) for f in sorted(os.listdir(CSRC)) for line in _source(f).splitlines()
             if re.search(r"constexpr\s+int\s+k\w*\s*=\s*2048\b", line)]
    assert len(found) == 1 and found[0][0].endswith(".cuh"), found
