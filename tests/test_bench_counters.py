"""bench.py reports committed DRAM counters only beside the kernel they were taken
from: the hash that ties them to it changes with everything that makes the
kernel, and the updates a launch stands for are the kernel's own."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2510_11042_gb300", "csrc")


@pytest.mark.parametrize("two_d,name,old,new", [
    (True, "step_cell.cuh", "static __device__ __forceinline__ unsigned pack(", "static __device__ unsigned pack("),
    (True, "march.cuh", "constexpr int kRows = 16;", "constexpr int kRows = 8;"),
    (True, "march.cu", "#pragma unroll 1\n", "#pragma unroll 2\n"),
    (True, "lbem_internal.cuh", "constexpr int kMarchSteps = 4;", "constexpr int kMarchSteps = 2;"),
    (True, "lbem_internal.cuh", "constexpr int kMarchMinRows = 4;", "constexpr int kMarchMinRows = 8;"),
    (True, "lbem_internal.cuh", "    float inv_scale, scale;\n", "    float scale, inv_scale;\n"),
    (False, "step_cell.cuh", "static __device__ __forceinline__ unsigned pack(", "static __device__ unsigned pack("),
    (False, "step2.cu", "constexpr long long kWaitNs", "constexpr  long long kWaitNs"),
    (False, "lbem_internal.cuh", "    int rows_per_block; ", "    int rows_of_block; "),
])
def test_the_hash_changes_with_the_kernel(tmp_path, monkeypatch, two_d, name, old, new):
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_source_hash(two_d)
    path = tmp_path / CSRC / name
    text = path.read_text()
    assert old in text
    path.write_text(text.replace(old, new))
    assert bench.kernel_source_hash(two_d) != before


def test_updates_per_pass():
    assert [bench.updates_per_pass(m, f) for m, f in (("ez", 2), ("hz", 2), ("3d", 2), ("ez", 1), ("3d", 1))] == \
        [4, 4, 2, 1, 1]
