"""Kernel names: no two kernels of the library share one (a profiler's filter and a launch list tell them apart by it), and
the names that the benchmark prints for the collision layouts are kernels that exist."""
import collections
import glob
import os
import re

import bench

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_06773_gb300", "csrc")


def _kernels():
    found = []
    for path in glob.glob(os.path.join(SRC, "*.cu")) + glob.glob(os.path.join(SRC, "*.cuh")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        found += re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(\w+)\s*\(", text)
    return found


def test_no_two_kernels_share_a_name():
    names = _kernels()
    assert len(names) > 12
    assert [n for n, c in collections.Counter(names).items() if c > 1] == []


def test_benchmark_names_kernels_that_exist():
    names = set(_kernels())
    for variant, text in bench.COLLIDE_KERNELS.items():
        for name in re.findall(r"\w+_kernel", text):
            assert name in names, (variant, name)
    for variant in (4, 7):           # a listing and a kernel over the list
        assert len(re.findall(r"\w+_kernel", bench.COLLIDE_KERNELS[variant])) == 2
