"""The order of an object's hypotheses in its collision tiles, computed on the host (csrc/tile_order.h, compiled here by
itself): strips of at least one and at most n_b grid_b values, whatever the object's speed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2005_06773_gb300 import scenarios as S

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "tile_order.h"
extern "C" int order(int kind, int flags, int n_a, int n_b, const float *grid_a, const float *grid_b, float v0) {
    mhc_object o{};
    o.kind = kind; o.flags = flags; o.n_a = n_a; o.n_b = n_b; o.grid_a = grid_a; o.grid_b = grid_b; o.v0 = v0;
    return mhc::host::tile_order(o);
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile_order")
    src, lib = str(d / "shim.cc"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2005_06773_gb300", "csrc"), src, "-o", lib])
    fn = ctypes.CDLL(lib).order
    fp = ctypes.POINTER(ctypes.c_float)

    def call(n_a, n_b, v0, kind=S.VEHICLE, flags=0, lo=-8.0, hi=3.0, width=0.3):
        a = np.ascontiguousarray(np.linspace(lo, hi, n_a), np.float32)
        b = np.ascontiguousarray(np.linspace(-width, width, n_b), np.float32)
        return fn(kind, flags, n_a, n_b, a.ctypes.data_as(fp), b.ctypes.data_as(fp), ctypes.c_float(v0))

    return call


def test_near_standstill(order):
    """Steering hardly separates the hypotheses of a car that stands: strips of all its angles, not of one."""
    for v0 in (1e-3, 1e-6, 1e-8, 1e-12, 1e-30):
        for n_b in (2, 5, 16):
            assert order(21, n_b, v0) == 2 * n_b, (v0, n_b)
        assert order(21, 17, v0) == 3                  # many angles: one acceleration per strip, along the angles
    assert order(21, 9, 0.0) == 0                      # no distance at all: ascending


def test_range(order):
    rng = np.random.default_rng(5)
    for _ in range(2000):
        n_a, n_b = (int(v) for v in rng.integers(1, 40, 2))
        v0 = float(np.float32(10.0 ** rng.uniform(-40, 38)))
        kind = int(rng.choice([S.VEHICLE, S.PEDESTRIAN]))
        flags = int(rng.choice([0, S.PED_ACCEL_GRID])) if kind == S.PEDESTRIAN else 0
        w = 10.0 ** rng.uniform(-30, 1)
        got = order(n_a, n_b, v0, kind, flags, 0.0, float(10.0 ** rng.uniform(-30, 38)), w)
        if n_a < 2 or n_b < 2:
            assert got == 0
        elif got & 1:
            assert got in (3, 5) and n_b > 16 and n_a >= got >> 1
        else:
            assert 0 <= got >> 1 <= n_b


def test_usual_grids(order):
    assert order(21, 21, 10.0) >> 1 in (4, 5, 6)       # the 11-object scene's cars
    assert order(64, 32, 11.0) >> 1 in (3, 4)          # the 32-car scene's
