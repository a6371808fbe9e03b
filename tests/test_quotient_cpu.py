"""The quotient iteration of the path generation (csrc/quotient.h, compiled here by itself; its products, sums and fused
operations round the same on the device) against IEEE division, bit for bit: random and edge mantissas, dividends on both
sides of the line from which it takes the division, and every wheelbase that validation accepts, up to an infinite sum."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <cstdint>
#include <cstring>
#include "quotient.h"
static uint64_t state;
static uint32_t next32() {
    state += 0x9E3779B97F4A7C15ull;
    uint64_t z = state;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}
static float of_bits(uint32_t b) { float f; std::memcpy(&f, &b, 4); return f; }
static uint32_t bits(float f) { uint32_t b; std::memcpy(&b, &f, 4); return b; }
static bool differs(float a, float b) {
    const float want = a / b, got = mhc::quotient(a, b, 1.0f / b);
    return (want == want) ? bits(want) != bits(got) : got == got;
}
// n random pairs, the divisor's exponent (biased) in [lo, hi], any dividend's; the failures, the first of them in bad
extern "C" long long random_pairs(long long n, int lo, int hi, uint64_t seed, float *bad) {
    long long wrong = 0;
    state = seed;
    for (long long q = 0; q < n; ++q) {
        const uint32_t eb = lo + next32() % (uint32_t)(hi - lo + 1), ea = next32() % 256u;
        const float a = of_bits((next32() & 0x807fffffu) | ea << 23), b = of_bits((next32() & 0x7fffffu) | eb << 23);
        if (differs(a, b) && wrong++ == 0) { bad[0] = a; bad[1] = b; }
    }
    return wrong;
}
extern "C" int pair(float a, float b) { return differs(a, b); }
extern "C" long long edge_mantissas(float *bad) {
    const uint32_t edge[] = {0, 1, 2, 3, 0x3fffff, 0x400000, 0x400001, 0x2aaaaa, 0x555555, 0x7ffffd, 0x7ffffe, 0x7fffff};
    long long wrong = 0;
    for (int ea = 0; ea < 256; ++ea)
        for (int eb = 0; eb < 256; ++eb)
            for (uint32_t ma : edge)
                for (uint32_t mb : edge) {
                    const float a = of_bits(ma | (uint32_t)ea << 23), b = of_bits(mb | (uint32_t)eb << 23);
                    if (differs(a, b) && wrong++ == 0) { bad[0] = a; bad[1] = b; }
                }
    return wrong;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotient")
    src, so = str(d / "shim.cc"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2005_06773_gb300", "csrc"), src, "-o", so])
    lib = ctypes.CDLL(so)
    lib.random_pairs.restype = lib.edge_mantissas.restype = ctypes.c_longlong
    lib.random_pairs.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_uint64, ctypes.c_void_p]
    lib.pair.argtypes = [ctypes.c_float, ctypes.c_float]
    return lib


@pytest.mark.parametrize("lo,hi", [(126, 131), (100, 150), (0, 255)])
def test_random_mantissas(lib, lo, hi):
    """Divisors of a car's wheelbase (1 to 32 m), of 1e-8 to 1e7, and any."""
    bad = (ctypes.c_float * 2)()
    assert lib.random_pairs(5_000_000, lo, hi, 7 * lo + hi, bad) == 0, tuple(bad)


def test_edge_mantissas(lib):
    bad = (ctypes.c_float * 2)()
    assert lib.edge_mantissas(bad) == 0, tuple(bad)


@pytest.mark.parametrize("b", [float("inf"), 3e38, 1e30, 1.1e12, 9e11, 1.1e-12, 9e-13, 1e-30, 1e-38, 1e-39, 1e-45, 2.7])
@pytest.mark.parametrize("a", [0.0, -0.0, 1e-45, 9.9e-21, 1e-20, 1.1e-20, -0.3, 0.5, 9.9e19, 1.1e20, 1e38, float("inf")])
def test_range(lib, a, b):
    assert not lib.pair(a, b)
