"""The near field's integer square root (csrc/q2x_nfmath.cuh) has the bits of
the C library's, which IEEE 754 rounds correctly: with the host's seed, and
with seeds as far off as the device's reciprocal root (2^-22)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
static float g_off = 0.0f;  // relative error of the seed
static float seed_sqrtf(float x) { return std::sqrt(x) * (1.0f + g_off); }
#define sqrtf seed_sqrtf
#define Q2X_NF_TABLE static const
#include "table.inc"
namespace q2x { using ::NF_LN2_63; using ::NF_LN2_55; using ::NF_PI_61; }
#include "q2x_nfmath.cuh"
extern "C" int same(double x)
{
    const double a = q2x::nf_sqrt(x), b = std::sqrt(x);
    return std::memcmp(&a, &b, 8) == 0;
}
extern "C" long differing(int seed, long n, double off)
{
    std::mt19937_64 g(seed);
    g_off = (float)off;
    long bad = 0;
    for (long i = 0; i < n; ++i) {
        // any mantissa, two binades; squares of 27-bit numbers and their neighbours
        double x = std::ldexp((double)((1ull << 52) + (g() & 0xfffffffffffffull)), (int)(i & 1) - 52);
        if ((i & 7) == 7) {
            const double r = (double)(g() >> 37);
            x = r * r + 1.0;
            if (i & 8) x = std::nextafter(x, (i & 16) ? 0.0 : 1e300);
        }
        bad += !same(x);
    }
    g_off = 0.0f;
    return bad;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2107_10942_gb300 import gen_nearfield
    d = tmp_path_factory.mktemp("nfroot")
    gen_nearfield.write(str(d / "table.inc"))
    (d / "t.cpp").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2107_10942_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", csrc, "-o", str(d / "t.so"),
                    str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    so.same.argtypes = [ctypes.c_double]
    so.differing.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.c_double]
    so.differing.restype = ctypes.c_long
    return so


def test_argument_close_to_a_midpoint(lib):
    assert lib.same(float.fromhex("0x1.335c9a9e3209fp+1"))


@pytest.mark.parametrize("off", [0.0, 2.0 ** -22, -(2.0 ** -22), 2.0 ** -23])
def test_bits_of_the_library(lib, off):
    assert lib.differing(1, 4_000_000, off) == 0
