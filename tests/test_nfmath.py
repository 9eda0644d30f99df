"""The near field's integer sqrt, log1p of a quotient and atan2
(csrc/q2x_nfmath.cuh), compiled for the host and compared with the C
library's long double functions.

Tolerance in units of 2^-53 of the result's binade: the root is correctly
rounded (0.5, and the two corrections leave 2^-61: 0.51); the others round
once (0.5) after at most some six truncations at 2^-62 of values no smaller
than 2^-8 (0.1 each there): 1.1."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cmath>
#include <cstdint>
#include <random>
#define Q2X_NF_TABLE static const
#include "table.inc"
namespace q2x { using ::NF_LN2_63; using ::NF_LN2_55; using ::NF_PI_61; }
#include "q2x_nfmath.cuh"
using namespace q2x;
typedef long double ld;
static double ulps(double got, ld want)
{
    return (double)(fabsl((ld)got - want) / ldexpl(1, ilogbl(want) - 52));
}
extern "C" double worst(int which, int range, int n)
{
    std::mt19937_64 g(which * 10 + range);
    const NfTables t{nf_log_k, nf_log_t, nf_atan_t};
    const double spread[5] = {1, 4, 12, 60, 200}, s = spread[range];
    auto rnd = [&](double lo, double hi) { return std::exp2(std::uniform_real_distribution<double>(lo, hi)(g)); };
    double w = 0;
    for (int i = 0; i < n; ++i) {
        double u;
        if (which == 0) {
            // spread values, and neighbours of powers of two and of squares
            const double b = (i & 3) == 0 ? std::exp2((int)(g() % 40) - 20) : (i & 3) == 1 ? std::floor(rnd(0, 20)) * std::floor(rnd(0, 5)) + 1 : rnd(-s, s);
            const double x = (i & 8) ? std::nextafter(b, (i & 16) ? 0.0 : 1e300) : b;
            u = ulps(nf_sqrt(x), sqrtl((ld)x));
        } else if (which == 1) {
            double a = rnd(-s, s), b = rnd(-s, s), c = (i & 1) ? 1.0 : rnd(-s, s), d = rnd(-s, s), f = rnd(-s, s);
            if ((i & 6) == 6) f = a * b * c / d * rnd(-2, 14);  // quotients about and below one
            u = ulps(nf_log1p_ratio(a, b, c, d, f, t), log1pl((ld)a * b * c / ((ld)d * f)));
        } else {
            double a = rnd(-s, s), b = rnd(-s, s);
            if ((i & 6) == 6) b = a * (1 + std::ldexp((double)(g() % 1000), -50));
            if ((i & 6) == 4) b = a * ((double)(g() % 65) / 64 + std::ldexp((double)(g() % 1000), -45)) + 1e-30;
            if (i & 1) b = -b;
            u = ulps(nf_atan2(a, b, t), atan2l((ld)a, (ld)b));
        }
        if (!(u <= w)) w = u;
    }
    return w;
}
extern "C" double special(int k)
{
    const NfTables t{nf_log_k, nf_log_t, nf_atan_t};
    const double inf = INFINITY;
    switch (k) {
    case 0: return nf_sqrt(0.0);
    case 1: return nf_sqrt(inf);
    case 2: return nf_sqrt(-1.0);
    case 3: return nf_sqrt(4e-320);
    case 4: return nf_log1p_ratio(1, 1, 1, 1, 0.0, t);
    case 5: return nf_log1p_ratio(1e200, 1e200, 1, 1e-200, 1, t);
    case 6: return nf_log1p_ratio(1e-300, 1e-30, 1, 1, 1, t);
    case 7: return nf_atan2(1.0, 0.0, t);
    case 8: return nf_atan2(1e-310, 1.0, t);
    case 9: return nf_atan2(1.0, -inf, t);
    case 10: return nf_atan2(3.0, -3.0, t);
    default: return nf_atan2(NAN, 1.0, t);
    }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import ctypes

    from paper_2107_10942_gb300 import gen_nearfield
    d = tmp_path_factory.mktemp("nf")
    gen_nearfield.write(str(d / "table.inc"))
    (d / "t.cpp").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2107_10942_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", csrc, "-o", str(d / "t.so"),
                    str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    so.worst.restype = so.special.restype = ctypes.c_double
    return so


@pytest.mark.parametrize("which,tol", [(0, 0.51), (1, 1.1), (2, 1.1)])
@pytest.mark.parametrize("span", range(5))
def test_within_a_unit(lib, which, tol, span):
    assert lib.worst(which, span, 400000) <= tol


def test_special_arguments(lib):
    import math
    v = [lib.special(k) for k in range(12)]
    assert v[0] == 0 and v[1] == math.inf and math.isnan(v[2]) and v[3] == math.sqrt(4e-320)
    assert v[4] == math.inf and v[5] == math.inf and v[6] == 0.0
    assert v[7] == math.pi / 2 and v[8] == math.atan2(1e-310, 1.0) and v[9] == math.pi
    assert v[10] == math.atan2(3.0, -3.0) and math.isnan(v[11])
