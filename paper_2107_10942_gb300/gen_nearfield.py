"""Writes the constant tables of the near field's integer functions
(csrc/q2x_nfmath.cuh) as a CUDA source fragment.  Run by the build.

Logarithm (table-driven, after P. T. P. Tang, ACM TOMS 16 (1990) 378): for the
256 intervals [1 + i/256, 1 + (i+1)/256) a short reciprocal K_i / 1024 of the
interval's middle (K_0 = 1024, so that values just above one keep their
relative accuracy) and -log(K_i / 1024) to 63 bits.  Arctangent: atan(i/64)
to 62 bits.  Exact integer arithmetic, rounded once."""
from __future__ import annotations

import sys

FRAC = 120
ONE = 1 << FRAC


def atanh_series(num, den):
    """atanh(num / den) in fixed point."""
    x = (num << FRAC) // den
    x2, term, out, k = (x * x) >> FRAC, x, 0, 1
    while term:
        out += term // k
        term = (term * x2) >> FRAC
        k += 2
    return out


def log_ratio(num, den):
    """log(num / den), num >= den > 0, num < 2 den + 1."""
    return 2 * atanh_series(num - den, num + den)


def atan_series(num, den):
    """atan(num / den) for num <= den / 2 by its power series."""
    x = (num << FRAC) // den
    x2, term, out, k, s = (x * x) >> FRAC, x, 0, 1, 1
    while term:
        out += s * (term // k)
        term = (term * x2) >> FRAC
        k, s = k + 2, -s
    return out


def atan_fixed(num, den):
    """atan of 0 <= num / den <= 1: atan(x) = atan(1/2) + atan((2x - 1) / (x + 2)) above one half."""
    if 2 * num <= den:
        return atan_series(num, den)
    return atan_series(1, 2) + atan_series(2 * num - den, num + 2 * den)


def rounded(v, bits):
    s = FRAC - bits
    return (v + (1 << (s - 1))) >> s


def tables():
    ks = [1024] + [round(1024 * 512 / (512 + 2 * i + 1)) for i in range(1, 256)]
    logs = [rounded(log_ratio(1024, k), 63) if k != 1024 else 0 for k in ks]
    atans = [rounded(atan_fixed(i, 64), 62) if i else 0 for i in range(65)]
    pi = 4 * (4 * atan_series(1, 5) - atan_series(1, 239))
    return ks, logs, atans, rounded(log_ratio(2, 1), 63), rounded(log_ratio(2, 1), 55), rounded(pi, 61)


def write(path):
    ks, logs, atans, ln2, ln2_55, pi = tables()
    with open(path, "w") as f:
        f.write("// Generated by gen_nearfield.py: constant tables of the near field's integer functions.\n")
        f.write("Q2X_NF_TABLE unsigned nf_log_k[256] = {%s};\n" % ",".join(map(str, ks)))
        f.write("Q2X_NF_TABLE unsigned long long nf_log_t[256] = {%s};\n" % ",".join("%dull" % v for v in logs))
        f.write("Q2X_NF_TABLE unsigned long long nf_atan_t[65] = {%s};\n" % ",".join("%dull" % v for v in atans))
        f.write("constexpr unsigned long long NF_LN2_63 = %dull, NF_LN2_55 = %dull, NF_PI_61 = %dull;\n" % (ln2, ln2_55, pi))


if __name__ == "__main__":
    write(sys.argv[1])
