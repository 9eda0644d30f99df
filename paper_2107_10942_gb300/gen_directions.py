"""Writes the constant tables of the direction kernels (csrc/q2x_dir.cuh) as
a CUDA source fragment.  Run by the build, once per output folder.

A null vector a (complex, a.a = 0) makes (a.y)^n a harmonic polynomial of
degree n, and p + 1 of them in general position determine every R_n^m of
degree n <= p: with w the stereographic coordinate of a point of the sphere,

    a(w) = (1 - w^2, -i (1 + w^2), -2 w) / (1 + |w|^2),
    (a.y)^n = (2 / (1 + |w|^2))^n sum_m T_n^m w^(n+m),

T_n^m the paper's tilde values of n! R_n^m (Eq. (rec10): T_n^m = [w^m]
(-xi w - z + eta / w)^n).  |Re a| = |Im a| = 1, so |a.y| <= |y|.  The points
are a Fibonacci spiral on the half sphere (antipodes give the complex
conjugate, so the other half adds nothing): for p <= 20 the matrix from the
scaled values N_n^m = T_n^m sqrt((n+m)! (n-m)!) / n! to the p + 1 complex
samples has no singular value below 0.74, so samples of a given accuracy give
coefficients of the same accuracy.

Per degree bound p (0 .. 20) the tables hold the p + 1 vectors a, and a left
inverse per degree n: real coefficient (packed column k = n^2 + n + m: the
component of T_n^m that lands in the column, not yet signed or scaled) as a
combination of the 2 (p + 1) sample parts.  All of it is exact rational
arithmetic from points rounded to 2^-20, refined to well below 2^-62 and
rounded once to fixed point.
"""
from __future__ import annotations

import math
import sys

import numpy as np

P_MAX = 20
FRAC = 400  # fractional bits of the integer arithmetic (w^(2p) reaches 2^140)
ONE = 1 << FRAC


def _div(a, b):
    """a / b of two fixed-point numbers, rounded to nearest."""
    q = ((abs(a) << FRAC) + (abs(b) >> 1)) // abs(b)
    return q if (a < 0) == (b < 0) else -q


def _mul(a, b):
    return (a * b + (ONE >> 1)) >> FRAC


def points(n):
    """n points w = (re, im) in units of 2^-20, a Fibonacci spiral on the half sphere z > 0."""
    golden = math.pi * (3.0 - math.sqrt(5.0))
    out = []
    for k in range(n):
        z = (k + 0.6) / n if n > 1 else 0.5
        r = math.sqrt(1.0 - z * z) / (1.0 - z)  # |w| of the stereographic projection
        ph = k * golden + 0.37
        out.append((int(round(r * math.cos(ph) * 1048576)), int(round(r * math.sin(ph) * 1048576))))
    return out


def samples(p):
    """The vectors a (p + 1 rows of three (re, im) pairs) and, per degree n,
    the sample matrix [2 (p + 1)][2n + 1] over the scaled values in packed
    order (fixed point)."""
    vec, rows = [], [[] for _ in range(p + 1)]
    scale = []
    for n in range(p + 1):
        # n! / sqrt((n+m)! (n-m)!)
        scale.append([math.isqrt((math.factorial(n) ** 2 << (2 * FRAC)) //
                                 (math.factorial(n + m) * math.factorial(n - m))) for m in range(n + 1)])
    for wr, wi in points(p + 1):
        wr, wi = wr << (FRAC - 20), wi << (FRAC - 20)
        w2r, w2i = _mul(wr, wr) - _mul(wi, wi), 2 * _mul(wr, wi)
        den = ONE + _mul(wr, wr) + _mul(wi, wi)
        vec.append([(_div(ONE - w2r, den), _div(-w2i, den)), (_div(w2i, den), _div(-(ONE + w2r), den)),
                    (_div(-2 * wr, den), _div(-2 * wi, den))])
        inv = _div(2 * ONE, den)
        powers = [(ONE, 0)]  # w^k
        for _ in range(2 * p):
            r, i = powers[-1]
            powers.append((_mul(r, wr) - _mul(i, wi), _mul(r, wi) + _mul(i, wr)))
        f = ONE
        for n in range(p + 1):
            re, im = [0] * (2 * n + 1), [0] * (2 * n + 1)
            for m in range(n + 1):
                c = _mul(scale[n][m], f)
                ur, ui = (_mul(c, v) for v in powers[n + m])
                if m == 0:
                    re[n], im[n] = ur, ui
                    continue
                sg = -1 if m & 1 else 1  # T^-m = (-1)^m conj T^m
                vr, vi = (sg * _mul(c, v) for v in powers[n - m])
                # T = a + i b: (a + i b) u + (a - i b) v
                a_re, a_im, b_re, b_im = ur + vr, ui + vi, -(ui - vi), ur - vr
                # packed: the Re column takes a for even m and b for odd m
                ka, kb = (n + m, n - m) if m % 2 == 0 else (n - m, n + m)
                re[ka], im[ka], re[kb], im[kb] = a_re, a_im, b_re, b_im
            rows[n] += [re, im]
            f = _mul(f, inv)
    return vec, rows


def left_inverse(A):
    """X with X A = 1 (fixed point): the float pseudo-inverse, refined."""
    A = np.array(A, dtype=object)
    X = np.linalg.pinv((A / ONE).astype(np.float64))
    X = np.array([[int(v * 2.0 ** 60) << (FRAC - 60) for v in r] for r in X], dtype=object)
    eye = np.array([[2 * ONE if i == j else 0 for j in range(A.shape[1])] for i in range(A.shape[1])], dtype=object)
    for _ in range(2):
        X = ((eye - (X.dot(A) >> FRAC)).dot(X)) >> FRAC
    return X


def split(v, hi_bits, lo_bits):
    """v (fixed point) as round(v 2^(hi_bits + lo_bits)) = h 2^lo_bits + l, l balanced."""
    t = (v + (1 << (FRAC - hi_bits - lo_bits - 1))) >> (FRAC - hi_bits - lo_bits)
    h = (t + (1 << (lo_bits - 1))) >> lo_bits
    l = t - (h << lo_bits)
    assert abs(h) < (1 << 31) and abs(l) < (1 << 30)  # (the kernels double and negate l)
    return h, l


def _ints(name, vals, kind="int", per=12):
    lines = ["static __device__ const %s %s[%d] = {" % (kind, name, len(vals))]
    for i in range(0, len(vals), per):
        lines.append(",".join(str(v) for v in vals[i:i + per]) + ",")
    return "\n".join(lines + ["};"])


def write(path):
    vec_off, inv_off, vecs, invs = [], [], [], []
    for p in range(P_MAX + 1):
        vec, rows = samples(p)
        vec_off.append(len(vecs) // 2)
        inv_off.append(len(invs) // 2)
        for a in vec:  # re x, y, z then im x, y, z: (h, l) each
            for part in (0, 1):
                for d in range(3):
                    vecs += split(a[d][part], 31, 31)
        ncol = (p + 1) ** 2
        table = [[0] * ncol for _ in range(2 * p + 2)]
        for n in range(p + 1):
            X = left_inverse(rows[n])
            for k in range(2 * n + 1):
                for s in range(2 * p + 2):
                    table[s][n * n + k] = int(X[k, s])
        for row in table:
            for v in row:
                invs += split(v, 30, 28)
    with open(path, "w") as f:
        f.write("// Generated by gen_directions.py: constant tables of the direction kernels.\n")
        f.write(_ints("g_dir_vec", vecs) + "\n")
        f.write(_ints("g_dir_inv", invs) + "\n")
        f.write("static const int h_dir_vec_off[%d] = {%s};\n" % (P_MAX + 1, ",".join(map(str, vec_off))))
        f.write("static const int h_dir_inv_off[%d] = {%s};\n" % (P_MAX + 1, ",".join(map(str, inv_off))))
        # per column and hat depth d: n! / (sqrt((n+m)! (n-m)!) (n+d)!), and the same / 4 pi
        pi = 0
        x5, x239 = 5, 239  # Machin: pi = 16 atan(1/5) - 4 atan(1/239)
        for mult, x in ((16, x5), (-4, x239)):
            term, k, s = ONE // x, 0, 1
            while term:
                pi += mult * s * (term // (2 * k + 1))
                term //= x * x
                k, s = k + 1, -s
        cols = []
        for norm in (0, 1):
            for d in range(4):
                for n in range(P_MAX + 1):
                    for m in range(-n, n + 1):
                        a = abs(m)
                        q = (math.factorial(n) ** 2 << (2 * FRAC)) // (math.factorial(n + a) * math.factorial(n - a))
                        v = _div(math.isqrt(q << 160), (math.factorial(n + d) << FRAC))  # 2^80 times the value
                        if norm == 0:
                            v = _div(v, 4 * pi)
                        cols.append(v / (1 << FRAC) / 2.0 ** 80)
        f.write("static __device__ const double g_dir_col[%d] = {%s};\n" % (len(cols), ",".join(float(v).hex() for v in cols)))


if __name__ == "__main__":
    write(sys.argv[1])
