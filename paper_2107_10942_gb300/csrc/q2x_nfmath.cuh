// q2x_nfmath.cuh -- square root, log(1 + n/d) and atan2 of doubles by integer
// arithmetic, for the near field.
//
// A warp-wide FP64 instruction holds its pipe for 80 cycles on this part, an
// integer multiply-add for 4, and the CUDA library's double sqrt, division,
// log1p and atan2 are ten to forty FP64 instructions each.  These compute on
// the mantissas as 64-bit integers: 24-bit seeds from the FP32 special
// functions, corrected digit by digit; table-driven logarithm and arctangent
// (gen_nearfield.py) with short polynomials whose high coefficients need 32
// bits.  The root is correctly rounded, the others are within one unit in the
// last place of the exact value of their arguments (the host tests); zeros,
// denormals, infinities and NaN take the library's functions, out of line.  The code also compiles for
// the host, where its tests run.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define NF_FN __host__ __device__ __forceinline__
#else
#define NF_FN inline
#endif

namespace q2x {

typedef unsigned long long nf_u64;
typedef long long nf_i64;

// what a caller passes: the tables, in whatever memory it keeps them
struct NfTables {
    const unsigned* log_k;
    const nf_u64* log_t;
    const nf_u64* atan_t;
};

NF_FN nf_u64 nf_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (nf_u64)__double_as_longlong(x);
#else
    nf_u64 b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
NF_FN double nf_double(nf_u64 b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
NF_FN float nf_float(unsigned b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}
NF_FN unsigned nf_fbits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned b;
    memcpy(&b, &x, 4);
    return b;
#endif
}
NF_FN int nf_clz(nf_u64 v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
// FP32 seeds, good to 2^-22
NF_FN float nf_rsqrtf(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / sqrtf(x);
#endif
}
NF_FN float nf_rcpf(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}
// y 2^30 of a seed y in (1/4, 2)
NF_FN unsigned nf_seed30(float y)
{
    const unsigned b = nf_fbits(y);
    return ((b & 0x7fffffu) | 0x800000u) << ((int)(b >> 23) - 120);
}

// 32 x 32 -> 64, one instruction each on the device
NF_FN nf_u64 nf_wu(unsigned a, unsigned b)
{
#ifdef __CUDA_ARCH__
    nf_u64 d;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (nf_u64)a * b;
#endif
}
NF_FN nf_i64 nf_ws(int a, int b)
{
#ifdef __CUDA_ARCH__
    nf_i64 d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (nf_i64)a * b;
#endif
}

// upper half of a 64 x 64-bit product, at most three units too small
NF_FN nf_u64 nf_mulhi(nf_u64 a, nf_u64 b)
{
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
    return nf_wu(ah, bh) + (nf_wu(ah, bl) >> 32) + (nf_wu(al, bh) >> 32);
}

// v 2^-s as a double, v > 0, rounded to nearest; s within +-1000
NF_FN double nf_to_double(nf_u64 v, int s)
{
    const int z = nf_clz(v);
    const nf_u64 m = v << z;
    const nf_u64 r = (m >> 11) + ((m >> 10) & 1);  // 2^52 .. 2^53
    return nf_double(((nf_u64)(1023 + 62 - z - s) << 52) + r);
}

// the library's functions
#ifdef __CUDACC__
#define NF_SLOW static __host__ __device__ __noinline__
#else
#define NF_SLOW static inline
#endif
NF_SLOW double nf_slow_sqrt(double x) { return sqrt(x); }
NF_SLOW double nf_slow_log1p_ratio(double a, double b, double c, double d, double f)
{
    return log1p(a * b * c / (d * f));
}
NF_SLOW double nf_slow_atan2(double a, double b) { return atan2(a, b); }

// ------------------------------------------------------------------ sqrt

// sqrt of x >= 0.  x = X 2^-62 4^k, X in [2^62, 2^64); g0 = sqrt(X) from an
// FP32 reciprocal root, then two corrections E / (2 g) with the exact
// remainder E, each adding some 22 bits: the root is known to a few units of
// 2^-64, and whether it lies above the midpoint 2 r + 1 of its two neighbours r
// and r + 1 (at 2^53) is decided by the exact sign of m 2^(54 + odd) - (2 r + 1)^2,
// which is far below 2^63 here and never zero.
NF_FN double nf_sqrt(double x)
{
    const nf_u64 b = nf_bits(x);
    const int e = (int)(b >> 52);
    if (e == 0 || e >= 2047) return nf_slow_sqrt(x);
    const int odd = (e - 1023) & 1, k = (e - 1023 - odd) / 2;
    const nf_u64 m = (b & 0xfffffffffffffull) | (1ull << 52);
    const nf_u64 X = m << (10 + odd);
    const unsigned Y = nf_seed30(nf_rsqrtf(nf_float(((unsigned)(m >> 29) & 0x7fffffu) | (unsigned)(127 + odd) << 23)));
    const nf_u64 p = nf_wu((unsigned)(X >> 32), Y) >> 29;
    const unsigned g = p > 0xffffffffull ? 0xffffffffu : (unsigned)p;  // sqrt(X) to 22 bits
    const nf_i64 E = (nf_i64)(X - nf_wu(g, g));
    const nf_i64 d = nf_ws((int)(E >> 13), (int)Y) >> 17;  // in 2^-32 of g
    const int dh = (int)(d >> 16);
    const nf_i64 E1 = (nf_i64)(((nf_u64)E << 31) - (nf_u64)g * (nf_u64)d - (nf_u64)(nf_ws(dh, dh) >> 1));
    const nf_i64 d2 = nf_ws((int)(E1 >> 24), (int)Y) >> 37;
    const nf_u64 G = ((nf_u64)g << 32) + (nf_u64)(d + d2);
    const nf_u64 r = G >> 11, mid = 2 * r + 1;
    const nf_i64 above = (nf_i64)((m << (54 + odd)) - mid * mid);  // modulo 2^64
    return nf_double(((nf_u64)(k + 1022) << 52) + r + (above > 0 ? 1u : 0u));
}

// -------------------------------------------------------------- quotient

// N / D 2^62 of two 64-bit integers with their top bits set
NF_FN nf_u64 nf_div(nf_u64 N, nf_u64 D)
{
    const int Y = (int)nf_seed30(nf_rcpf(nf_float(((unsigned)(D >> 40) & 0x7fffffu) | 127u << 23)));
    const unsigned q0 = (unsigned)(nf_wu((unsigned)(N >> 32), (unsigned)Y) >> 32);  // 2^29 N / D
    const nf_i64 R = (nf_i64)(N - (nf_wu(q0, (unsigned)(D >> 32)) << 3) - (nf_wu(q0, (unsigned)D) >> 29));
    const int q1 = (int)(nf_ws((int)(R >> 13), Y) >> 29);  // next digit, in units of 2^11
    const int dh = (int)(D >> 33), dl = (int)((D >> 2) & 0x7fffffffu);
    const nf_i64 R2 = R - ((nf_ws(q1, dh) + (nf_ws(q1, dl) >> 31)) >> 18);
    return ((nf_u64)q0 << 33) + (nf_u64)((nf_i64)q1 << 11) + (nf_u64)(nf_ws((int)R2, Y) >> 31);
}

// r b of r at 2^70 (|r| < 2^-7) and |b| < 1 at 2^62, at 2^63
NF_FN nf_i64 nf_mulfix(nf_i64 r, nf_i64 b)
{
    const int rh = (int)(r >> 32), rl = (int)((unsigned)r >> 1), bh = (int)(b >> 31), bl = (int)b & 0x7fffffff;
    return (nf_ws(rh, bh) + (nf_ws(rl, bh) >> 31) + (nf_ws(rh, bl) >> 31)) >> 6;
}

struct NfMant {
    nf_u64 m;  // top bit set
    int e;     // value m 2^(e - 63)
};
// usable: not zero, denormal, infinite or NaN
NF_FN bool nf_normal(nf_u64 b)
{
    const unsigned f = (unsigned)(b >> 52) & 0x7ffu;
    return f - 1u < 2046u;
}
NF_FN NfMant nf_mant(nf_u64 b)
{
    return NfMant{((b & 0xfffffffffffffull) | (1ull << 52)) << 11, (int)((b >> 52) & 0x7ff) - 1023};
}
NF_FN NfMant nf_norm(nf_u64 m, int e)
{
    const int z = nf_clz(m);
    return NfMant{m << z, e - z};
}

// ------------------------------------------------------------- logarithm

// log1p(a b c / (d f)) of five positive doubles.
//   u = the quotient; v = 1 + u = M 2^e1 with M in [1, 2) (u below 2^-8: v is
//   left alone and r = u); r = M K_i / 1024 - 1, |r| < 2^-7.9;
//   log v = e1 log 2 - log(K_i / 1024) + r (1 - r/2 + r^2/3 - .. + r^6/7).
NF_FN double nf_log1p_ratio(double a, double b, double c, double d, double f, const NfTables& t)
{
    const nf_u64 ba = nf_bits(a), bb = nf_bits(b), bc = nf_bits(c), bd = nf_bits(d), bf = nf_bits(f);
    NfMant N{0, 0}, D{0, 0};
    const bool normal = nf_normal(ba) && nf_normal(bb) && nf_normal(bc) && nf_normal(bd) && nf_normal(bf);
    if (normal) {
        const NfMant ma = nf_mant(ba), mb = nf_mant(bb), mc = nf_mant(bc), md = nf_mant(bd), mf = nf_mant(bf);
        N = nf_norm(nf_mulhi(nf_mulhi(ma.m, mb.m), mc.m), ma.e + mb.e + mc.e + 2);
        D = nf_norm(nf_mulhi(md.m, mf.m), md.e + mf.e + 1);
    }
    const int k = N.e - D.e;
    if (!normal || k > 150 || k < -900) return nf_slow_log1p_ratio(a, b, c, d, f);
    const nf_u64 Q = nf_div(N.m, D.m);  // u = Q 2^(k - 62)
    const bool small = k <= -9;
    nf_i64 r;
    nf_u64 T = 0;
    int e1 = 0;
    if (small) {
        const int sh = -k - 8;
        r = sh < 63 ? (nf_i64)(Q >> sh) : 0;
    } else {
        nf_u64 M;
        if (k < 0) {  // u below one
            M = (Q >> (-k - 1)) + (1ull << 63);
        } else {
            const nf_u64 V = Q + (k < 63 ? (1ull << 62) >> k : 0);
            const int z = nf_clz(V);
            M = V << z;
            e1 = k + 1 - z;
        }
        const unsigned i = (unsigned)(M >> 55) & 255u;
        const unsigned K = t.log_k[i];
        r = (nf_i64)((M >> 3) * K + ((((unsigned)M & 7u) * K) >> 3));  // modulo 2^64: 2^70 (M K / 1024 - 1)
        T = t.log_t[i];
    }
    const int rh = (int)(r >> 32);
    // 1/7, 1/6, 1/5, 1/4 at 2^31, 1/3 at 2^62
    int q = 306783378;
    q = 357913941 - (int)(nf_ws(rh, q) >> 38);
    q = 429496730 - (int)(nf_ws(rh, q) >> 38);
    q = 536870912 - (int)(nf_ws(rh, q) >> 38);
    const nf_i64 q3 = 1537228672809129301ll - (nf_ws(rh, q) >> 7);
    const nf_i64 q2 = (1ll << 61) - (nf_mulfix(r, q3) >> 1);
    const nf_i64 w = nf_mulfix(r, q2) >> 1;  // log1p(r) = r (1 - w)
    if (small) return nf_to_double(nf_mulhi(Q << 1, (nf_u64)((1ll << 62) - w) << 1), 62 - k);
    const nf_u64 tot = T + (nf_u64)(((r + 64) >> 7) - nf_mulfix(r, w));  // at 2^63, below log 2
    if (e1 <= 1) return nf_to_double(tot + (e1 ? NF_LN2_63 : 0), 63);
    return nf_to_double((tot >> 8) + (nf_u64)e1 * NF_LN2_55, 55);
}

// ------------------------------------------------------------ arctangent

// atan2(a, b) of a > 0 and any b, in (0, pi).
//   z = the smaller over the larger of a, |b|; i = 64 z rounded (z below 2^-7:
//   i = 0, nothing subtracted); atan z = atan(i/64) + atan(y), y = (z - i/64) /
//   (1 + z i/64) formed from the mantissas, |y| <= 2^-7;
//   atan y = y (1 - s/3 + s^2/5 - s^3/7), s = y^2.
NF_FN double nf_atan2(double a, double b, const NfTables& t)
{
    const nf_u64 ba = nf_bits(a), bb = nf_bits(b) & 0x7fffffffffffffffull;
    const bool neg = (nf_bits(b) >> 63) != 0, swap = ba > bb;
    const NfMant hi = nf_mant(swap ? ba : bb), lo = nf_mant(swap ? bb : ba);
    int k = lo.e - hi.e;
    if (!nf_normal(ba) || !nf_normal(bb) || k < -900) return nf_slow_atan2(a, b);
    NfMant N = lo, D = hi;
    bool minus = false;
    nf_u64 T = 0;
    const bool small = k <= -8;
    if (!small) {
        const float nf = nf_float(((unsigned)(lo.m >> 40) & 0x7fffffu) | (unsigned)(127 + k) << 23);
        const float df = nf_float(((unsigned)(hi.m >> 40) & 0x7fffffu) | 127u << 23);
        const unsigned i = (unsigned)(nf * nf_rcpf(df) * 64.0f + 0.5f);
        const nf_u64 n = lo.m >> -k;
        nf_i64 d = (nf_i64)(n - (hi.m >> 6) * i);  // modulo 2^64, small
        minus = d < 0;
        if (minus) d = -d;
        T = t.atan_t[i];
        if (d == 0) d = 1;
        N = nf_norm((nf_u64)d, 0);
        D = nf_norm((hi.m >> 1) + (n >> 7) * i, 1);
        k = N.e - D.e;
    }
    const nf_u64 Q = nf_div(N.m, D.m);  // y = Q 2^(k - 62), below 2^-6.99
    const int sh = -k - 7;
    const nf_u64 z = sh < 63 ? Q >> sh : 0;  // at 2^69
    const nf_u64 s = nf_mulhi(z, z);         // at 2^74
    const int s45 = (int)(s >> 29);
    // 1/7, 1/5 at 2^31, 1/3 at 2^62
    const int q5 = 429496730 - (int)(nf_ws(s45, 306783378) >> 45);
    const nf_i64 q3 = 1537228672809129301ll - (nf_ws(s45, q5) >> 14);
    const nf_u64 w = nf_mulhi(s << 3, (nf_u64)q3 << 1) >> 14;
    const nf_u64 yp = nf_mulhi(Q << 1, ((1ull << 62) - w) << 1);  // atan y = yp 2^(k - 62)
    if (small && !swap && !neg) return nf_to_double(yp, 62 - k);
    const nf_u64 y62 = -k < 63 ? yp >> -k : 0;
    nf_u64 th = (minus ? T - y62 : T + y62) >> 1;  // at 2^61
    if (swap) th = (NF_PI_61 >> 1) - th;
    if (neg) th = NF_PI_61 - th;
    return nf_to_double(th, 61);
}

}  // namespace q2x
