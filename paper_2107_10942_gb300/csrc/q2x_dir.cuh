// q2x_dir.cuh -- FP64 leaf sums by directions: the recursions of Lemmas 1-5 as
// scalar complex recurrences, in 64-bit fixed point on the integer pipe.
//
// The tilde stencil of Eq. (rec10) multiplies a row by the Laurent polynomial
// -xi w - z + eta / w, so at a fixed w it is multiplication by one complex
// number, and every level of a chain becomes a scalar recurrence
//     x_n = u_v x_{n-1} + source_n,      u_v = a(w) . (vertex v),
// with a(w) a null vector (gen_directions.py).  p + 1 well-spread w determine
// all (p+1)^2 coefficients (the sample matrix has singular values of at least
// 0.74), and since the map back is linear it is applied once per tile of
// elements, to the sums.  What an element costs is then one complex
// multiply-add per level, direction and degree, with no neighbouring orders,
// no rows and no staging: a lane owns a direction and walks over elements,
// and the leaf sum is an addition in the lane.
//
// Number format.  A warp-wide FP64 instruction holds a sub-partition's FP64
// pipe for 80 cycles on this part, a 32 x 32 + 64-bit integer multiply-add its
// pipe for 4 (both measured).  The recurrences therefore run in fixed point:
// |u| < 1 is kept to 2^-62 and a value x to one unit of a 61-bit integer, both
// as two 32-bit halves, and a real product is three multiply-adds.  What a value
// rounds is relative to its own element, level and degree, as in floating
// point: every element has its own power of two for its length and for its
// weight, what its length takes off from degree to degree is shifted back in,
// every level has the unit of its own size, and the sums of every degree have
// that degree's unit (DirCfg).  So neither heavy elements beside light ones nor
// large ones beside small ones cost digits, at any degree: per degree, errors
// against sums in 113 bits are those of the FP64 row kernel or smaller (kinds,
// degrees to 20, weights up to 1e8 apart; at the top degree of p = 20, in the
// root of the sum of squares of its terms, 1.7e-16 for segments, 2.0e-16
// triangles, 2.6e-16 tetrahedra, the rows 6e-16 to 7e-16; linear density 1.5e-16 to
// 7e-16, the largest where a tenth of a tile's elements carry the degree, the rows
// 4e-16 to 5.6e-16).
//
// What bounds it: the integer multiplies, 36 per step of the triangle chain, and
// beside them the shifts and additions of the format.  The level-9 sphere at p =
// 16 takes 12.5 ms (one scale a tile instead, which lost digits at the high
// degrees of ordinary leaves and all of them in very uneven ones, 11.0; the FP64
// row kernel 36.2).
//
// One CTA per tile of one leaf's elements: thread t < G J owns direction
// t mod J and elements t / J, t / J + G, .. (at most eight, the number
// format's head room).  The accumulators, one complex number per degree and
// thread, live in shared memory: one 16-byte load and store per step cost
// nothing beside its multiplies, and the degree loop needs no registers per
// degree, so one kernel serves every degree.
#pragma once

#include <type_traits>

#include "q2x_batch.cuh"

namespace q2x {

#define Q2X_HD __device__ __forceinline__

// Products and sums are written as mul.wide + add.s64 in one asm block each:
// the assembler makes one 32 x 32 + 64-bit multiply-add (4 cycles of the
// integer pipe) of such a pair, where it splits a mad.wide, or a reordered sum
// of C++ products, into a multiply and carry chains (measured: 245 cycles a
// step of the triangle chain with mad.wide, 196 this way).
Q2X_HD int hi32(long long v) { return (int)(v >> 32); }
Q2X_HD long long madw(int a, int b, long long c)
{
    long long d;
    asm("{.reg .b64 m; mul.wide.s32 m, %1, %2; add.s64 %0, %3, m;}" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// A multiplier of 62 fractional bits, a = h 2^31 + l / 2, |l| <= 2^31 (the
// lower half doubled, for mul2).
struct Fx {
    int h, l;
};
Q2X_HD Fx fx_split(long long v)
{
    Fx f;
    f.h = (int)((v + (1ll << 30)) >> 31);
    f.l = (int)((v - ((long long)f.h << 31)) * 2);
    return f;
}

// A running value: an integer v, |v| <= 2^61 for recurrence values (< 2^62
// for the points' coordinates), and h with v = h 2^32 + (int)v.
struct Cx {
    long long re, im;
};
struct CxH {
    int rh, ih;
};
Q2X_HD int high_of(long long v) { return (int)((unsigned)hi32(v) + ((unsigned)(int)v >> 31)); }
Q2X_HD CxH high_of(const Cx& x) { return CxH{high_of(x.re), high_of(x.im)}; }

// A complex multiplier: halves of the parts and of the negated imaginary part.
struct Mul {
    int rh, rl, ih, il, nh, nl;
};
Q2X_HD Mul mul_of(long long re, long long im)
{
    const Fx r = fx_split(re);
    Fx i = fx_split(im);
    i.l = max(i.l, -0x7fffffff);  // (its negative has to exist)
    return Mul{r.h, r.l, i.h, i.l, -i.h, -i.l};
}

// a x + b y + s for real a, b with a^2 + b^2 <= 1 (halves ah, al, bh, bl) and
// values x, y.  The low products are summed at 2^-31 of a unit from `rnd`: at
// most sqrt(2) (2^62 + 2^60), below 2^63.  Their upper word is worth two units
// and joins the high products, so the result is rounded to two units (rnd =
// 2^31).  The products of two low halves, at most half a unit, are left out.
template <bool S>
Q2X_HD long long mul2(int ah, int al, int bh, int bl, int xl, int xh, int yl, int yh, long long s, long long rnd)
{
    long long o;
    asm("{.reg .b64 a, b, m, z; .reg .b32 t, h;\n"
        "mul.wide.s32 m, %1, %5; add.s64 a, m, %9;\n"
        "mul.wide.s32 m, %2, %6; add.s64 a, a, m;\n"
        "mul.wide.s32 m, %3, %7; add.s64 a, a, m;\n"
        "mul.wide.s32 m, %4, %8; add.s64 a, a, m;\n"
        "mov.b64 {t, h}, a; cvt.s64.s32 z, h;\n"
        "mul.wide.s32 m, %1, %6; add.s64 b, m, z;\n"
        "mul.wide.s32 m, %3, %8; add.s64 %0, b, m;}"
        : "=l"(o)
        : "r"(ah), "r"(al), "r"(bh), "r"(bl), "r"(xl), "r"(xh), "r"(yl), "r"(yh), "l"(rnd));
    return S ? o + o + s : o + o;
}
// u x + s, complex
template <bool S>
Q2X_HD Cx mul_add(const Mul& u, const Cx& x, const CxH& h, const Cx& s, long long rnd)
{
    const int xr = (int)x.re, xi = (int)x.im;
    return Cx{mul2<S>(u.rh, u.rl, u.nh, u.nl, xr, h.rh, xi, h.ih, s.re, rnd),
              mul2<S>(u.ih, u.il, u.rh, u.rl, xr, h.rh, xi, h.ih, s.im, rnd)};
}
// s + a x, real a
Q2X_HD long long mul1(Fx a, int xl, int xh, long long s, long long rnd)
{
    long long o;
    asm("{.reg .b64 a, m, z; .reg .b32 t, h;\n"
        "mul.wide.s32 m, %1, %3; add.s64 a, m, %5;\n"
        "mul.wide.s32 m, %2, %4; add.s64 a, a, m;\n"
        "mov.b64 {t, h}, a; cvt.s64.s32 z, h;\n"
        "mul.wide.s32 m, %1, %4; add.s64 %0, m, z;}"
        : "=l"(o)
        : "r"(a.h), "r"(a.l), "r"(xl), "r"(xh), "l"(rnd));
    return o + o + s;
}
// a . y of one direction part (three Fx) and a point, in 62-bit fixed point
Q2X_HD long long dir_dot(const Fx* a, const long long* y, long long rnd)
{
    const long long o = mul2<false>(a[0].h, a[0].l, a[1].h, a[1].l, (int)y[0], high_of(y[0]), (int)y[1],
                                          high_of(y[1]), 0, rnd);
    return mul1(a[2], (int)y[2], high_of(y[2]), o, rnd);
}
// direction j of the shared table, the lower halves doubled
Q2X_HD void dir_of(const int2* dirs, int j, Fx (&a)[6])
{
#pragma unroll
    for (int d = 0; d < 6; ++d) a[d] = Fx{dirs[j * 6 + d].x, dirs[j * 6 + d].y};
}
Q2X_HD void dir_load(int2* dirs, const int2* vec, int J)
{
    for (int i = threadIdx.x; i < 6 * J; i += blockDim.x) dirs[i] = make_int2(vec[i].x, 2 * vec[i].y);
}

// v >> n, the sign alone from 63 on (which C++ leaves open)
Q2X_HD long long shift_down(long long v, int n)
{
    long long o;
    asm("shr.s64 %0, %1, %2;" : "=l"(o) : "l"(v), "r"(n));
    return o;
}

// y 2^(bits - E) rounded to an integer, E = ex - 1022 the exponent of a bound
// 2^E > |y| (ex its biased exponent, at least 1).
Q2X_HD long long dir_fixed(unsigned long long ybits, int ex, int bits)
{
    const int f = (int)((ybits >> 52) & 0x7FF);
    unsigned long long m = ybits & 0xFFFFFFFFFFFFFull;
    if (f) m |= 1ull << 52;
    const int sh = (f ? f : 1) - ex + bits - 53;
    long long v;
    if (sh >= 0)
        v = (long long)(m << (sh < 10 ? sh : 10));
    else if (sh > -60)
        v = (long long)((m + (1ull << (-sh - 1))) >> -sh);
    else
        v = 0;
    return (ybits >> 63) ? -v : v;
}

struct DirArgs {
    BatchKind kind;
    int64_t n_leaves;
    const double* leaf_c;
    const int32_t* leaf_p;
    int p_max, np, norm, accumulate;
    int J, G;          // directions, element groups per CTA
    long long rnd;     // mul2's start
    const int2* vec;     // [J][6]
    const int2* inv;     // [2 J][np]
    const double* col;   // [norm][d][441]
    const BatchTile* tiles;
    const int64_t* n_tiles_dev;
    unsigned long long* counter;
    const double* wvec;  // vector density: SoA 3 x n_elem components per element
    const double* gal_w; // receiver side: weights [n_leaves][np] of the packed columns,
    double* gal_out;     // and its results [n_elem]
    double* partial[3];
    double* coef[3];
    unsigned* err;
};

// What one CTA's shared memory holds: the directions, the elements' records
// (later the sums), the accumulators [layer][degree][thread] of 16 bytes.
constexpr int DIR_NO_E = -100000;  // the exponent of a tile without weight
template <int KIND, int DENS, int OUTS>
struct DirCfg {
    static constexpr int NV = KIND + 2;
    static constexpr bool LIN = KIND == KIND_TRI && DENS == DENS_LINEAR;
    static constexpr bool DBL = KIND == KIND_TRI && (OUTS & 2) != 0;
    // a vector density: unit-density values, three weighted sums
    static constexpr bool VEC = (OUTS & 4) != 0;
    // receiver side: each element's own value against weights (one layer)
    static constexpr bool GAL = (OUTS & 8) != 0;
    static constexpr bool SGL = (OUTS & 1) != 0 || VEC;
    static constexpr int NL = KIND + 2 + (LIN ? 2 : 0);  // q, p | j, i | b, a; linear: q, j, E, i, Iw
    static constexpr int LAYERS = VEC ? 3 : (SGL ? 1 : 0) + (DBL ? 1 : 0);
    // Number format.  A seed's largest magnitude is 2^SEED, and what an element's
    // length takes off from degree to degree is made up for before every odd one.
    // The values of level k are sums of up to binom(n + k, k) products (order k;
    // linear density: q 0, j 1, E and i 2, W 3): with ue halvings a order before
    // the degrees 1, 3, 7 and 15, all of them stay below 2^61, and a level joins
    // the next one 2^ue smaller, so that a level's rounding is relative to its own
    // size as in floating point.  An element leaves out the halvings that its own
    // bounds, the same recurrence on its vertices' distances, do not need.  The
    // same bounds give the sums' unit per degree, 2^-59 of the tile's largest
    // (eight elements of a group add up to 2^62).
    static constexpr int SEED = 60, ORDER = LIN ? 3 : KIND + 1;
    static constexpr int ACC = VEC ? 60 : 59;  // (a vector density's weights are halves)
    // sums of rounded values; else of values rounded down, half a unit an element
    // added at the end, which costs less and, where most of a tile's elements
    // carry little weight at a degree, half a unit for each
    static constexpr bool TIGHT = KIND == KIND_TET || LIN;
    __host__ __device__ static constexpr int order(int k) { return LIN ? (k == 4 ? 3 : k >= 2 ? 2 : k) : k; }
    // 8-byte words of a record: vertices, the normal, the densities, the seed
    // and its exponents (of a vector density's components too)
    static constexpr int R_NRM = 3 * NV, R_DENS = R_NRM + (DBL ? 3 : 0), R_SEED = R_DENS + (LIN || VEC ? 3 : 0);
    static constexpr int R_EXP = R_SEED + 1, REC = R_EXP + (VEC ? 2 : 1);
    __host__ __device__ static constexpr size_t rec_bytes(int p, int T)
    {
        // the records' space is reused for the sums
        const size_t a = (size_t)T * REC * 8, s = (size_t)(p + 1) * 2 * (p + 1) * LAYERS * 8;
        return ((a > s ? a : s) + 15) / 16 * 16;
    }
    // receiver side: the weights [degree][direction] (16 bytes), the scaled
    // column weights (8) they come from, and the elements' values per direction
    // [element][direction]
    __host__ __device__ static constexpr size_t gal_bytes(int p)
    {
        return (size_t)(p + 1) * (p + 1) * 24 + 16;
    }
    __host__ __device__ static constexpr size_t smem(int p, int T, int nt)
    {
        if (GAL) return (size_t)(p + 1) * 48 + ((size_t)T * REC * 8 + 15) / 16 * 16 + gal_bytes(p) + (size_t)T * (p + 1) * 8;
        return (size_t)(p + 1) * 48 + rec_bytes(p, T) + (size_t)LAYERS * (p + 1) * nt * 16;
    }
};

__device__ __forceinline__ Fx as_fx(int2 v) { return Fx{v.x, v.y}; }
__device__ __forceinline__ long long as_ll(int2 v) { return ((long long)v.y << 32) | (unsigned)v.x; }

// Receiver side: out[e] = sum_c w_c P_c(e) over the packed columns c of an
// element's own coefficients.  The weights are carried to the directions
// (the transposed map, exact products per degree), and sum_n W_n h_n(u1, u2,
// u3) of the chain's values h is nested Horner steps from the highest degree
// down, one per level and degree:
//   c_n = W_n + u1 c_{n+1}, b_n = c_n + u3 b_{n+1}, a_n = b_n + u2 a_{n+1},
// the value a_0 (double layer: of the weights one degree up, times the
// normal's multiplier).  With the vertices' distances r and the largest of them
// rho, B = sum_n h_n(r) max_j |W_nj| bounds a direction's value, and
//   |a_n| <= B rho^-n, |b_n| <= B / h_n(r2, max(r1, r3)), |c_n| <= B / h_n(r),
// while what b_n or c_n rounds grows by no more than these.  So a_n has the unit
// 2^(S + t(n)), 2^S = 2^-60 B and t(n) >= -n log2 rho in steps of two degrees, b_n
// and c_n units 2^ue and 4^ue finer, ue by the element's own h_n: what is lost is
// relative to the element's own terms, wherever it lies in its leaf and
// whichever degrees its value comes from.  Measured against sums in 113 bits, in
// units of the terms (root of their sum of squares), weights of all degrees alike
// in the leaf's scale or growing eightfold a degree: 1.1e-16 to 2e-16 (p = 20,
// growing: to 4e-16), a value from the FP64 rows 1.7e-16 to 3.4e-16.  What it
// costs: level-7 sphere at p = 12 0.54 ms, 0.43 with one scale a tile, the FP64
// row kernel 1.31.
template <typename D>
__device__ __forceinline__ void dir_gal_tile(const DirArgs& a, int T, const BatchTile& t, int n_el, bool live, bool over,
                                             double w, int ey, int lf, int Ej, const float (&rk)[D::NV], int2* rec,
                                             const int2* dirs, int g, int j)
{
    constexpr bool DBL = D::DBL;
    const int tid = threadIdx.x, lane = tid & 31, NT = blockDim.x;
    const int J = a.J, p = a.p_max, np = a.np;
    unsigned char* base = reinterpret_cast<unsigned char*>(rec) + ((size_t)T * D::REC * 8 + 15) / 16 * 16;
    longlong2* W = reinterpret_cast<longlong2*>(base);                       // [p + 1][J], of exponent s_e
    int2* col = reinterpret_cast<int2*>(W + (p + 1) * J);                    // [np]
    long long* val = reinterpret_cast<long long*>(base + D::gal_bytes(p));   // [T][J]
    __shared__ int s_e[Q2X_P_MAX + 1], s_nan;
    __shared__ int s_exp[Q2X_P_MAX + 1];     // a degree's largest weight, s_top 2^s_exp
    __shared__ float s_top[Q2X_P_MAX + 1];
    constexpr int d = DBL ? KIND_TRI : KIND_TRI + 1;
    constexpr int NONE = -1000000;
    const double* wt = a.gal_w + (int64_t)t.leaf * np;
    if (tid == 0) s_nan = 0;
    __syncthreads();
    for (int n = tid >> 5; n <= p; n += NT >> 5) {
        double v[2] = {0.0, 0.0};
        int top = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q = lane + 32 * c;
            if (q <= 2 * n && !(DBL && n == 0)) {
                const int k = n * n + q;
                v[c] = __ldg(wt + k) * __ldg(a.col + (a.norm * 4 + d) * 441 + k);
                if ((col_desc(k) >> (5 + a.norm)) & 1) v[c] = -v[c];
                top = max(top, hi32(__double_as_longlong(v[c])) & 0x7fffffff);
            }
        }
        top = __reduce_max_sync(0xffffffffu, top);
        const int e1 = max(top >> 20, 1);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q = lane + 32 * c;
            if (q <= 2 * n) {
                const long long x = top < 0x7ff00000 ? dir_fixed((unsigned long long)__double_as_longlong(v[c]), e1, 56) : 0;
                const int h = (int)((x + (1ll << 27)) >> 28);
                col[n * n + q] = make_int2(h, (int)(x - ((long long)h << 28)));
            }
        }
        __syncwarp();
        float most = 0.f;
        long long prod[2] = {0, 0};
        int bits = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int s = lane + 32 * c;
            if (s < 2 * J) {
                long long hh = 0, mid = 1ll << 27;
                const int2* P = a.inv + s * np + n * n;
#pragma unroll 4
                for (int q = 0; q <= 2 * n; ++q) {
                    const int2 m = __ldg(P + q), x = col[n * n + q];
                    mid = madw(m.x, x.y, mid);
                    mid = madw(m.y, x.x, mid);
                    hh = madw(m.x, x.x, hh);
                }
                hh += mid >> 28;
                prod[c] = hh;
                bits = max(bits, 64 - __clzll(hh < 0 ? -hh : hh));
                most = fmaxf(most, fabsf((float)hh));
            }
        }
        bits = __reduce_max_sync(0xffffffffu, bits);
        most = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(most)));
        // the largest at 2^61 .. 2^62, so that an element's unit only ever shifts to the right
        const int up = bits ? 62 - bits : 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int s = lane + 32 * c;  // (Re(conj(w) h): the imaginary weight enters negated)
            if (s < 2 * J) reinterpret_cast<long long*>(W + n * J)[s] = (s & 1) ? -(prod[c] << up) : prod[c] << up;
        }
        if (lane == 0) {
            // (weights beyond FP64 make the tile's results NaN)
            if (top >= 0x7ff00000) s_nan = 1;
            s_e[n] = e1 - 1022 - 58 - up;
            s_exp[n] = e1 - 1022;
            s_top[n] = most * 4.907e-18f;  // 2^-58 sqrt(2), both parts together
        }
    }
    __syncthreads();
    int S = 0, halvings = 0;  // 3 bits for each of the degrees 1, 3, 7 and 15
    if (live) {
        const float inv = 1.f / fmaxf(fmaxf(rk[0], rk[1]), fmaxf(rk[2], 1e-30f)), r1 = rk[0] * inv, r2 = rk[1] * inv,
                    r3 = rk[2] * inv, r13 = fmaxf(r1, r3);
        float B = 0.f, h1 = 1.f, h2 = 1.f, h3 = 1.f, b1 = 1.f, b2 = 1.f;
        int most = NONE, at = 0;  // B 2^most, every degree's length factor 2^at less
        for (int n = 0; n <= p - (DBL ? 1 : 0); ++n, at += 65536 * ey - lf) {
            if (n) {  // complete homogeneous sums of the distances over the length
                h1 *= r1;
                h2 = fmaf(r2, h2, h1);
                h3 = fmaf(r3, h3, h2);
                b1 *= r13;
                b2 = fmaf(r2, b2, b1);
            }
            if ((n & (n + 1)) == 0 && n) {  // 2^ue <= 2 b, 4^ue <= 2 h
                const int eb = (__float_as_int(1.999f * b2) >> 23) - 127, eh = (__float_as_int(1.999f * h3) >> 23) - 127;
                halvings |= max(0, min(eb, eh >> 1)) << (3 * (30 - __clz(n + 1)));
            }
            const int e = s_exp[n + (DBL ? 1 : 0)] + ((at + 65535) >> 16);
            const float v = s_top[n + (DBL ? 1 : 0)] * h3;
            if (v > 0.f) {
                const float f = __int_as_float((127 + max(min(most, e) - max(most, e), -126)) << 23);
                B = e > most ? fmaf(B, f, v) : fmaf(v, f, B);
                most = max(most, e);
            }
        }
        if (B > 0.f) S = most + (__float_as_int(1.01f * B) >> 23) - 126 - 60;
    }
    if (tid < n_el) {
        rec[tid * D::REC + D::R_SEED] = make_int2(halvings, 0);
        rec[tid * D::REC + D::R_EXP] = make_int2(S, ey * 131072 + lf);
    }
    __syncthreads();
    const long long rnd = a.rnd;
    const int top = DBL ? p - 1 : p;  // the chain's highest degree
    // t of degrees 2 q and 2 q + 1
    const auto shift_of = [](int q, int lf) { return ((2 * q + 1) * lf + 65535) >> 16; };
    if (g < a.G) {
#pragma unroll 1
        for (int e = g; e < n_el; e += a.G) {
            const int2* r = rec + e * D::REC;
            Mul u[3], nu{};
            {
                Fx da[6];
                dir_of(dirs, j, da);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const long long y[3] = {as_ll(r[3 * k]), as_ll(r[3 * k + 1]), as_ll(r[3 * k + 2])};
                    u[k] = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
                }
                if (DBL) {
                    const long long y[3] = {as_ll(r[D::R_NRM]), as_ll(r[D::R_NRM + 1]), as_ll(r[D::R_NRM + 2])};
                    nu = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
                }
            }
            const int2 xp = r[D::R_EXP];
            const int ey = xp.y >> 17, lf = xp.y & 0x1ffff;
            long long res = 0;
            if (top >= 0) {
                int ts = shift_of(top >> 1, lf);
                int off = xp.x + ts - top * ey;  // the unit's exponent less the length's power
                const longlong2* q = W + (top + (DBL ? 1 : 0)) * J + j;
                const int* qe = s_e + top + (DBL ? 1 : 0);
                const int halvings = r[D::R_SEED].x;
                int iv = 31 - __clz(top + 1), ue = iv ? (halvings >> (3 * iv - 3)) & 7 : 0;
                const auto rounding = [&]() { return rnd + (1ll << 30) - ((1ll << 30) >> ue); };
                long long rs = rounding();  // (with a source that is rounded down in its shift by ue)
                const auto down = [&](const Cx& v) { return Cx{v.re >> ue, v.im >> ue}; };
                const auto weight = [&]() {
                    const longlong2 w0 = *q;
                    const int sh = (int)min((unsigned)(off - *qe - 2 * ue), 63u);
                    const long long half = (long long)((1ull << sh) >> 1);
                    return Cx{(w0.x + half) >> sh, (w0.y + half) >> sh};
                };
                Cx c = weight(), b = down(c), x = down(b);
                CxH hc, hb, hx;
#pragma unroll 2
                for (int n = top - 1; n >= 0; --n) {
                    q -= J;
                    --qe;
                    off += ey;
                    if (n & 1) {  // the next two degrees' unit
                        const int tn = shift_of(n >> 1, lf), dn = ts - tn;
                        ts = tn;
                        off -= dn;
                        c = Cx{c.re << dn, c.im << dn};
                        b = Cx{b.re << dn, b.im << dn};
                        x = Cx{x.re << dn, x.im << dn};
                    }
                    if (((n + 1) & (n + 2)) == 0) {
                        --iv;
                        const int un = iv ? (halvings >> (3 * iv - 3)) & 7 : 0, du = ue - un;
                        const long long hb = (1ll << du) >> 1, hc = (1ll << 2 * du) >> 1;
                        ue = un;
                        rs = rounding();
                        c = Cx{(c.re + hc) >> 2 * du, (c.im + hc) >> 2 * du};
                        b = Cx{(b.re + hb) >> du, (b.im + hb) >> du};
                    }
                    hc = high_of(c);
                    hb = high_of(b);
                    hx = high_of(x);
                    c = mul_add<true>(u[0], c, hc, weight(), rnd);
                    b = mul_add<true>(u[2], b, hb, down(c), rs);
                    x = mul_add<true>(u[1], x, hx, down(b), rs);
                }
                hx = high_of(x);
                res = DBL ? mul2<false>(nu.rh, nu.rl, nu.nh, nu.nl, (int)x.re, hx.rh, (int)x.im, hx.ih, 0, rnd) : x.re;
            }
            val[e * J + j] = res;
        }
    }
    __syncthreads();
    if (tid < n_el) {
        long long hi = 0, lo = 0;  // (J values of up to 2^61)
        for (int k = 0; k < J; ++k) {
            hi += hi32(val[tid * J + k]);
            lo += (unsigned)(int)val[tid * J + k];
        }
        double v = live ? ((double)hi * 4294967296.0 + (double)lo) * w : 0.0;
        int e2 = S + shift_of(0, lf) + (DBL ? 1 : 0) + (KIND_TRI + 1) * Ej;  // (half the normal)
        if (e2 > 1000 || e2 < -1000) {
            const int h = max(-2000, min(2000, e2)) / 2;
            v *= pow2d(h);
            e2 = max(-2000, min(2000, e2)) - h;
        }
        v *= pow2d(e2);
        if (over || s_nan) v = __longlong_as_double(0x7ff8000000000000ll);
        a.gal_out[t.e_lo + tid] = v;
    }
}

// MAX_NT 256: two CTAs of up to 128 registers a thread; 128: six of up to 80.
template <int KIND, int DENS, int OUTS, int MAX_NT>
__global__ void __launch_bounds__(MAX_NT, MAX_NT == 256 ? 2 : 6) q2x_dir_kernel(const DirArgs a, int T)
{
    using D = DirCfg<KIND, DENS, OUTS>;
    constexpr int NV = D::NV;
    constexpr int NL = D::NL;
    constexpr bool LIN = D::LIN, DBL = D::DBL, SGL = D::SGL, VEC = D::VEC, GAL = D::GAL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, NT = blockDim.x;
    const int J = a.J, G = a.G, np = a.np;
    int2* dirs = reinterpret_cast<int2*>(smem_raw);
    int2* rec = reinterpret_cast<int2*>(smem_raw + (size_t)J * 48);
    longlong2* acc = reinterpret_cast<longlong2*>(smem_raw + (size_t)J * 48 + D::rec_bytes(a.p_max, T));
    __shared__ BatchTile s_tile;
    // the tile's exponents: of its largest J sigma r^n (per component of a vector density), of the sums
    constexpr int NE = VEC ? 3 : 1;
    __shared__ int s_more, s_over, s_live[NE], s_E[NE][Q2X_P_MAX + 1], s_bits[3][Q2X_P_MAX + 1];
    dir_load(dirs, a.vec, J);
    const int g = tid / J, j = tid - g * J;
    const long long rnd = a.rnd;
    const long long n_tiles = *a.n_tiles_dev;

#pragma unroll 1
    while (true) {
        __syncthreads();  // the last tile's shared memory is free
        if (tid == 0) {
            const unsigned long long ti = atomicAdd(a.counter, 1ull);
            s_more = ti < (unsigned long long)n_tiles;
            if (s_more) s_tile = a.tiles[ti];
            s_over = 0;
        }
        if (tid < NE * (Q2X_P_MAX + 1)) s_E[0][tid] = DIR_NO_E;
        if (tid < NE) s_live[tid] = 0;
        __syncthreads();
        if (!s_more) break;
        const BatchTile t = s_tile;
        const int n_el = (int)(t.e_hi - t.e_lo);
        const int64_t L = t.leaf;
        int pL = a.leaf_p ? __ldg(a.leaf_p + L) : a.p_max;
        unsigned errbits = 0;
        if (pL < 0 || pL > a.p_max) {
            errbits |= 4u;  // leaf degree out of range: a zero row
            pL = -1;
        }
        // ---- element e = t.e_lo + tid: vertices about the centre, the seed
        double y[NV][3], w = 0.0, nrm[3] = {0.0, 0.0, 0.0}, s[3] = {0.0, 0.0, 0.0};
        double ed[NV - 1][3];
        double dens0 = 0.0;
        bool live = false;
        if (tid < n_el && pL >= 0) {
            const int64_t e = t.e_lo + tid;
            const double c[3] = {__ldg(a.leaf_c + L), __ldg(a.leaf_c + a.n_leaves + L),
                                 __ldg(a.leaf_c + 2 * a.n_leaves + L)};
            live = true;
            int64_t vid[NV];
            bool finite = finite_bits(c[0]) && finite_bits(c[1]) && finite_bits(c[2]);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int64_t v = __ldg(a.kind.idx + (int64_t)k * a.kind.n_elem + e);
                if (v < 0 || v >= a.kind.n_vert) {
                    errbits |= 1u;
                    live = false;
                    v = 0;
                }
                vid[k] = v;
            }
            double x0[3];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double x[3] = {__ldg(a.kind.vx + vid[k]), __ldg(a.kind.vy + vid[k]), __ldg(a.kind.vz + vid[k])};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    finite = finite && finite_bits(x[d]);
                    y[k][d] = x[d] - c[d];
                    if (k == 0)
                        x0[d] = x[d];
                    else
                        ed[k > 0 ? k - 1 : 0][d] = x[d] - x0[d];
                }
            }
            if (LIN) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    s[k] = __ldg(a.kind.sigma + vid[k]);
                    finite = finite && finite_bits(s[k]);
                }
            } else if (VEC) {
                dens0 = 1.0;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    s[k] = __ldg(a.wvec + (int64_t)k * a.kind.n_elem + e);
                    finite = finite && finite_bits(s[k]);
                }
            } else {
                dens0 = __ldg(a.kind.sigma + e);
                finite = finite && finite_bits(dens0);
            }
            if (!finite) {
                errbits |= 2u;
                live = false;
            }
        }
        if (errbits) atomicOr(a.err, errbits);
        // The element's own scales: y as 62-bit integers of 2^ey, |y| <=
        // 2^(ey - lf / 65536), and the seed of 2^ew.
        bool over = false;  // a difference of finite coordinates, or a weight, that overflows
        long long yi[NV][3], seed = 0;
        int ey = 0, lf = 0, ew = 0, Ej = 0, es[3] = {1, 1, 1};
        float rk[NV], mw = 0.f, sf[3] = {0.f, 0.f, 0.f};  // vertices' distances over 2^ey, significands
        if (live) {
            int ym = 0;
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) ym = max(ym, hi32(__double_as_longlong(y[k][d])) & 0x7fffffff);
            over = ym >= 0x7ff00000;
            if (over) live = false;
            const int ex = max(ym >> 20, 1);  // every component below 2^(ex - 1022)
            float r2 = 0.f;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float q = 0.f;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    yi[k][d] = dir_fixed((unsigned long long)__double_as_longlong(y[k][d]), ex, 61);
                    const float f = (float)hi32(yi[k][d]) * 1.862645149230957e-9f;  // 2^-29
                    q = fmaf(f, f, q);
                }
                r2 = fmaxf(r2, q);
                rk[k] = q;
            }
            const bool big = r2 > 0.998f;  // the length could pass one: halved
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) yi[k][d] <<= big ? 0 : 1;
            ey = ex - 1022 + (big ? 1 : 0);
            lf = min(max((int)(-32768.f * log2f(big ? 0.25f * r2 : r2)) - 1, 0), 65535);
#pragma unroll
            for (int k = 0; k < NV; ++k) rk[k] = sqrtf(rk[k]) * (big ? 0.500005f : 1.00001f);
        }
        if (live) {
            // edges scaled (exactly) where their products could leave the range
            if (ey > 200 || ey < -200) {
                Ej = ey;
                const double sc = pow2d(-Ej);
#pragma unroll
                for (int k = 0; k < NV - 1; ++k)
#pragma unroll
                    for (int d = 0; d < 3; ++d) ed[k][d] *= sc;
            }
            double J64;
            if constexpr (KIND == KIND_SEG) {
                J64 = sqrt(ed[0][0] * ed[0][0] + ed[0][1] * ed[0][1] + ed[0][2] * ed[0][2]);
            } else {
                constexpr int kv = NV >= 3 ? 1 : 0;
                const double qx = ed[0][1] * ed[kv][2] - ed[0][2] * ed[kv][1];
                const double qy = ed[0][2] * ed[kv][0] - ed[0][0] * ed[kv][2];
                const double qz = ed[0][0] * ed[kv][1] - ed[0][1] * ed[kv][0];
                if constexpr (KIND == KIND_TRI) {
                    J64 = sqrt(qx * qx + qy * qy + qz * qz);
                    if (DBL) {
                        const double inv = (J64 > 0.0) ? 1.0 / J64 : 0.0;
                        nrm[0] = qx * inv;
                        nrm[1] = qy * inv;
                        nrm[2] = qz * inv;
                    }
                } else {
                    J64 = fabs(qx * ed[NV - 2][0] + qy * ed[NV - 2][1] + qz * ed[NV - 2][2]);
                }
            }
            w = LIN ? J64 : J64 * dens0;
            const int wm = hi32(__double_as_longlong(w)) & 0x7fffffff, wx = max(wm >> 20, 1);
            if (wm >= 0x7ff00000)
                over = !GAL;  // (the receiver side multiplies by w itself)
            else
                seed = dir_fixed((unsigned long long)__double_as_longlong(w), wx, D::SEED);
            ew = wx - 1022 + (KIND + 1) * Ej;
            // the significand (0.5 .. 1) of an upper word, rounded up
            const auto significand = [](int hi) {
                return (hi >> 20) ? __int_as_float((((hi & 0xfffff) + 1) << 3) + (126 << 23)) : 1.f;
            };
            mw = significand(wm);
            if (LIN) {
                int sm = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k) sm = max(sm, hi32(__double_as_longlong(s[k])) & 0x7fffffff);
                es[0] = es[1] = es[2] = max(sm >> 20, 1);
                ew += es[0] - 1022;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const long long v = dir_fixed((unsigned long long)__double_as_longlong(s[k]), es[0], 61);
                    sf[k] = ((float)abs(hi32(v)) + 1.f) * 9.313225746154785e-10f;  // 2^-30
                }
            }
            if (VEC) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int sm = hi32(__double_as_longlong(s[k])) & 0x7fffffff;
                    es[k] = max(sm >> 20, 1);
                    sf[k] = significand(sm);
                }
            }
        }
        if (!GAL && over) atomicOr(&s_over, 1);
        if (tid < n_el) {
            int2* r = rec + tid * D::REC;
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const long long v = live ? yi[k][d] : 0;
                    r[3 * k + d] = make_int2((int)v, hi32(v));
                }
            if (DBL) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {  // half the unit normal
                    const long long v = live ? dir_fixed((unsigned long long)__double_as_longlong(nrm[d]), 1023, 62) : 0;
                    r[D::R_NRM + d] = make_int2((int)v, hi32(v));
                }
            }
            if (LIN || VEC) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {  // half the scaled densities: below one also when rounded
                    const Fx f = fx_split(live ? dir_fixed((unsigned long long)__double_as_longlong(s[k]), es[k], 61) : 0);
                    r[D::R_DENS + k] = make_int2(f.h, f.l);
                }
            }
            r[D::R_SEED] = make_int2((int)seed, hi32(seed));
            r[D::R_EXP] = make_int2(ew * 16, ey * 131072 + lf);
            if (VEC) r[D::R_EXP + (VEC ? 1 : 0)] = make_int2((es[0] - 1022) * 65536 + es[1], es[2] - 1022);
        }
        if constexpr (GAL) {
            dir_gal_tile<D>(a, T, t, n_el, live, over, w, ey, lf, Ej, rk, rec, dirs, g, j);
            continue;
        }
        // per degree, the bounds of the element's values: the tile's largest, rounded
        // up to a power of two, and the halvings that the levels need
        if ((tid & ~31) < n_el) {
            bool counts[NE];
#pragma unroll
            for (int c = 0; c < NE; ++c) {
                counts[c] = live && seed != 0 && (!VEC || s[c] != 0.0) && (!LIN || s[0] != 0.0 || s[1] != 0.0 || s[2] != 0.0);
                const unsigned m = __ballot_sync(0xffffffffu, counts[c]);
                if ((tid & 31) == 0) atomicAdd(&s_live[c], __popc(m));
            }
            float b[NL];
            float top[4] = {0.f, 0.f, 0.f, 0.f};  // per order, the values' largest over some degrees
            int needs[4] = {0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < NL; ++k) b[k] = 1.f;
            if (LIN) {
                b[2] = sf[1] + sf[2];
                b[NL - 1] = b[2] + sf[0];
            }
#pragma unroll 1
            for (int n = 0; n <= pL; ++n) {
                if (n && live) {
                    const float f = __int_as_float((127 + ((((n - 1) & ~1) * lf) >> 16)) << 23);
                    const auto mark = [&]() {
#pragma unroll
                        for (int k = 1; k < NL; ++k) top[D::order(k)] = fmaxf(top[D::order(k)], b[k] * f);
                    };
                    if (n & 1) mark();  // (the shift comes before the degree's products)
                    b[0] *= rk[1];
                    if constexpr (LIN) {
                        b[1] = fmaf(rk[2], b[1], b[0]);
                        b[2] = fmaf(rk[2], b[2], fmaf(sf[1] * (float)(n + 1), b[0], sf[2] * b[1]));
                        b[3] = fmaf(rk[0], b[3], b[1]);
                        b[NL - 1] = fmaf(rk[0], b[NL - 1], fmaf(sf[0], b[3], b[2]));
                    } else {
#pragma unroll
                        for (int k = 1; k < NL; ++k) b[k] = fmaf(rk[(k == NL - 1) ? 0 : k + 1], b[k], b[k - 1]);
                    }
                    mark();
                    if (LIN) top[1] = fmaxf(top[1], (float)(n + 1) * b[0] * f);
                    if (((n + 1) & (n + 2)) == 0 || n == pL) {
                        const int iv = 30 - __clz(n + 1);
                        int need = 0;
#pragma unroll
                        for (int o = 1; o <= D::ORDER; ++o) {  // 2^x <= top < 2^(x + 1): at most 2^(1 + o need)
                            need = max(need, ((__float_as_int(top[o]) >> 23) - 127 + o - 1) / o);
                            top[o] = 0.f;
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) needs[q] = q == iv ? need : needs[q];
                    }
                }
#pragma unroll
                for (int c = 0; c < NE; ++c) {
                    const float m = mw * b[NL - 1] * (VEC ? sf[c] : 1.f) * 1.0001f;
                    const int E = __reduce_max_sync(
                        0xffffffffu,
                        counts[c] ? ew + (VEC ? es[c] - 1022 : 0) + n * ey + (__float_as_int(m) >> 23) - 126 : DIR_NO_E);
                    if ((tid & 31) == 0) atomicMax(&s_E[c][n], E);
                }
            }
            if (tid < n_el) {  // at most one more a time, and never fewer
#pragma unroll
                for (int q = 2; q >= 0; --q) needs[q] = max(needs[q], needs[q + 1] - 1);
                int bits = 0, u = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (needs[q] > u) {
                        bits |= 1 << q;
                        ++u;
                    }
                rec[tid * D::REC + D::R_EXP].x = ew * 16 + bits;
            }
        }
        __syncthreads();

        // ---- the recurrences: this thread's direction, elements g, g + G, ..
        if (g < G) {
            longlong2* at0 = acc + tid;
            if (g >= n_el) {
                // (summed over the first min(G, n_el) groups only)
            } else if (pL >= 0) {
#pragma unroll 1
                for (int e = g; e < n_el; e += G) {
                    const bool add = e >= G;
                    const int2* r = rec + e * D::REC;
                    Mul u[NV];
                    Mul nu{};
                    {
                        Fx da[6];
                        dir_of(dirs, j, da);
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            const long long yv[3] = {as_ll(r[3 * k]), as_ll(r[3 * k + 1]), as_ll(r[3 * k + 2])};
                            u[k] = mul_of(dir_dot(da, yv, rnd), dir_dot(da + 3, yv, rnd));
                        }
                        if (DBL) {
                            const long long nv[3] = {as_ll(r[D::R_NRM]), as_ll(r[D::R_NRM + 1]), as_ll(r[D::R_NRM + 2])};
                            nu = mul_of(dir_dot(da, nv, rnd), dir_dot(da + 3, nv, rnd));
                        }
                    }
                    Fx s1{}, s2{}, s3{};
                    if (LIN || VEC) {
                        s1 = as_fx(r[D::R_DENS]);
                        s2 = as_fx(r[D::R_DENS + 1]);
                        s3 = as_fx(r[D::R_DENS + 2]);
                    }
                    const int2 xp = r[D::R_EXP];
                    const long long seed = as_ll(r[D::R_SEED]);
                    const int ey = xp.y >> 17, lf = xp.y & 0x1ffff;
                    int esv[3] = {0, 0, 0};
                    if (VEC) {
                        const int2 c = r[D::R_EXP + (VEC ? 1 : 0)];
                        esv[0] = c.x >> 16;
                        esv[1] = (c.x & 0xffff) - 1022;
                        esv[2] = c.y;
                    }
                    // a value at degree n is 2^-(s_E[n] + off) units of the sums; off is
                    // followed down the degrees
                    int off = D::SEED - D::ACC - (xp.x >> 4), ls = 0, bits = xp.x & 15;
                    const auto amount = [&](int c, int n) { return s_E[c][n] + off - esv[c]; };
                    // degree 0: every level equals the seed (linear: its densities' sums)
                    Cx x[NL];
                    CxH h[NL];
                    long long E0 = seed, W0 = seed;
                    if (LIN) {
                        const int sh = high_of(seed);
                        E0 = mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)seed, sh, (int)seed, sh, 0, rnd);
                        W0 = mul1(s1, (int)seed, sh, E0, rnd);
                    }
                    longlong2* at = at0;
                    longlong2* at1 = at0 + (SGL ? (a.p_max + 1) * NT : 0);
                    const auto add_to = [&](longlong2* p, long long re, long long im) {
                        if (add) {
                            const longlong2 b = *p;
                            re += b.x;
                            im += b.y;
                        }
                        *p = make_longlong2(re, im);
                    };
                    // rounded, and shifted either way; else down (half a unit a live
                    // element is added to the tile's sums)
                    const auto put = [&](auto tight_c, longlong2* p, const Cx& v, int sh) {
                        const int l = max(-sh, 0);
                        if constexpr (decltype(tight_c)::value) {
                            const int r = min(max(sh, 0), 63);
                            const long long half = (long long)((1ull << r) >> 1);
                            add_to(p, ((v.re << l) + half) >> r, ((v.im << l) + half) >> r);
                        } else {
                            const int r = max(sh, 0);
                            add_to(p, shift_down(v.re << l, r), shift_down(v.im << l, r));
                        }
                    };
                    int sh = 0;
                    static_for<0, NE>([&](auto c_c) {  // a vector density's three sums, the weights times the unit-density value
                        constexpr int c = decltype(c_c)::value;
                        const Fx sc = c == 0 ? s1 : c == 1 ? s2 : s3;
                        sh = amount(c, 0);
                        if (SGL)
                            put(std::true_type{}, at + c * (a.p_max + 1) * NT,
                                Cx{VEC ? mul1(sc, (int)seed, high_of(seed), 0, rnd) : W0, 0}, sh);
                    });
                    if (DBL) add_to(at1, 0, 0);
                    static_for<0, NL>([&](auto k_c) {
                        constexpr int k = decltype(k_c)::value;
                        x[k] = Cx{LIN && k == 2 ? E0 : LIN && k == 4 ? W0 : seed, 0};
                    });
                    int ue = 0;
                    long long rs = rnd;  // with a source that is rounded down in its shift by ue
                    // odd_c: the degrees that begin with the lengths' shift; the step before
                    // leaves h of the new values to it
                    const auto step = [&](auto odd_c, int n) {
                        constexpr bool odd = decltype(odd_c)::value;
                        if constexpr (odd) {
                            const bool halve = (n & (n + 1)) == 0 && (bits & 1);
                            if ((n & (n + 1)) == 0) bits >>= 1;
                            if (halve) {
                                ++ue;
                                off -= D::ORDER;
                                sh -= D::ORDER;
                                rs = rnd + (1ll << 30) - ((1ll << 30) >> ue);
                                static_for<0, NL>([&](auto k_c) {
                                    constexpr int k = decltype(k_c)::value, o = D::order(k);
                                    constexpr long long half = (1ll << o) >> 1;
                                    if (o) x[k] = Cx{(x[k].re + half) >> o, (x[k].im + half) >> o};
                                });
                            }
                            const int l = ((n - 1) * lf) >> 16, d = l - ls;
                            ls = l;
                            off += d;
                            sh += d;
                            static_for<0, NL>([&](auto k_c) {
                                constexpr int k = decltype(k_c)::value;
                                x[k] = Cx{x[k].re << d, x[k].im << d};
                                h[k] = high_of(x[k]);
                            });
                        }
                        const auto down = [&](const Cx& v) { return Cx{v.re >> ue, v.im >> ue}; };
                        if (DBL) {
                            at1 += NT;
                            put(std::true_type{}, at1, mul_add<false>(nu, x[NL - 1], h[NL - 1], Cx{0, 0}, rnd),
                                sh - 1);  // (half the normal: a unit half as large)
                        }
                        off -= ey;
                        if constexpr (LIN) {
                            x[0] = mul_add<false>(u[1], x[0], h[0], Cx{0, 0}, rnd);
                            const long long half = (1ll << ue) >> 1;  // (rounded: the factor n + 1 follows)
                            const Cx q{(x[0].re + half) >> ue, (x[0].im + half) >> ue};
                            x[1] = mul_add<true>(u[2], x[1], h[1], q, rnd);
                            h[1] = high_of(x[1]);
                            const long long qr = q.re * (n + 1), qi = q.im * (n + 1);
                            const Cx E{mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)qr, high_of(qr), (int)x[1].re, h[1].rh, 0,
                                                   rnd),
                                       mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)qi, high_of(qi), (int)x[1].im, h[1].ih, 0,
                                                   rnd)};
                            x[2] = mul_add<true>(u[2], x[2], h[2], down(E), rs);
                            x[3] = mul_add<true>(u[0], x[3], h[3], down(x[1]), rs);
                            h[3] = high_of(x[3]);
                            const Cx W{mul1(s1, (int)x[3].re, h[3].rh, x[2].re, rnd),
                                       mul1(s1, (int)x[3].im, h[3].ih, x[2].im, rnd)};
                            x[4] = mul_add<true>(u[0], x[4], h[4], down(W), rs);
                            if constexpr (odd) {
                                h[0] = high_of(x[0]);
                                h[2] = high_of(x[2]);
                                h[4] = high_of(x[4]);
                            }
                        } else {
                            static_for<0, NL>([&](auto k_c) {
                                constexpr int k = decltype(k_c)::value;
                                constexpr int v = (k == NL - 1) ? 0 : k + 1;  // x2, x3, x4, then x1
                                x[k] = mul_add<(k > 0)>(u[v], x[k], h[k], down(x[k > 0 ? k - 1 : 0]), k > 0 ? rs : rnd);
                                if (odd || (VEC && k == NL - 1)) h[k] = high_of(x[k]);
                            });
                        }
                        at += SGL ? NT : 0;
                        static_for<0, NE>([&](auto c_c) {
                            constexpr int c = decltype(c_c)::value;
                            const Fx sc = c == 0 ? s1 : c == 1 ? s2 : s3;
                            sh = amount(c, n);
                            if (VEC)
                                put(std::false_type{}, at + c * (a.p_max + 1) * NT,
                                    Cx{mul1(sc, (int)x[NL - 1].re, h[NL - 1].rh, 0, rnd),
                                       mul1(sc, (int)x[NL - 1].im, h[NL - 1].ih, 0, rnd)},
                                    sh);
                            else if (SGL)
                                put(std::integral_constant<bool, D::TIGHT>{}, at, x[NL - 1], sh);
                        });
                    };
#pragma unroll 1
                    for (int n = 1; n <= pL; n += 2) {
                        step(std::true_type{}, n);
                        if (n == pL) break;
                        step(std::false_type{}, n + 1);
                    }
                }
            }
        }
        __syncthreads();

        // ---- sums over the groups, 96-bit, cut to 56 bits of each degree's
        // largest: a warp per degree and layer, so that the largest is a warp
        // reduction
        const int Ga = min(G, n_el);
        int2* sums = rec;  // [layer][degree][2 J]
        for (int r = tid >> 5; r < (pL + 1) * D::LAYERS; r += NT >> 5) {
            int ly = 0, n = r;
            while (n > pL) n -= pL + 1, ++ly;
            long long H[2] = {0, 0}, Lo[2] = {0, 0};
            int bits = 0;
#pragma unroll
            for (int c = 0; c < 2; ++c) {  // 2 J <= 42 columns
                const int q = (tid & 31) + 32 * c;
                if (q < 2 * J) {
                    const long long* p = reinterpret_cast<const long long*>(acc + (ly * (a.p_max + 1) + n) * NT) + q;
#pragma unroll 4
                    for (int k = 0; k < Ga; ++k) {
                        const long long v = p[k * 2 * J];
                        H[c] += hi32(v);
                        Lo[c] += (unsigned)(int)v;
                    }
                    if (n > 0 && !D::TIGHT && SGL && (VEC || ly == 0)) Lo[c] += s_live[VEC ? ly : 0] >> 1;  // (rounded down)
                    H[c] += Lo[c] >> 32;
                    bits = max(bits, 64 - __clzll(H[c] < 0 ? ~H[c] : H[c]));
                }
            }
            bits = __reduce_max_sync(0xffffffffu, bits);  // |value| < 2^(bits + 32) -> below 2^56
            const int sh = bits - 24;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int q = (tid & 31) + 32 * c;
                if (q < 2 * J) {
                    const unsigned long long hi = (unsigned long long)H[c], lo = (unsigned)(int)Lo[c];
                    long long o;
                    if (sh <= 0)
                        o = (long long)((hi << 32) | lo) << -sh;
                    else if (sh < 32)
                        o = (long long)((hi << (32 - sh)) | (lo >> sh));
                    else
                        o = H[c] >> (sh - 32);
                    const int hq = (int)((o + (1ll << 27)) >> 28);
                    sums[r * 2 * J + q] = make_int2(hq, (int)(o - ((long long)hq << 28)));
                }
            }
            if ((tid & 31) == 0) s_bits[ly][n] = bits;
        }
        __syncthreads();

        // ---- coefficients: the left inverse's row of each packed column
        const bool direct = (t.flags & 1) != 0;
        for (int i = tid; i < np * D::LAYERS; i += NT) {
            int ly = 0, k = i;
            while (k >= np) k -= np, ++ly;
            const bool second = !VEC && (!SGL || ly == 1);  // double layer
            const int desc = col_desc(k), n = desc & 31;
            double v = 0.0;
            if (n <= pL) {
                const int2* P = a.inv + k;
                const int2* S = sums + (ly * (pL + 1) + n) * 2 * J;
                long long hh = 0, mid = 1ll << 27;
#pragma unroll 8
                for (int q = 0; q < 2 * J; ++q) {
                    const int2 c = __ldg(P + q * np);
                    const int2 x = S[q];
                    mid = madw(c.x, x.y, mid);
                    mid = madw(c.y, x.x, mid);
                    hh = madw(c.x, x.x, hh);
                }
                hh += mid >> 28;
                constexpr int d0 = LIN ? 3 : KIND + 1;
                const int d = second ? d0 - 1 : d0;
                const int ns = second ? n - 1 : n;  // the frame's power
                v = (double)hh * __ldg(a.col + (a.norm * 4 + d) * 441 + k);
                if (second && n == 0) v = 0.0;
                int e2 = s_bits[ly][n] - 24 - 2 - D::ACC + s_E[VEC ? ly : 0][max(ns, 0)];
                if (LIN || VEC) e2 += 1;
                if (e2 > 1000 || e2 < -1000) {
                    const int h = max(-2000, min(2000, e2)) / 2;
                    v *= pow2d(h);
                    e2 = max(-2000, min(2000, e2)) - h;
                }
                v *= pow2d(e2);
                if ((desc >> (5 + a.norm)) & 1) v = -v;
                if (s_over) v = __longlong_as_double(0x7ff8000000000000ll);
            }
            if (VEC && a.coef[ly] == nullptr) continue;
            double* out = (direct ? a.coef[ly] + L * np : a.partial[ly] + t.slot * np) + k;
            *out = (direct && a.accumulate) ? *out + v : v;
        }
    }
}

struct DirFns {
    cudaError_t (*launch)(const DirArgs&, int nt, int T, int grid, cudaStream_t);
    cudaError_t (*occupancy)(int* blocks_per_sm, int p, int nt, int T);
};
// [CTA class: 0 up to 256 threads, 1 up to 128][combo]; combos: 0 segments, 1-3
// triangles constant density (single, double, both), 4-6 linear density, 7
// tetrahedra, 8 segments carrying a vector density (the element kernel's
// order), 9 and 10 the receiver side, single layer and normal derivative
const DirFns& dir_fns(int cls, int combo);
// A call's CTAs: class, threads, elements per tile.
struct DirShape {
    int cls, nt, T;
};
DirShape dir_shape(int p, int layers, int64_t n_elem, int64_t n_leaves, int num_sms);
// The most tiles dir_shape can cut up to n_elem elements into, leaves apart:
// full tiles of the smallest CTA, or, where they are spread over the SMs, tiles
// of at least n_elem / num_sms (rounded down, so up to two an SM).
int64_t dir_most_tiles(int p, int64_t n_elem, int num_sms);
// Elements a tile may hold: eight a group (the number format's head room), at
// most one a thread (the frames).
inline int dir_tile_elems(int p, int nt)
{
    const int t = 8 * (nt / (p + 1));
    return t < nt ? t : nt;
}
// The device tables of degree bound p: vectors [J][6], left inverse [2 J][np],
// column constants [norm][d][441].
struct DirTables {
    const int2 *vec, *inv;
    const double* col;
};
cudaError_t dir_tables(int p, DirTables* t);
// Fills the tables and group counts of a call (a.p_max set).
cudaError_t dir_setup(DirArgs& a, int nt);

}  // namespace q2x
