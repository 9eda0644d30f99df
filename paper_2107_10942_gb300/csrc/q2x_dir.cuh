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
// |u| < 1 is kept to 2^-62 and a value x to one unit of a 60-bit integer, both
// as two 32-bit halves, and a real product is three multiply-adds.  Each step
// rounds to about a unit of 2^-59 of the level's bound (FP64: 2^-53 of the
// value), so the sums are as near the exact ones as the FP64 row kernel's
// (measured over kinds, degrees and leaf sizes).  The tile's own scales keep
// the format filled whatever the units of the input: vertices are scaled by
// the tile's radius (in steps of 2^(1/8), exact to 62 bits), seeds J sigma by
// their largest.
//
// What bounds it: the integer multiplies, 36 per step of the triangle chain
// (190 cycles with the additions between them; 196 measured in a loop of its
// own), then the tile's other phases: of the level-9 sphere's 11.2 ms at p =
// 16 the recurrences are 64 %, the map to coefficients and the frames 13 %
// each, the sums over groups 8 %.  The FP64 row kernel took 36.2 ms.
//
// One CTA per tile of one leaf's elements: thread t < G J owns direction
// t mod J and elements t / J, t / J + G, .. (at most eight, the number
// format's head room).  The accumulators, one complex number per degree and
// thread, live in shared memory: one 16-byte load and store per step cost
// nothing beside its multiplies, and the degree loop needs no registers per
// degree, so one kernel serves every degree.
#pragma once

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

// A 62-bit fixed-point constant as h 2^31 + l, |l| <= 2^30.
struct Fx {
    int h, l;
};
Q2X_HD Fx fx_split(long long v)
{
    Fx f;
    f.h = (int)((v + (1ll << 30)) >> 31);
    f.l = (int)(v - ((long long)f.h << 31));
    return f;
}

// A running value: the integer v (|v| < 2^60 for recurrence values, < 2^62
// for the multipliers u) stored as v + BIAS 2^32, and h with
// v = h 2^31 + (int)v (h even).
struct Cx {
    long long re, im;
};
struct CxH {
    int rh, ih;
};
template <int BIAS>
Q2X_HD int high_of(long long v)
{
    const int h = (int)((unsigned)hi32(v) + ((unsigned)(int)v >> 31));
    return h + h - 2 * BIAS;
}
template <int BIAS>
Q2X_HD CxH high_of(const Cx& x)
{
    return CxH{high_of<BIAS>(x.re), high_of<BIAS>(x.im)};
}
__host__ __device__ constexpr long long dir_bias(int k) { return (long long)k << 32; }

// A complex multiplier: halves of the parts and of the negated imaginary part.
struct Mul {
    int rh, rl, ih, il, nh, nl;
};
Q2X_HD Mul mul_of(long long re, long long im)
{
    const int ih = high_of<0>(im), il = (int)im;
    return Mul{high_of<0>(re), (int)re, ih, il, -ih, -il};
}

// a x + b y + s for real a, b (halves ah, al, bh, bl) and values x, y.  The
// low products are summed at 2^-31 of a unit (the products of two low halves
// are below 2^-31 units and are left out); their upper word is worth two
// units.  The sum starts at `rnd` = 2^63 + 2^31, which rounds it and makes it
// positive, so that the word is added twice without a sign extension: the
// result carries 2^32 on top of what s carries.
template <bool S>
Q2X_HD long long mul2(int ah, int al, int bh, int bl, int xl, int xh, int yl, int yh, long long s, long long rnd)
{
    long long o;
    if (S)
        asm("{.reg .b64 a, b, m, z; .reg .b32 t, h;\n"
            "mul.wide.s32 m, %1, %5; add.s64 a, m, %10;\n"
            "mul.wide.s32 m, %2, %6; add.s64 a, a, m;\n"
            "mul.wide.s32 m, %3, %7; add.s64 a, a, m;\n"
            "mul.wide.s32 m, %4, %8; add.s64 a, a, m;\n"
            "mov.b64 {t, h}, a;\n"
            "mul.wide.s32 m, %1, %6; add.s64 b, m, %9;\n"
            "mul.wide.s32 m, %3, %8; add.s64 b, b, m;\n"
            "cvt.u64.u32 z, h; add.s64 b, b, z; add.s64 %0, b, z;}"
            : "=l"(o)
            : "r"(ah), "r"(al), "r"(bh), "r"(bl), "r"(xl), "r"(xh), "r"(yl), "r"(yh), "l"(s), "l"(rnd));
    else
        asm("{.reg .b64 a, b, m, z; .reg .b32 t, h;\n"
            "mul.wide.s32 m, %1, %5; add.s64 a, m, %9;\n"
            "mul.wide.s32 m, %2, %6; add.s64 a, a, m;\n"
            "mul.wide.s32 m, %3, %7; add.s64 a, a, m;\n"
            "mul.wide.s32 m, %4, %8; add.s64 a, a, m;\n"
            "mov.b64 {t, h}, a;\n"
            "mul.wide.s32 b, %1, %6;\n"
            "mul.wide.s32 m, %3, %8; add.s64 b, b, m;\n"
            "cvt.u64.u32 z, h; add.s64 b, b, z; add.s64 %0, b, z;}"
            : "=l"(o)
            : "r"(ah), "r"(al), "r"(bh), "r"(bl), "r"(xl), "r"(xh), "r"(yl), "r"(yh), "l"(rnd));
    return o;
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
    asm("{.reg .b64 a, b, m, z; .reg .b32 t, h;\n"
        "mul.wide.s32 m, %1, %3; add.s64 a, m, %6;\n"
        "mul.wide.s32 m, %2, %4; add.s64 a, a, m;\n"
        "mov.b64 {t, h}, a;\n"
        "mul.wide.s32 m, %1, %4; add.s64 b, m, %5;\n"
        "cvt.u64.u32 z, h; add.s64 b, b, z; add.s64 %0, b, z;}"
        : "=l"(o)
        : "r"(a.h), "r"(a.l), "r"(xl), "r"(xh), "l"(s), "l"(rnd));
    return o;
}
// a . y of one direction part (three Fx) and a point (three Fx), in the same
// form: 62-bit fixed point, without a bias
Q2X_HD long long dir_dot(const Fx* a, const Fx* y, long long rnd)
{
    const long long o = mul2<false>(a[0].h, a[0].l, a[1].h, a[1].l, y[0].l, y[0].h, y[1].l, y[1].h, 0, rnd);
    return mul1(a[2], y[2].l, y[2].h, o, rnd) - dir_bias(2);
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
    int seed_bits;     // a seed's largest magnitude is 2^seed_bits
    int event[4];      // before each of these degrees every value is divided by 2^DIR_EVENT
    long long rnd;     // mul2's start
    const int2* vec;     // [J][6]
    const int2* inv;     // [2 J][np]
    const int2* eighth;  // [15]
    const double* pw;    // [15][24]
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
constexpr int DIR_EVENT = 3;  // bits dropped when the values' bound has grown by them
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
    // what the stored values of level k carry, in units of 2^32 (mul2)
    __host__ __device__ static constexpr int bias(int k) { return LIN && k >= 2 ? k : k + 1; }
    static constexpr int LAYERS = VEC ? 3 : (SGL ? 1 : 0) + (DBL ? 1 : 0);
    // 8-byte words of a record: vertices, then the normal, then the densities, then the seed
    static constexpr int R_NRM = 3 * NV, R_DENS = R_NRM + (DBL ? 3 : 0), R_SEED = R_DENS + (LIN || VEC ? 3 : 0);
    static constexpr int REC = R_SEED + 1;
    __host__ __device__ static constexpr size_t rec_bytes(int p, int T)
    {
        // the records' space is reused for the sums
        const size_t a = (size_t)T * REC * 8, s = (size_t)(p + 1) * 2 * (p + 1) * LAYERS * 8;
        return ((a > s ? a : s) + 15) / 16 * 16;
    }
    // receiver side: the fixed-point weights [degree][direction] (16 bytes), the
    // scaled column weights (8) and products (8) they come from, and the
    // elements' values per direction [element][direction]
    __host__ __device__ static constexpr size_t gal_bytes(int p)
    {
        return (size_t)(p + 1) * (p + 1) * 40 + 16;
    }
    __host__ __device__ static constexpr size_t smem(int p, int T, int nt)
    {
        if (GAL) return (size_t)(p + 1) * 48 + ((size_t)T * REC * 8 + 15) / 16 * 16 + gal_bytes(p) + (size_t)T * (p + 1) * 8;
        return (size_t)(p + 1) * 48 + rec_bytes(p, T) + (size_t)LAYERS * (p + 1) * nt * 16;
    }
};

__device__ __forceinline__ Fx as_fx(int2 v) { return Fx{v.x, v.y}; }

// Receiver side: out[e] = sum_c w_c P_c(e) over the packed columns c of an
// element's own coefficients.  The weights are carried to the directions
// (the transposed map, exact products per degree), and sum_n W_n h_n(u1, u2,
// u3) of the chain's values h is nested Horner steps from the highest degree
// down, one per level and degree:
//   c_n = W_n + u1 c_{n+1}, b_n = c_n + u3 b_{n+1}, a_n = b_n + u2 a_{n+1},
// the value a_0 (double layer: of the weights one degree up, times the
// normal's multiplier).  The weights are scaled so that the bound of all
// partial sums is 2^59.
template <typename D>
__device__ __forceinline__ void dir_gal_tile(const DirArgs& a, int T, const BatchTile& t, int n_el, int kr, int ex,
                                             int Ej, const int2* rec, const int2* dirs, int g, int j)
{
    constexpr bool DBL = D::DBL;
    const int tid = threadIdx.x, lane = tid & 31, NT = blockDim.x;
    const int J = a.J, p = a.p_max, np = a.np;
    unsigned char* base = reinterpret_cast<unsigned char*>(const_cast<int2*>(rec)) + ((size_t)T * D::REC * 8 + 15) / 16 * 16;
    longlong2* W = reinterpret_cast<longlong2*>(base);                       // [p + 1][J]
    long long* prod = reinterpret_cast<long long*>(W + (p + 1) * J);         // [p + 1][2 J]
    int2* col = reinterpret_cast<int2*>(prod + (p + 1) * 2 * J);             // [np]
    long long* val = reinterpret_cast<long long*>(base + D::gal_bytes(p));   // [T][J]
    __shared__ int s_e[Q2X_P_MAX + 1], s_scale;
    __shared__ double s_sum[Q2X_P_MAX + 1];
    constexpr int d = DBL ? KIND_TRI : KIND_TRI + 1;
    const double* w = a.gal_w + (int64_t)t.leaf * np;
    for (int n = tid >> 5; n <= p; n += NT >> 5) {
        const int ns = DBL ? n - 1 : n;  // the frame's power
        const double fr = ns > 0 ? __ldg(a.pw + (kr + 7) * 24 + ns) : 1.0;
        double v[2] = {0.0, 0.0};
        int top = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q = lane + 32 * c;
            if (q <= 2 * n && !(DBL && n == 0)) {
                const int k = n * n + q;
                v[c] = __ldg(w + k) * __ldg(a.col + (a.norm * 4 + d) * 441 + k) * fr;
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
        double sum = 0.0;
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
                prod[n * 2 * J + s] = hh;
                sum += fabs((double)hh);
            }
        }
        for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) {
            // (weights beyond FP64 make the tile's results NaN)
            s_sum[n] = top < 0x7ff00000 ? sum * (DBL ? 0.5 * n * (n + 1) : 0.5 * (n + 1) * (n + 2))
                                        : __longlong_as_double(0x7ff0000000000000ll);
            s_e[n] = e1 - 1022 - 58 + (ns > 0 ? ns * (ex - 1022) : 0);
        }
    }
    __syncthreads();
    if (tid == 0) {
        int most = -1000000;
        for (int n = 0; n <= p; ++n)
            if (s_sum[n] > 0.0) most = max(most, s_e[n] + (hi32(__double_as_longlong(s_sum[n])) >> 20) - 1022);
        double B = 0.0;
        for (int n = 0; n <= p; ++n) B += s_sum[n] * pow2d(max(s_e[n] - most, -1000));
        int scale = 0;
        if (B > 0.0) scale = 59 - (most + (hi32(__double_as_longlong(B)) >> 20) - 1022);
        s_scale = B < 1e300 ? scale : 0x7fffffff;
    }
    __syncthreads();
    const int scale = s_scale;
    for (int i = tid; i < (p + 1) * J; i += NT) {
        const int n = i / J, jj = i - n * J;
        const int sh = scale == 0x7fffffff ? -100 : s_e[n] + scale;
        auto put = [&](long long v) {
            if (sh >= 0) return v << min(sh, 62);
            if (sh < -62) return 0ll;
            return (v + (1ll << (-sh - 1))) >> -sh;
        };
        longlong2 o;
        o.x = put(prod[n * 2 * J + 2 * jj]);
        o.y = -put(prod[n * 2 * J + 2 * jj + 1]);
        W[i] = o;
    }
    __syncthreads();
    const long long rnd = a.rnd;
    if (g < a.G) {
#pragma unroll 1
        for (int e = g; e < n_el; e += a.G) {
            const int2* r = rec + e * D::REC;
            Mul u[3], nu{};
            {
                Fx da[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) da[c] = as_fx(dirs[j * 6 + c]);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const Fx y[3] = {as_fx(r[3 * k]), as_fx(r[3 * k + 1]), as_fx(r[3 * k + 2])};
                    u[k] = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
                }
                if (DBL) {
                    const Fx y[3] = {as_fx(r[D::R_NRM]), as_fx(r[D::R_NRM + 1]), as_fx(r[D::R_NRM + 2])};
                    nu = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
                }
            }
            long long res = 0;
            if (!DBL || p > 0) {
                const longlong2* q = W + p * J + j;
                longlong2 w0 = *q;
                Cx c{w0.x + dir_bias(1), w0.y + dir_bias(1)}, b{w0.x + dir_bias(2), w0.y + dir_bias(2)},
                    x{w0.x + dir_bias(3), w0.y + dir_bias(3)};
                CxH hc = high_of<1>(c), hb = high_of<2>(b), hx = high_of<3>(x);
#pragma unroll 4
                for (int n = p - 1; n >= (DBL ? 1 : 0); --n) {
                    q -= J;
                    w0 = *q;
                    c = mul_add<true>(u[0], c, hc, Cx{w0.x, w0.y}, rnd);
                    hc = high_of<1>(c);
                    b = mul_add<true>(u[2], b, hb, c, rnd);
                    hb = high_of<2>(b);
                    x = mul_add<true>(u[1], x, hx, b, rnd);
                    hx = high_of<3>(x);
                }
                if (DBL)
                    res = mul2<false>(nu.rh, nu.rl, nu.nh, nu.nl, (int)x.re, hx.rh, (int)x.im, hx.ih, 0, rnd) - dir_bias(1);
                else
                    res = x.re - dir_bias(3);
            }
            val[e * J + j] = res;
        }
    }
    __syncthreads();
    if (tid < n_el) {
        long long sum = 0;
        for (int k = 0; k < J; ++k) sum += val[tid * J + k];
        const int2 sd = rec[tid * D::REC + D::R_SEED];
        double v = (double)sum * __longlong_as_double(((long long)sd.y << 32) | (unsigned)sd.x);
        int e2 = -scale + (DBL ? 1 : 0) + (KIND_TRI + 1) * Ej;  // (half the normal)
        if (e2 > 1000 || e2 < -1000) {
            const int h = max(-2000, min(2000, e2)) / 2;
            v *= pow2d(h);
            e2 = max(-2000, min(2000, e2)) - h;
        }
        v *= pow2d(e2);
        if (scale == 0x7fffffff) v = __longlong_as_double(0x7ff8000000000000ll);
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
    __shared__ int s_more, s_ymax, s_r2, s_wmax, s_smax, s_bits[3][Q2X_P_MAX + 1];
    for (int i = tid; i < 6 * J; i += NT) dirs[i] = a.vec[i];
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
            s_ymax = s_r2 = s_wmax = s_smax = 0;
        }
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
        int ym = 0;
        bool over = false;  // a difference of finite coordinates that overflows
        if (live) {
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) ym = max(ym, hi32(__double_as_longlong(y[k][d])) & 0x7fffffff);
            over = ym >= 0x7ff00000;
            if (over) live = false;
        }
        {
            const int m = __reduce_max_sync(0xffffffffu, live ? ym : 0);
            if ((tid & 31) == 0 && m) atomicMax(&s_ymax, m);
        }
        __syncthreads();
        const int ex = max(s_ymax >> 20, 1);  // |y| < 2^(ex - 1022)
        long long yi[NV][3];
        int r2i = 0, sm = 0, wm = 0;
        // edges scaled (exactly) where their products could leave the range
        const int Ej = (ex - 1022 > 200 || ex - 1022 < -200) ? ex - 1022 : 0;
        if (live) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float r2 = 0.f;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    yi[k][d] = dir_fixed((unsigned long long)__double_as_longlong(y[k][d]), ex, 61);
                    const float f = (float)hi32(yi[k][d]) * 1.862645149230957e-9f;  // 2^-29
                    r2 = fmaf(f, f, r2);
                }
                r2i = max(r2i, __float_as_int(r2));
            }
            if (Ej) {
                const double es = pow2d(-Ej);
#pragma unroll
                for (int k = 0; k < NV - 1; ++k)
#pragma unroll
                    for (int d = 0; d < 3; ++d) ed[k][d] *= es;
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
            wm = hi32(__double_as_longlong(w)) & 0x7fffffff;
            if (LIN || VEC) {
#pragma unroll
                for (int k = 0; k < 3; ++k) sm = max(sm, hi32(__double_as_longlong(s[k])) & 0x7fffffff);
            }
        }
        if (over) wm = 0x7ff00000;
        {
            const int m = __reduce_max_sync(0xffffffffu, r2i);
            const int mw = __reduce_max_sync(0xffffffffu, wm);
            const int ms = (LIN || VEC) ? __reduce_max_sync(0xffffffffu, sm) : 0;
            if ((tid & 31) == 0) {
                if (m) atomicMax(&s_r2, m);
                if (mw) atomicMax(&s_wmax, mw);
                if ((LIN || VEC) && ms) atomicMax(&s_smax, ms);
            }
        }
        __syncthreads();
        const int wmax = s_wmax;
        const int ew = max(wmax >> 20, 1), es = max(s_smax >> 20, 1);
        // the radius step: the largest k in -7..7 with r 2^(k/8) below one
        int kr = 7;
        {
            const float r2 = __int_as_float(s_r2);
            if (r2 > 0.f) kr = max(-7, min(7, (int)floorf(4.f * log2f(0.998f / r2))));
        }
        if (tid < n_el) {
            const Fx C = as_fx(__ldg(a.eighth + kr + 7));
            int2* r = rec + tid * D::REC;
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    long long v = 0;
                    if (live) {
                        const Fx q = fx_split(yi[k][d]);
                        v = (madw(q.h, C.l, madw(q.l, C.h, 1ll << 30)) >> 31) + (long long)q.h * C.h;
                        v *= 4;
                    }
                    const Fx f = fx_split(v);
                    r[3 * k + d] = make_int2(f.h, f.l);
                }
            if (DBL) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {  // half the unit normal
                    const Fx f = fx_split(
                        live ? dir_fixed((unsigned long long)__double_as_longlong(nrm[d]), 1023, 62) : 0);
                    r[D::R_NRM + d] = make_int2(f.h, f.l);
                }
            }
            if (LIN || VEC) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {  // half the scaled densities: below one also when rounded
                    const Fx f = fx_split(live ? dir_fixed((unsigned long long)__double_as_longlong(s[k]), es, 61) : 0);
                    r[D::R_DENS + k] = make_int2(f.h, f.l);
                }
            }
            long long sd = 0;
            if (GAL)  // the factor of the element's value
                sd = live ? __double_as_longlong(w) : over ? 0x7ff8000000000000ll : 0;
            else if (live && wmax < 0x7ff00000)
                sd = dir_fixed((unsigned long long)__double_as_longlong(w), ew, a.seed_bits);
            r[D::R_SEED] = make_int2((int)sd, hi32(sd));
        }
        __syncthreads();
        if constexpr (GAL) {
            dir_gal_tile<D>(a, T, t, n_el, kr, ex, Ej, rec, dirs, g, j);
            continue;
        }

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
#pragma unroll
                        for (int d = 0; d < 6; ++d) da[d] = as_fx(dirs[j * 6 + d]);
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            Fx yv[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d) yv[d] = as_fx(r[3 * k + d]);
                            u[k] = mul_of(dir_dot(da, yv, rnd), dir_dot(da + 3, yv, rnd));
                        }
                        if (DBL) {
                            Fx nv[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d) nv[d] = as_fx(r[D::R_NRM + d]);
                            nu = mul_of(dir_dot(da, nv, rnd), dir_dot(da + 3, nv, rnd));
                        }
                    }
                    Fx s1{}, s2{}, s3{};
                    if (LIN || VEC) {
                        s1 = as_fx(r[D::R_DENS]);
                        s2 = as_fx(r[D::R_DENS + 1]);
                        s3 = as_fx(r[D::R_DENS + 2]);
                    }
                    const int2 sd = r[D::R_SEED];
                    const long long seed = ((long long)sd.y << 32) | (unsigned)sd.x;
                    // degree 0: every level equals the seed (linear: its densities' sums)
                    Cx x[NL];
                    CxH h[NL];
                    long long E0 = seed, W0 = seed;
                    if (LIN) {
                        const int sh = high_of<0>(seed);
                        E0 = mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)seed, sh, (int)seed, sh, 0, rnd);
                        W0 = mul1(s1, (int)seed, sh, E0, rnd) - dir_bias(2);
                        E0 -= dir_bias(1);
                    }
                    longlong2* at = at0;
                    longlong2* at1 = at0 + (SGL ? (a.p_max + 1) * NT : 0);
                    auto put = [&](longlong2* p, const Cx& v) {
                        longlong2 o = make_longlong2(v.re, v.im);
                        if (add) {
                            const longlong2 b = *p;
                            o.x += b.x;
                            o.y += b.y;
                        }
                        *p = o;
                    };
                    // a vector density's three sums, the weights times the unit-density value
                    auto put3 = [&](longlong2* p, const Cx& v, const CxH& vh, long long b) {
                        const int st = (a.p_max + 1) * NT;
                        put(p, Cx{mul1(s1, (int)v.re, vh.rh, -b, rnd), mul1(s1, (int)v.im, vh.ih, -b, rnd)});
                        put(p + st, Cx{mul1(s2, (int)v.re, vh.rh, -b, rnd), mul1(s2, (int)v.im, vh.ih, -b, rnd)});
                        put(p + 2 * st, Cx{mul1(s3, (int)v.re, vh.rh, -b, rnd), mul1(s3, (int)v.im, vh.ih, -b, rnd)});
                    };
                    if (VEC)
                        put3(at, Cx{seed, 0}, CxH{high_of<0>(seed), 0}, dir_bias(1));
                    else if (SGL)
                        put(at, Cx{W0, 0});
                    if (DBL) put(at1, Cx{0, 0});
                    static_for<0, NL>([&](auto k_c) {
                        constexpr int k = decltype(k_c)::value, B = D::bias(k);
                        x[k] = Cx{(LIN && k == 2 ? E0 : LIN && k == 4 ? W0 : seed) + dir_bias(B), dir_bias(B)};
                        h[k] = high_of<B>(x[k]);
                    });
                    auto steps = [&](int n0, int n1) {
#pragma unroll 4
                        for (int n = n0; n < n1; ++n) {
                            if (DBL) {
                                at1 += NT;
                                put(at1, mul_add<false>(nu, x[NL - 1], h[NL - 1], Cx{0, 0}, rnd));
                            }
                            if constexpr (LIN) {
                                x[0] = mul_add<false>(u[1], x[0], h[0], Cx{0, 0}, rnd);
                                h[0] = high_of<1>(x[0]);
                                x[1] = mul_add<true>(u[2], x[1], h[1], x[0], rnd);
                                h[1] = high_of<2>(x[1]);
                                const long long qr = (x[0].re - dir_bias(1)) * (n + 1);
                                const long long qi = (x[0].im - dir_bias(1)) * (n + 1);
                                const Cx E{mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)qr, high_of<0>(qr), (int)x[1].re,
                                                       h[1].rh, 0, rnd),
                                           mul2<false>(s2.h, s2.l, s3.h, s3.l, (int)qi, high_of<0>(qi), (int)x[1].im,
                                                       h[1].ih, 0, rnd)};
                                x[2] = mul_add<true>(u[2], x[2], h[2], E, rnd);
                                h[2] = high_of<2>(x[2]);
                                x[3] = mul_add<true>(u[0], x[3], h[3], x[1], rnd);
                                h[3] = high_of<3>(x[3]);
                                const Cx W{mul1(s1, (int)x[3].re, h[3].rh, x[2].re, rnd),
                                           mul1(s1, (int)x[3].im, h[3].ih, x[2].im, rnd)};
                                x[4] = mul_add<true>(u[0], x[4], h[4], W, rnd);
                                h[4] = high_of<4>(x[4]);
                            } else {
                                x[0] = mul_add<false>(u[1], x[0], h[0], Cx{0, 0}, rnd);
                                h[0] = high_of<1>(x[0]);
                                static_for<1, NL>([&](auto k_c) {
                                    constexpr int k = decltype(k_c)::value;
                                    constexpr int v = (k == NL - 1) ? 0 : k + 1;  // x2, x3, x4, then x1
                                    x[k] = mul_add<true>(u[v], x[k], h[k], x[k - 1], rnd);
                                    h[k] = high_of<k + 1>(x[k]);
                                });
                            }
                            if (SGL) {
                                at += NT;
                                if (VEC)
                                    put3(at, x[NL - 1], h[NL - 1], 0);
                                else
                                    put(at, x[NL - 1]);
                            }
                        }
                    };
                    int n0 = 1;
#pragma unroll 1
                    for (int v = 0;; ++v) {
                        const int n1 = v < 4 ? min(a.event[v], pL + 1) : pL + 1;
                        steps(n0, n1);
                        if (n1 > pL) break;
                        n0 = n1;
                        constexpr long long half = 1ll << (DIR_EVENT - 1);
                        static_for<0, NL>([&](auto k_c) {
                            constexpr int k = decltype(k_c)::value, B = D::bias(k);
                            x[k].re = ((x[k].re - dir_bias(B) + half) >> DIR_EVENT) + dir_bias(B);
                            x[k].im = ((x[k].im - dir_bias(B) + half) >> DIR_EVENT) + dir_bias(B);
                            h[k] = high_of<B>(x[k]);
                        });
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
            const bool once = VEC || !SGL || ly == 1;  // a product of the level's value: one bias
            const int bias = n ? n_el * (once ? 1 : D::bias(NL - 1)) : 0;
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
                    H[c] += (Lo[c] >> 32) - bias;
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
                if (ns > 0) v *= __ldg(a.pw + (kr + 7) * 24 + ns);
                int e2 = s_bits[ly][n] - 24 - 2 - a.seed_bits + DIR_EVENT * ((n >= a.event[0]) + (n >= a.event[1]) + (n >= a.event[2]) + (n >= a.event[3])) + (ew - 1022) +
                         (ns > 0 ? ns * (ex - 1022) : 0) + (KIND + 1) * Ej;
                if (second) e2 += 1;
                if (LIN || VEC) e2 += es - 1022 + 1;
                if (e2 > 1000 || e2 < -1000) {
                    const int h = max(-2000, min(2000, e2)) / 2;
                    v *= pow2d(h);
                    e2 = max(-2000, min(2000, e2)) - h;
                }
                v *= pow2d(e2);
                if ((desc >> (5 + a.norm)) & 1) v = -v;
                if (wmax >= 0x7ff00000) v = __longlong_as_double(0x7ff8000000000000ll);
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
// 2^(k/8 - 1) [15], 2^(-k n / 8) [15][24], column constants [norm][d][441].
struct DirTables {
    const int2 *vec, *inv, *eighth;
    const double *pw, *col;
};
cudaError_t dir_tables(int p, DirTables* t);
// Fills the tables, group counts and number format of a call (a.p_max set).
cudaError_t dir_setup(DirArgs& a, int kind, int dens, int nt);

}  // namespace q2x
