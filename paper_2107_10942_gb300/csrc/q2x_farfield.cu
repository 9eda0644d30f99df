// q2x_farfield.cu -- far-field potentials and curls by directions: the path of
// q2x_evaluate and q2x_evaluate_curl for many targets (declared in
// q2x_farfield.h; the general FP64 kernels are in q2x_evaluate.cu).
//
// S_n^m(x) r^(2n+1) = (-1)^(n+m) (n-m)! (n+m)! R_n^m(x) (Eqs. (bas1)-(bas2)),
// so an expansion's potential is (1/r) L(x / r^2) with L = sum_n H_n a sum of
// harmonic polynomials, and each H_n is a combination of the 2 (p + 1) parts
// of (a_j . y)^n for the null vectors a_j of gen_directions.py: with v = a_j . y
//     phi(x) = (1/r) sum_j Re sum_n c_{n,j} v^n,
// one complex Horner step per direction and degree, run in the 64-bit fixed
// point of q2x_dir.cuh.  y = rho x / r^2 with rho just below the distance that
// all but a few of the expansion's targets have, so |v| < 1; the c_{n,j} are
// scaled by the bound of their sums, so no partial sum leaves the format.
//
// Three kernels: how often each distance occurs, per expansion, in a sample of
// the targets; the c_{n,j} of each expansion (one CTA, exact dot products with
// the left inverse's rows); one thread per target over its list.  The fixed
// point's error is relative to the terms at rho, so a target where the terms'
// bound has fallen below a sixteenth of that (far out without a monopole), one
// nearer than rho, and an expansion whose scale leaves FP64, takes the general
// FP64 evaluation.  With rho from the nearest target, one close target sent
// all the others there (2^20 targets at p = 12 1,467 us, now 327; the curl at 2^18
// 2,900, now 517).
#include <cuda_runtime.h>

#include <algorithm>

#include "q2x_dir.cuh"
#include "q2x_farfield.h"

namespace q2x {

namespace {

constexpr int FAR_NT = 128;

// distances are counted in classes of r^2, two an octave, modulo FAR_CLASSES
// (the largest of a residue stands for it)
constexpr int FAR_CLASSES = 32;
constexpr int FAR_SAMPLE = 4096;  // targets an expansion to be counted, on average
constexpr int FAR_FEW = 1024;     // one in so many targets may be nearer than rho

struct FarMeta {
    double rho;  // 0: not usable
    int scale;   // c = value 2^scale
    float bound[Q2X_P_MAX + 1];  // the degrees' shares of the terms' bound at distance rho
};

struct FarArgs {
    EvalArgs ev;
    DirTables tab;
    int J, comps;  // 1 potential, 3 curl
    long long rnd;
    int* count;       // [n_exp][FAR_CLASSES]
    int* cls;         // [n_exp][FAR_CLASSES] the class, upper word of r^2 >> 19
    int64_t step;     // every step'th warp's targets are counted
    FarMeta* meta;    // [n_exp]
    longlong2* c;     // [comps][n_exp][J][p + 1]
};

__device__ __forceinline__ double offset_r2(const EvalArgs& a, int64_t t, int64_t e, double (&x)[3])
{
    x[0] = __ldg(a.tgt + t) - __ldg(a.exp_c + e);
    x[1] = __ldg(a.tgt + a.n_tgt + t) - __ldg(a.exp_c + a.n_exp + e);
    x[2] = __ldg(a.tgt + 2 * a.n_tgt + t) - __ldg(a.exp_c + 2 * a.n_exp + e);
    return x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
}

// the list of target t; bad ranges (reported by the evaluation) are empty
__device__ __forceinline__ void list_of(const EvalArgs& a, int64_t t, int64_t& j0, int64_t& j1, bool& bad)
{
    j0 = __ldg(a.tgt_off + t);
    j1 = __ldg(a.tgt_off + t + 1);
    bad = j0 < 0 || j1 < j0 || (j1 > j0 && a.exp_idx == nullptr);
    if (bad) j0 = j1 = 0;
}

__global__ void far_count_kernel(const FarArgs f)
{
    const EvalArgs& a = f.ev;
    const int64_t warp = (int64_t)blockIdx.x * (FAR_NT / 32) + (threadIdx.x >> 5);
    const int64_t t = warp * f.step * 32 + (threadIdx.x & 31);
    int64_t j0 = 0, j1 = 0;
    bool bad;
    if (t < a.n_tgt) list_of(a, t, j0, j1, bad);
    for (int64_t j = j0; __any_sync(0xffffffffu, j < j1); ++j) {
        int64_t e = -1;
        int cls = 0;
        if (j < j1) {
            e = __ldg(a.exp_idx + j);
            if (e >= 0 && e < a.n_exp) {
                double x[3];
                const int key = hi32(__double_as_longlong(offset_r2(a, t, e, x)));
                cls = key >> 19;
                if (key < 0x00100000 || key >= 0x7ff00000) e = -1;  // not a normal positive number
            } else {
                e = -1;
            }
        }
        // one atomic a warp and class where the warp shares the expansion, as most do
        int n = e >= 0 ? 1 : 0;
        const int64_t e0 = __shfl_sync(0xffffffffu, e, 0);
        if (__all_sync(0xffffffffu, e == e0)) {
            const unsigned same = __match_any_sync(0xffffffffu, cls);
            n = (threadIdx.x & 31) == __ffs(same) - 1 ? __popc(same) : 0;
        }
        if (e >= 0 && n) {
            const int64_t at = e * FAR_CLASSES + (cls & (FAR_CLASSES - 1));
            atomicAdd(f.count + at, n);
            if (cls > *(volatile int*)(f.cls + at)) atomicMax(f.cls + at, cls);
        }
    }
}

// One CTA per expansion: the scaled weights of the packed
// columns, degree by degree (a warp each), their exact products with the left
// inverse, and the common scale.
__global__ void __launch_bounds__(FAR_NT) far_prepare_kernel(const FarArgs f)
{
    const EvalArgs& a = f.ev;
    const int64_t e = blockIdx.x;
    const int J = f.J, p = a.p, np = a.np;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int2 s_g[(Q2X_P_MAX + 1) * (Q2X_P_MAX + 1)];
    __shared__ long long s_r[3][(Q2X_P_MAX + 1) * 2 * (Q2X_P_MAX + 1)];
    __shared__ int s_e[3][Q2X_P_MAX + 1];
    __shared__ double s_top[3][Q2X_P_MAX + 1];
    // rho: the lower end of the first class at or below which one in FAR_FEW of the
    // counted targets lies (a warp runs the general path for a single lane of it:
    // with one in 16, lists of 5 of 64 expansions 1,155 us against 456)
    __shared__ int s_cls;
    if (warp == 0) {
        const int n = f.count[e * FAR_CLASSES + lane], cls = f.cls[e * FAR_CLASSES + lane];
        int all = 0, upto = 0;
        for (int o = 0; o < 32; ++o) {
            const int no = __shfl_sync(0xffffffffu, n, o), co = __shfl_sync(0xffffffffu, cls, o);
            all += no;
            if (co <= cls) upto += no;
        }
        const int first = __reduce_min_sync(0xffffffffu, n > 0 && FAR_FEW * (int64_t)upto >= all ? cls : 0x7fffffff);
        if (lane == 0) s_cls = first == 0x7fffffff ? 0 : first;
    }
    __syncthreads();
    const double rr = sqrt(__longlong_as_double((long long)s_cls << 51)) * (1.0 - 1e-6);
    const double inv = rr > 0.0 ? 1.0 / rr : 0.0;
    for (int k3 = 0; k3 < f.comps; ++k3) {
        const double* F = a.coef + ((int64_t)k3 * a.n_exp + e) * np;
        for (int n = warp; n <= p; n += FAR_NT / 32) {
            double rn = 1.0;
            for (int i = 0; i < n; ++i) rn *= inv;
            double g[2] = {0.0, 0.0};
            int top = 0;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int q = lane + 32 * c;  // column n^2 + q, order m = q - n
                if (q <= 2 * n) {
                    const int m = q < n ? n - q : q - n;
                    const double len = 1.0 / __ldg(f.tab.col + (4 + 0) * 441 + n * n + q);  // sqrt((n+m)! (n-m)!)
                    double w = (m ? 2.0 : 1.0) * len * __ldg(F + n * n + q) * rn;
                    if (a.norm == 0) {
                        if ((n + m) & 1) w = -w;
                        if (q < n) w = -w;
                    } else {
                        w *= INV_4PI;  // F = (1/4pi) (-1)^(n+m) conj M
                    }
                    if (column_negative(1, n, q - n)) w = -w;
                    g[c] = w;
                    top = max(top, hi32(__double_as_longlong(w)) & 0x7fffffff);
                }
            }
            top = __reduce_max_sync(0xffffffffu, top);
            const int ex = max(top >> 20, 1);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int q = lane + 32 * c;
                if (q <= 2 * n) {
                    const long long v =
                        top < 0x7ff00000 ? dir_fixed((unsigned long long)__double_as_longlong(g[c]), ex, 56) : 0;
                    const int h = (int)((v + (1ll << 27)) >> 28);
                    s_g[n * n + q] = make_int2(h, (int)(v - ((long long)h << 28)));
                }
            }
            __syncwarp();
            float most = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int s = lane + 32 * c;
                if (s < 2 * J) {
                    long long hh = 0, mid = 1ll << 27;
                    for (int q = 0; q <= 2 * n; ++q) {
                        const int2 P = __ldg(f.tab.inv + s * np + n * n + q);
                        const int2 x = s_g[n * n + q];
                        mid = madw(P.x, x.y, mid);
                        mid = madw(P.y, x.x, mid);
                        hh = madw(P.x, x.x, hh);
                    }
                    hh += mid >> 28;
                    s_r[k3][n * 2 * J + s] = hh;
                    most = fmaxf(most, fabsf((float)hh));
                }
            }
            most = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(most)));
            if (lane == 0) {
                s_e[k3][n] = ex - 1022 - 58;
                // (a direction's two parts together)
                s_top[k3][n] = top < 0x7ff00000 ? 1.41422 * most : __longlong_as_double(0x7ff0000000000000ll);
            }
            __syncwarp();
        }
        __syncthreads();
    }
    // the common scale: sum_n (n + 1, for the derivatives) max_j |c| below 2^58,
    // so that the J directions' values add up below 2^63
    __shared__ int s_scale;
    if (threadIdx.x == 0) {
        int most = -100000;  // exponent of the largest degree's sum
        for (int k3 = 0; k3 < f.comps; ++k3)
            for (int n = 0; n <= p; ++n)
                if (s_top[k3][n] > 0.0)
                    most = max(most, s_e[k3][n] + (int)((__double_as_longlong(s_top[k3][n]) >> 52) & 0x7ff) - 1022);
        double B = 0.0;
        for (int k3 = 0; k3 < f.comps; ++k3) {
            double b = 0.0;
            for (int n = 0; n <= p; ++n)
                b += (f.comps == 3 ? n + 1.0 : 1.0) * s_top[k3][n] * pow2d(max(s_e[k3][n] - most, -1000));
            B = fmax(B, b);
        }
        // B 2^most bounds every partial sum
        int scale = 0;
        bool ok = rr > 0.0 && inv < 1e300 && B < 1e300;  // (an infinite weight takes the general path)
        if (B > 0.0) scale = 58 - (most + (int)((__double_as_longlong(B) >> 52) & 0x7ff) - 1022);
        if (scale > 1000 || scale < -1000) ok = false;
        FarMeta m;
        m.rho = ok ? rr : 0.0;
        m.scale = scale;
        for (int n = 0; n <= p; ++n) {
            double b = 0.0;
            for (int k3 = 0; k3 < f.comps; ++k3) b = fmax(b, s_top[k3][n] * pow2d(max(s_e[k3][n] - most, -1000)));
            m.bound[n] = B > 0.0 ? (float)((f.comps == 3 ? n + 1.0 : 1.0) * b / B) : 0.f;
        }
        if (!(B > 0.0)) m.bound[0] = 1.f;
        f.meta[e] = m;
        s_scale = scale;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < f.comps * J * (p + 1); i += FAR_NT) {
        const int k3 = i / (J * (p + 1)), r = i - k3 * J * (p + 1);
        const int j = r / (p + 1), n = r - j * (p + 1);
        const int sh = s_e[k3][n] + s_scale;  // c = value 2^sh
        auto put = [&](long long v) {
            if (sh >= 0) return v << min(sh, 62);
            if (sh < -62) return 0ll;
            return (v + (1ll << (-sh - 1))) >> -sh;
        };
        // Re(conj(w) v^n): the imaginary weight enters negated
        longlong2 o;
        o.x = put(s_r[k3][n * 2 * J + 2 * j]);
        o.y = -put(s_r[k3][n * 2 * J + 2 * j + 1]);
        f.c[((k3 * a.n_exp + e) * J + j) * (p + 1) + n] = o;
    }
}

// the general evaluation, out of line: few targets take it here
__device__ __noinline__ double general_potential(const double* F, int p, int norm, double x, double y, double z)
{
    return eval_one(F, p, norm, x, y, z);
}
__device__ __noinline__ void general_gradient(const double* F3, int64_t stride, int p, double x, double y, double z,
                                              double g[3][3])
{
    grad_one(F3, stride, p, x, y, z, g);
}

// y = rho x / r^2 at 2^62 and 1/r; false where the general path applies
__device__ __forceinline__ bool far_point(const FarMeta& m, int p, const double (&x)[3], double r2, long long (&y)[3],
                                          double& ir)
{
    ir = 1.0 / sqrt(r2);
    const double q = m.rho * ir, s = q * ir;  // q = |y|
    if (!(q > 0.0) || !(q < 0.99999999)) return false;
    const float qf = (float)q;
    float b = m.bound[p];
    for (int n = p - 1; n >= 0; --n) b = fmaf(b, qf, m.bound[n]);
    if (!(b > 0.0625f)) return false;
#pragma unroll
    for (int d = 0; d < 3; ++d)
        y[d] = dir_fixed((unsigned long long)__double_as_longlong(x[d] * s), 1022, 62);
    return true;
}

__global__ void __launch_bounds__(FAR_NT) far_evaluate_kernel(const FarArgs f)
{
    const EvalArgs& a = f.ev;
    __shared__ int2 dirs[6 * (Q2X_P_MAX + 1)];
    const int J = f.J, p = a.p;
    dir_load(dirs, f.tab.vec, J);
    __syncthreads();
    const int64_t t = (int64_t)blockIdx.x * FAR_NT + threadIdx.x;
    if (t >= a.n_tgt) return;
    int64_t j0, j1;
    bool bad;
    list_of(a, t, j0, j1, bad);
    if (bad) atomicOr(a.err, 8u);
    const long long rnd = f.rnd;
    double acc = 0.0;
#pragma unroll 1
    for (int64_t l = j0; l < j1; ++l) {
        const int64_t e = __ldg(a.exp_idx + l);
        if (e < 0 || e >= a.n_exp) {
            atomicOr(a.err, 1u);
            continue;
        }
        double x[3];
        const double r2 = offset_r2(a, t, e, x);
        if (!(r2 > 0.0)) continue;  // at the centre the series does not apply
        const FarMeta& m = f.meta[e];
        long long y[3];
        double ir;
        if (!far_point(m, p, x, r2, y, ir)) {
            acc += general_potential(a.coef + e * (int64_t)a.np, p, a.norm, x[0], x[1], x[2]);
            continue;
        }
        const longlong2* c = f.c + e * J * (p + 1) + p;
        long long sum = 0;
#pragma unroll 1
        for (int j = 0; j < J; ++j, c += p + 1) {
            Fx da[6];
            dir_of(dirs, j, da);
            const Mul v = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
            longlong2 w = __ldg(c);
            Cx b{w.x, w.y};
            CxH h = high_of(b);
            if (p > 0) {
                const longlong2* q = c - 1;
#pragma unroll 4
                for (int n = p - 1; n > 0; --n, --q) {
                    w = __ldg(q);
                    b = mul_add<true>(v, b, h, Cx{w.x, w.y}, rnd);
                    h = high_of(b);
                }
                // the constant term: its real part alone
                b.re = mul2<true>(v.rh, v.rl, v.nh, v.nl, (int)b.re, h.rh, (int)b.im, h.ih, __ldg(q).x, rnd);
            }
            sum += b.re;
        }
        acc += (double)sum * pow2d(-m.scale) * ir;
    }
    a.out[t] = a.accumulate ? a.out[t] + acc : acc;
}

// H = curl A: values and derivatives of the three components' polynomials.
// With A = (1/r) L(y), y = rho x / r^2 and D = grad L (in y):
//   grad A = (rho D / r^2 - x (L + 2 y.D) / r^2) / r.
__global__ void __launch_bounds__(FAR_NT) far_curl_kernel(const FarArgs f)
{
    const EvalArgs& a = f.ev;
    __shared__ int2 dirs[6 * (Q2X_P_MAX + 1)];
    const int J = f.J, p = a.p;
    dir_load(dirs, f.tab.vec, J);
    __syncthreads();
    const int64_t t = (int64_t)blockIdx.x * FAR_NT + threadIdx.x;
    if (t >= a.n_tgt) return;
    int64_t j0, j1;
    bool bad;
    list_of(a, t, j0, j1, bad);
    if (bad) atomicOr(a.err, 8u);
    const long long rnd = f.rnd;
    double H[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
    for (int64_t l = j0; l < j1; ++l) {
        const int64_t e = __ldg(a.exp_idx + l);
        if (e < 0 || e >= a.n_exp) {
            atomicOr(a.err, 1u);
            continue;
        }
        double x[3];
        const double r2 = offset_r2(a, t, e, x);
        if (!(r2 > 0.0)) continue;
        const FarMeta& m = f.meta[e];
        long long y[3];
        double ir;
        double g[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};  // g[k][d] = d A_k / d x_d
        if (!far_point(m, p, x, r2, y, ir)) {
            general_gradient(a.coef + e * (int64_t)a.np, a.n_exp * (int64_t)a.np, p, x[0], x[1], x[2], g);
        } else {
            const double unit = pow2d(-m.scale), s = m.rho * ir * ir;
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
                const longlong2* c = f.c + (k * a.n_exp + e) * J * (p + 1) + p;
                long long val = 0, der[3] = {0, 0, 0};
#pragma unroll 1
                for (int j = 0; j < J; ++j, c += p + 1) {
                    Fx da[6];
                    dir_of(dirs, j, da);
                    const Mul v = mul_of(dir_dot(da, y, rnd), dir_dot(da + 3, y, rnd));
                    longlong2 w = __ldg(c);
                    // b: the polynomial, d: its derivative
                    Cx b{w.x, w.y}, d{0, 0};
                    CxH hb = high_of(b), hd = high_of(d);
                    const longlong2* q = c - 1;
#pragma unroll 2
                    for (int n = p - 1; n >= 0; --n, --q) {
                        w = __ldg(q);
                        d = mul_add<true>(v, d, hd, b, rnd);
                        hd = high_of(d);
                        b = mul_add<true>(v, b, hb, Cx{w.x, w.y}, rnd);
                        hb = high_of(b);
                    }
                    val += b.re;
#pragma unroll
                    for (int i = 0; i < 3; ++i)  // Re(a_i d)
                        der[i] += mul2<false>(da[i].h, da[i].l, -da[3 + i].h, -da[3 + i].l, (int)d.re, hd.rh, (int)d.im,
                                              hd.ih, 0, rnd);
                }
                const double L = (double)val * unit;
                double D[3], dot = 0.0;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    D[i] = (double)der[i] * unit;
                    dot += D[i] * (x[i] * s);
                }
                const double w = (L + 2.0 * dot) * ir * ir;
#pragma unroll
                for (int i = 0; i < 3; ++i) g[k][i] = (s * D[i] - x[i] * w) * ir;
            }
        }
        H[0] += g[2][1] - g[1][2];
        H[1] += g[0][2] - g[2][0];
        H[2] += g[1][0] - g[0][1];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double* o = a.out + d * a.n_tgt + t;
        *o = a.accumulate ? *o + H[d] : H[d];
    }
}

size_t up(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

size_t far_workspace(int p, int comps, int64_t n_exp)
{
    return 2 * up(sizeof(int) * FAR_CLASSES * (size_t)n_exp) + up(sizeof(FarMeta) * (size_t)n_exp) +
           up(sizeof(longlong2) * (size_t)n_exp * comps * (p + 1) * (p + 1));
}

cudaError_t far_run(const EvalArgs& ev, int comps, void* ws, cudaStream_t st)
{
    FarArgs f;
    f.ev = ev;
    cudaError_t e = dir_tables(ev.p, &f.tab);
    if (e != cudaSuccess) return e;
    f.J = ev.p + 1;
    f.comps = comps;
    f.rnd = 1ll << 31;
    unsigned char* w = static_cast<unsigned char*>(ws);
    f.count = reinterpret_cast<int*>(w);
    w += up(sizeof(int) * FAR_CLASSES * (size_t)ev.n_exp);
    f.cls = reinterpret_cast<int*>(w);
    w += up(sizeof(int) * FAR_CLASSES * (size_t)ev.n_exp);
    f.meta = reinterpret_cast<FarMeta*>(w);
    w += up(sizeof(FarMeta) * (size_t)ev.n_exp);
    f.c = reinterpret_cast<longlong2*>(w);
    e = cudaMemsetAsync(f.count, 0, 2 * up(sizeof(int) * FAR_CLASSES * (size_t)ev.n_exp), st);  // (and the classes)
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((ev.n_tgt + FAR_NT - 1) / FAR_NT);
    f.step = std::max<int64_t>(1, ev.n_tgt / (ev.n_exp * FAR_SAMPLE));
    const int64_t warps = ((ev.n_tgt + 31) / 32 + f.step - 1) / f.step, per = FAR_NT / 32;
    far_count_kernel<<<(unsigned)((warps + per - 1) / per), FAR_NT, 0, st>>>(f);
    far_prepare_kernel<<<(unsigned)ev.n_exp, FAR_NT, 0, st>>>(f);
    if (comps == 1)
        far_evaluate_kernel<<<grid, FAR_NT, 0, st>>>(f);
    else
        far_curl_kernel<<<grid, FAR_NT, 0, st>>>(f);
    return cudaGetLastError();
}

}  // namespace q2x
