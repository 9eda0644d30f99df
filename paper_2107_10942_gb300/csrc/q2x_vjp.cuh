// q2x_vjp.cuh -- adjoint of the triangle single-layer Q2X (constant density):
// given G = d loss / d coef (one row per leaf), accumulate d loss / d vertex
// coordinates and d loss / d density.
//
// With F_c = sigma J U_c(x1, x2, x3) the packed coefficients of one triangle
// (Eq. (bas10)), loss = sum_c G_c F_c, lambda_k the barycentric coordinate of
// vertex k and y = sum_k lambda_k x_k:
//   d loss / d x_k     = sigma [ (dJ/dx_k) sum_c G_c U_c + J sum_c G_c dU_c/dx_k ]
//   dU_c / dx_k        = (1/4pi)(-1)^n int_T lambda_k grad R_n^{-m}(y - r*) du dv
//   d loss / d sigma   = J sum_c G_c U_c
// The e_d component of int lambda_k grad R is a double-layer moment with unit
// "normal" e_d and linear density lambda_k (Eq. (bas8), Eq. (rec15)), so it is
// the stencil A_{e_d} applied to the lambda_k-weighted face row Iw^(k) of the
// linear-density chain one degree lower:
//   e_x: (b - a)/2 (m > 0), Re b (m = 0);  e_y: -(i/2)(a + b) (m > 0), Im b (m = 0);
//   e_z: -c  (a = x^{m-1}, b = x^{m+1}, c = x^m of that row).
// The chain carries q, j, i and, for k = 2, 3, E^(k) and Iw^(k) (sources
// (n+1) q and j); Iw^(1) = (n+3) i - Iw^(2) - Iw^(3) because sum_k lambda_k = 1.
// In the scaled frame y' = (y - r*)/rho, rho = 2^s: U_c = rho^n U'_c,
// dU_c/dx = rho^{n-1} dU'_c/dy', J = rho^2 J', so with G'_c = G_c rho^{n+1}
//   d loss / d x_k = sigma [ (dJ'/dy'_k) S_U + J' S_V,k ],  d loss / d sigma = rho J' S_U,
// S_U = sum_c G'_c U'_c, S_V,k = sum_c G'_c dU'_c/dy'_k.  q2x_vjp_weights folds
// rho^{n+1}, 1/(n+2)!, 1/4pi and the packing sign of each column into one
// weight per leaf and column.
#pragma once

#include <type_traits>

#include "q2x_kernels.cuh"

namespace q2x {

struct VjpArgs {
    int64_t n_elem, n_vert;
    const double* vx;
    const double* vy;
    const double* vz;
    const int32_t* idx;
    const double* sigma;
    int64_t n_leaves;
    const int64_t* leaf_off;  // NULL: per-element
    const double* leaf_c;
    const double* leaf_rho;
    const int32_t* leaf_p;
    int p_max, np_max, norm;
    const void* w;            // [n_leaves][np_max] weights (T)
    double* grad_v;           // SoA 3 x n_vert, accumulated
    double* grad_sigma;       // n_elem or NULL, overwritten
    unsigned* err;
};

// weight of column c of leaf L: G_c * rho^{n+1} * sign(c) / (n+2)! (/ 4pi for
// COEFF); half of it for the FP32 kernel
template <typename T>
__global__ void q2x_vjp_weights(const double* __restrict__ G, const double* __restrict__ leaf_rho,
                                const int32_t* __restrict__ leaf_p, int64_t n_leaves, int np, int p_max,
                                int norm, T* __restrict__ w)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_leaves * np) return;
    const int64_t L = i / np;
    const int c = (int)(i - L * np);
    int n, m;
    col_nm(c, n, m);
    const int pL = leaf_p ? leaf_p[L] : p_max;
    const int s = leaf_rho ? scale_exponent(leaf_rho[L]) : 0;
    double v = 0.0;
    if (n <= pL && pL <= p_max) {
        v = G[i] * c_inv_fact_d[n + 2] * pow2d(s * (n + 1));
        if (norm == 0) v *= INV_4PI;
        if (column_negative(norm, n, m)) v = -v;
    }
    w[i] = sizeof(T) == 4 ? T(0.5) * (T)v : (T)v;
}

// d loss / d x_k from the sums (FP64 accumulation) and d loss / d sigma
template <typename T>
__device__ __forceinline__ void vjp_scatter(const VjpArgs& a, int64_t e, int sexp, const Frame<T, 3>& F, T SU,
                                            const T (&SV)[3][3])
{
    const T sig = F.s1;
    const T eu[3] = {F.eu[0], F.eu[1], F.eu[2]};
    const T ev[3] = {F.ev[0], F.ev[1], F.ev[2]};
    const T J = F.J;
    const T nh[3] = {T(2) * F.XN, T(2) * F.YN, F.ZN};
    // dJ/dx2 = ev x n, dJ/dx3 = n x eu, dJ/dx1 = -(both)
    T dJ[3][3];
    dJ[1][0] = ev[1] * nh[2] - ev[2] * nh[1];
    dJ[1][1] = ev[2] * nh[0] - ev[0] * nh[2];
    dJ[1][2] = ev[0] * nh[1] - ev[1] * nh[0];
    dJ[2][0] = nh[1] * eu[2] - nh[2] * eu[1];
    dJ[2][1] = nh[2] * eu[0] - nh[0] * eu[2];
    dJ[2][2] = nh[0] * eu[1] - nh[1] * eu[0];
#pragma unroll
    for (int d = 0; d < 3; ++d) dJ[0][d] = -(dJ[1][d] + dJ[2][d]);

    double* gv[3] = {a.grad_v, a.grad_v + a.n_vert, a.grad_v + 2 * a.n_vert};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int64_t v = __ldg(a.idx + (int64_t)k * a.n_elem + e);
        if (v < 0 || v >= a.n_vert) continue;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double g = (double)sig * ((double)dJ[k][d] * (double)SU + (double)J * (double)SV[k][d]);
            atomicAdd(gv[d] + v, g);
        }
    }
    if (a.grad_sigma) a.grad_sigma[e] = pow2d(sexp) * (double)J * (double)SU;
}

template <typename T, int P>
__global__ void __launch_bounds__(128, 2) q2x_tri_vjp_kernel(const VjpArgs a)
{
    constexpr int NL = 7;  // q, j, i, E2, Iw2, E3, Iw3
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.n_elem) return;
    int64_t L = e;
    if (a.leaf_off) L = leaf_search(a.leaf_off, 0, a.n_leaves - 1, e);
    int pL = a.leaf_p ? __ldg(a.leaf_p + L) : a.p_max;
    unsigned errbits = 0;
    if (pL < 0 || pL > a.p_max) {
        errbits |= 4u;
        pL = -1;
    }
    const double cx = __ldg(a.leaf_c + L), cy = __ldg(a.leaf_c + a.n_leaves + L),
                 cz = __ldg(a.leaf_c + 2 * a.n_leaves + L);
    const int sexp = a.leaf_rho ? scale_exponent(__ldg(a.leaf_rho + L)) : 0;
    Frame<T, 3> F;
    load_frame<T, KIND_TRI, DENS_CONST>(a.vx, a.vy, a.vz, a.idx, a.sigma, a.n_elem, a.n_vert, e, true, cx, cy, cz,
                                        sexp, errbits, pL, F);
    if (errbits) atomicOr(a.err, errbits);
    if (pL < 0) {
        if (a.grad_sigma) a.grad_sigma[e] = 0.0;
        return;
    }
    // local vertex coordinates back from the stencil coefficients (x1: level i,
    // x2: level q, x3: level j); edges and the Jacobian from the frame (formed
    // from the exact splits of the FP64 inputs)
    const T x1[3] = {T(2) * F.LX[2], T(2) * F.LY[2], F.LZ[2]};
    const T x2[3] = {T(2) * F.LX[0], T(2) * F.LY[0], F.LZ[0]};
    const T x3[3] = {T(2) * F.LX[1], T(2) * F.LY[1], F.LZ[1]};
    const T* w = reinterpret_cast<const T*>(a.w) + L * (int64_t)a.np_max;
    // stencil vertex of each level
    const int vtx[NL] = {1, 2, 0, 2, 0, 2, 0};
    T LX[NL], LY[NL], LZ[NL];
    const T* xs[3] = {x1, x2, x3};
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        LX[k] = T(0.5) * xs[vtx[k]][0];
        LY[k] = T(0.5) * xs[vtx[k]][1];
        LZ[k] = xs[vtx[k]][2];
    }
    T Rr[NL][P + 2], Ri[NL][P + 2];
#pragma unroll
    for (int k = 0; k < NL; ++k)
#pragma unroll
        for (int m = 0; m <= P + 1; ++m) Rr[k][m] = Ri[k][m] = T(0);
    T SU = T(0), SV[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) SV[k][0] = SV[k][1] = SV[k][2] = T(0);

#pragma unroll 1
    for (int n = 0; n <= pL; ++n) {
        const T c2 = T(n + 1);
        const T c3 = T(n + 3);
        const T* wn = w + n * n + n;        // weights of degree n, column (n, 0)
        const T* wn1 = w + (n + 1) * (n + 1) + (n + 1);  // degree n + 1
        const bool grad_next = (n + 1 <= pL);
        T pr[NL], pi[NL];
#pragma unroll
        for (int k = 0; k < NL; ++k) pr[k] = pi[k] = T(0);
#pragma unroll
        for (int m = 0; m <= P; ++m) {
            if (m <= n) {
                T nr[NL], ni[NL];
#pragma unroll
                for (int k = 0; k < NL; ++k) {
                    const T cr = Rr[k][m], ci = Ri[k][m];
                    const T br = Rr[k][m + 1], bi = Ri[k][m + 1];
                    T sr, si;
                    if (k == 0) {
                        sr = (n == 0 && m == 0) ? T(1) : T(0);
                        si = T(0);
                    } else if (k == 1 || k == 2) {
                        sr = nr[k - 1];  // j <- q, i <- j
                        si = ni[k - 1];
                    } else if (k == 3) {
                        sr = c2 * nr[0];  // E2 <- (n+1) q
                        si = c2 * ni[0];
                    } else if (k == 5) {
                        sr = nr[1];  // E3 <- j
                        si = ni[1];
                    } else {
                        sr = nr[k - 1];  // Iw2 <- E2, Iw3 <- E3
                        si = ni[k - 1];
                    }
                    T vr, vi;
                    if (m == 0) {
                        vr = fma(T(2) * LX[k], br, sr);
                        vr = fma(T(2) * LY[k], bi, vr);
                        vr = fma(-LZ[k], cr, vr);
                        vi = T(0);
                    } else {
                        vr = fma(LX[k], br - pr[k], sr);
                        vr = fma(LY[k], bi + pi[k], vr);
                        vr = fma(-LZ[k], cr, vr);
                        vi = fma(LX[k], bi - pi[k], si);
                        vi = fma(-LY[k], br + pr[k], vi);
                        vi = fma(-LZ[k], ci, vi);
                    }
                    nr[k] = vr;
                    ni[k] = vi;
                    pr[k] = cr;
                    pi[k] = ci;
                    Rr[k][m] = vr;
                    Ri[k][m] = vi;
                }
                // S_U: forward moment i^ of (n, m)
                {
                    const T re_c = (m & 1) ? ni[2] : nr[2];
                    const T im_c = (m & 1) ? nr[2] : ni[2];
                    SU = fma(__ldg(wn + m), re_c, SU);
                    if (m > 0) SU = fma(__ldg(wn - m), im_c, SU);
                }
            }
        }
        // S_V: degree n + 1 from the rows Iw^(k)_n (now in Rr/Ri), m = 0..n+1
        if (grad_next) {
#pragma unroll
            for (int m = 0; m <= P + 1; ++m) {
                if (m <= n + 1) {
                    const T wre = __ldg(wn1 + m);
                    const T wim = (m > 0) ? __ldg(wn1 - m) : T(0);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        // row of Iw^(k): k = 1 derived, k = 2 level 4, k = 3 level 6
                        auto row = [&](int mm, T& r, T& i_) {
                            if (mm < 0 || mm > n) {
                                r = i_ = T(0);
                                return;
                            }
                            if (k == 0) {
                                r = c3 * Rr[2][mm] - Rr[4][mm] - Rr[6][mm];
                                i_ = c3 * Ri[2][mm] - Ri[4][mm] - Ri[6][mm];
                            } else {
                                const int lv = (k == 1) ? 4 : 6;
                                r = Rr[lv][mm];
                                i_ = Ri[lv][mm];
                            }
                        };
                        T ar, ai, br, bi, cr, ci;
                        row(m - 1, ar, ai);
                        row(m + 1, br, bi);
                        row(m, cr, ci);
                        T gx_r, gx_i, gy_r, gy_i, gz_r, gz_i;
                        if (m == 0) {
                            gx_r = br;
                            gy_r = bi;
                            gz_r = -cr;
                            gx_i = gy_i = gz_i = T(0);
                        } else {
                            gx_r = T(0.5) * (br - ar);
                            gx_i = T(0.5) * (bi - ai);
                            gy_r = T(0.5) * (bi + ai);
                            gy_i = T(-0.5) * (br + ar);
                            gz_r = -cr;
                            gz_i = -ci;
                        }
                        const T gr[3] = {gx_r, gy_r, gz_r};
                        const T gi[3] = {gx_i, gy_i, gz_i};
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const T re_c = (m & 1) ? gi[d] : gr[d];
                            const T im_c = (m & 1) ? gr[d] : gi[d];
                            SV[k][d] = fma(wre, re_c, SV[k][d]);
                            if (m > 0) SV[k][d] = fma(wim, im_c, SV[k][d]);
                        }
                    }
                }
            }
        }
    }
    vjp_scatter<T>(a, e, sexp, F, SU, SV);
}

// -------------------------------------------------------------- FP32 kernel
// The same recurrences and sums, operation for operation (the results are the
// same bits), in fewer instructions: the scalar form spent 195 per (n, m) and
// warp, 35 of them moves and 30 branches and their bookkeeping.
//  * Paired FP32: q, j and i as (re, im); E^(2), E^(3) have one stencil vertex
//    (x3) and Iw^(2), Iw^(3) the other (x1), so these are pairs over the level,
//    real and imaginary parts apart.
//  * The degree is the warp's, so its branches are uniform; lanes of smaller
//    degree (leaves meet in a warp) go on with rows of zeros.
//  * Factors 1/2 and signs of the gradient stencil are powers of two in the
//    weights (halved) and in the sums (z holds -1/2 of its sum, S_U 1/2).
//  * The leaf of an element: the warp finds its first and last element's leaf
//    in steps of 32, then each lane searches between them.
//  * At P = 12 a new entry m is written over the old entry m - 1 on the way up,
//    over m + 1 on the way down, both dead by then, and degrees alternate: no
//    moves, twice the code.  1.00 M triangles at p = 12: 736 us so, 783 with
//    one direction and moves, 947 in the scalar form.  Larger P spill, and
//    smaller ones are short enough: there the code's size costs more (forward
//    and adjoint, 0.8 M triangles at p = 16: 1,835 us scalar, 1,328 alternating,
//    1,308 in one direction; 0.2 M at p = 20: 969, 641, 626).
// Bound by the latency of 2 warps a scheduler (255 registers): a third of the
// slots issue.  Not kept: the rows E and Iw in shared memory and three CTAs an
// SM (777 us: the moves come back, and the instruction cache misses double);
// three and four CTAs an SM at P = 8 and 4 (spills: 285 -> 292 us, 265 -> 275).
__device__ __forceinline__ cf cf_dup(float x) { return cf_make(x, x); }

__device__ __forceinline__ int64_t leaf_search_warp(const int64_t* __restrict__ off, int64_t n_leaves, int64_t e,
                                                    int lane)
{
    int64_t lo = 0, hi = n_leaves - 1;  // the last L with off[L] <= e, e the warp's
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step;
        const unsigned le = __ballot_sync(0xffffffffu, at <= hi && __ldg(off + min(at, hi)) <= e);
        // offsets ascend: the first k probes lie at or below e
        const int k = __ffs(~le) ? __ffs(~le) - 1 : 32;
        lo += k * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

template <int P>
__global__ void __launch_bounds__(128, 2) q2x_tri_vjp_f32_kernel(const VjpArgs a)
{
    constexpr bool ALT = P == 12;  // rows updated without moves, alternately upwards and downwards
    constexpr int S = P + 2;       // slots of a row
    const int lane = threadIdx.x & 31;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e - lane >= a.n_elem) return;  // warp-uniform
    const bool active = e < a.n_elem;
    int64_t L = active ? e : a.n_elem - 1;
    if (a.leaf_off) {
        const int64_t first = leaf_search_warp(a.leaf_off, a.n_leaves, e - lane, lane);
        const int64_t last = leaf_search_warp(a.leaf_off, a.n_leaves, min(e - lane + 31, a.n_elem - 1), lane);
        L = leaf_search(a.leaf_off, first, last, L);
    }
    int pL = a.leaf_p ? __ldg(a.leaf_p + L) : a.p_max;
    unsigned errbits = 0;
    if (pL < 0 || pL > a.p_max) {
        if (active) errbits |= 4u;
        pL = -1;
    }
    const double cx = __ldg(a.leaf_c + L), cy = __ldg(a.leaf_c + a.n_leaves + L),
                 cz = __ldg(a.leaf_c + 2 * a.n_leaves + L);
    const int sexp = a.leaf_rho ? scale_exponent(__ldg(a.leaf_rho + L)) : 0;
    Frame<float, 3> F;
    load_frame<float, KIND_TRI, DENS_CONST>(a.vx, a.vy, a.vz, a.idx, a.sigma, a.n_elem, a.n_vert, e, active, cx, cy,
                                            cz, sexp, errbits, pL, F);
    if (errbits) atomicOr(a.err, errbits);
    if (!active) pL = -1;
    const bool on = pL >= 0;
    // stencils of x2 (q), x3 (j, E) and x1 (i, Iw)
    const float qy = on ? F.LY[0] : 0.0f, jy = on ? F.LY[1] : 0.0f, iy = on ? F.LY[2] : 0.0f;
    const cf qx2 = cf_dup(on ? F.LX[0] : 0.0f), qz2 = cf_dup(on ? -F.LZ[0] : 0.0f);
    const cf jx2 = cf_dup(on ? F.LX[1] : 0.0f), jz2 = cf_dup(on ? -F.LZ[1] : 0.0f), jy2 = cf_dup(jy);
    const cf ix2 = cf_dup(on ? F.LX[2] : 0.0f), iz2 = cf_dup(on ? -F.LZ[2] : 0.0f), iy2 = cf_dup(iy);
    const int n_max = __reduce_max_sync(0xffffffffu, pL);
    const bool mixed = __any_sync(0xffffffffu, pL != n_max);
    const float* w = reinterpret_cast<const float*>(a.w) + L * (int64_t)a.np_max;

    // rows: q, j, i as (re, im); E and Iw as (level 2, level 3), re and im
    cf Q[S], R[S], I[S], Er[S], Ei[S], Wr[S], Wi[S];
    const auto clear = [&]() {
#pragma unroll
        for (int m = 0; m < S; ++m) Q[m] = R[m] = I[m] = Er[m] = Ei[m] = Wr[m] = Wi[m] = cf_zero();
    };
    clear();
    float SU = 0.0f, S1[3] = {0.0f, 0.0f, 0.0f};  // S1: k = 1
    cf S23[3] = {cf_zero(), cf_zero(), cf_zero()};  // k = 2, 3

    // degree n from n - 1.  ALT, up: entry m lies in slot m + 1 before, m after;
    // down: in slot m before, m + 1 after.  Else in slot m
    const auto pass = [&](auto up_c, int n) {
        constexpr bool up = decltype(up_c)::value;
        const float c2 = (float)(n + 1);
        const float seed = (n == 0 && on) ? 1.0f : 0.0f;
        cf pQ = cf_zero(), pR = pQ, pI = pQ, pEr = pQ, pEi = pQ, pWr = pQ, pWi = pQ;
#pragma unroll
        for (int t = 0; t <= P; ++t) {
            const int m = up ? t : P - t;
            if (m <= n) {
                const int ic = ALT && up ? m + 1 : m, ib = ic + 1, ip = ic - 1;
                const int io = ALT && !up ? m + 1 : m;
                const auto at = [&](const cf* x, int k) { return k < S ? x[k] : cf_zero(); };
                const auto one = [&](cf* x, cf& prev, cf src, cf x2, float y, cf z2) {
                    const cf c = x[ic], b = at(x, ib);
                    float br, bi, sr, si, vr, vi, cr, ci;
                    cf_parts(b, br, bi);
                    cf v;
                    if (m == 0) {
                        float xr, zr, t_;
                        cf_parts(x2, xr, t_);
                        cf_parts(z2, zr, t_);
                        cf_parts(src, sr, si);
                        cf_parts(c, cr, ci);
                        vr = fma(2.0f * xr, br, sr);
                        vr = fma(2.0f * y, bi, vr);
                        vr = fma(zr, cr, vr);
                        v = cf_make(vr, 0.0f);
                    } else {
                        const cf p = ALT ? x[ip] : prev;
                        float pr, pi;
                        cf_parts(p, pr, pi);
                        v = cf_fma(x2, cf_sub(b, p), src);
                        cf_parts(v, vr, vi);
                        vr = fma(y, bi + pi, vr);
                        vi = fma(-y, br + pr, vi);
                        v = cf_fma(z2, c, cf_make(vr, vi));
                    }
                    prev = c;
                    x[io] = v;
                    return v;
                };
                const auto two = [&](cf* xr, cf* xi, cf& qr_, cf& qi_, cf sr, cf si, cf x2, float y, cf y2, cf z2) {
                    const cf cr = xr[ic], ci = xi[ic], br = at(xr, ib), bi = at(xi, ib);
                    cf vr, vi;
                    if (m == 0) {
                        float t0, t1;
                        cf_parts(x2, t0, t1);
                        vr = cf_fma(cf_dup(2.0f * t0), br, sr);
                        vr = cf_fma(cf_dup(2.0f * y), bi, vr);
                        vr = cf_fma(z2, cr, vr);
                        vi = cf_zero();
                    } else {
                        const cf pr = ALT ? xr[ip] : qr_, pi = ALT ? xi[ip] : qi_;
                        vr = cf_fma(x2, cf_sub(br, pr), sr);
                        vr = cf_fma(y2, cf_add(bi, pi), vr);
                        vr = cf_fma(z2, cr, vr);
                        vi = cf_fma(x2, cf_sub(bi, pi), si);
                        float s0, s1, v0, v1;
                        cf_parts(cf_add(br, pr), s0, s1);
                        cf_parts(vi, v0, v1);
                        vi = cf_make(fma(-y, s0, v0), fma(-y, s1, v1));
                        vi = cf_fma(z2, ci, vi);
                    }
                    qr_ = cr;
                    qi_ = ci;
                    xr[io] = vr;
                    xi[io] = vi;
                };
                const cf vq = one(Q, pQ, cf_make(m == 0 ? seed : 0.0f, 0.0f), qx2, qy, qz2);
                const cf vj = one(R, pR, vq, jx2, jy, jz2);
                one(I, pI, vj, ix2, iy, iz2);
                float qr, qi, jr, ji;
                cf_parts(vq, qr, qi);
                cf_parts(vj, jr, ji);
                two(Er, Ei, pEr, pEi, cf_make(c2 * qr, jr), cf_make(c2 * qi, ji), jx2, jy, jy2, jz2);
                two(Wr, Wi, pWr, pWi, Er[io], Ei[io], ix2, iy, iy2, iz2);
            }
        }
    };
    // S_U of degree n and S_V of degree n + 1; entry m in slot m + off
    const auto sums = [&](auto off_c, int n) {
        constexpr int off = decltype(off_c)::value;
        const float* wn = w + n * n + n;                  // weights of degree n, column (n, 0)
        const float* wn1 = w + (n + 1) * (n + 1) + n + 1;  // degree n + 1
        const float c3 = (float)(n + 3);
        // the next order's weights are loaded a step ahead: nothing else hides
        // their latency, with two warps a scheduler
        float h = __ldg(wn), g = 0.0f, hn = 0.0f, gn = 0.0f;
#pragma unroll
        for (int m = 0; m <= P; ++m) {
            if (m <= n) {
                if (m + 1 <= n) {
                    hn = __ldg(wn + m + 1);
                    gn = __ldg(wn - m - 1);
                }
                float re, im;
                cf_parts(I[m + off], re, im);
                SU = fma(h, (m & 1) ? im : re, SU);
                if (m > 0) SU = fma(g, (m & 1) ? re : im, SU);
                h = hn;
                g = gn;
            }
        }
        if (n + 1 > n_max) return;
        const auto at = [&](const cf* x, int m) { return m + off < S ? x[m + off] : cf_zero(); };
        // row of Iw^(1): (n + 3) i - Iw^(2) - Iw^(3)
        const auto row1 = [&](int m, float& r, float& i_) {
            float ir, ii, r2, r3, i2, i3;
            cf_parts(at(I, m), ir, ii);
            cf_parts(at(Wr, m), r2, r3);
            cf_parts(at(Wi, m), i2, i3);
            r = c3 * ir - r2 - r3;
            i_ = c3 * ii - i2 - i3;
        };
        float ar = 0.0f, ai = 0.0f, cr, ci, br, bi;
        row1(0, cr, ci);
        h = __ldg(wn1);
#pragma unroll
        for (int m = 0; m <= P; ++m) {
            if (m <= n + 1) {
                if (m + 1 <= n + 1) {
                    hn = __ldg(wn1 + m + 1);
                    gn = __ldg(wn1 - m - 1);
                }
                row1(m + 1, br, bi);
                const cf Br = at(Wr, m + 1), Bi = at(Wi, m + 1), Cr = at(Wr, m), Ci = at(Wi, m);
                if (m == 0) {
                    const float w0 = 2.0f * h;
                    S1[0] = fma(w0, br, S1[0]);
                    S1[1] = fma(w0, bi, S1[1]);
                    S1[2] = fma(h, cr, S1[2]);
                    S23[0] = cf_fma(cf_dup(w0), Br, S23[0]);
                    S23[1] = cf_fma(cf_dup(w0), Bi, S23[1]);
                    S23[2] = cf_fma(cf_dup(h), Cr, S23[2]);
                } else {
                    const cf h2 = cf_dup(h), g2 = cf_dup(g);
                    const cf Ar = at(Wr, m - 1), Ai = at(Wi, m - 1);
                    // x: (b - a) / 2; y: -(i/2)(a + b); z: -c; the weights are
                    // halved, z takes c (twice what it should, negated)
                    float s0, s1, y0, y1;
                    cf_parts(cf_add(Br, Ar), s0, s1);
                    if (m & 1) {
                        S1[0] = fma(g, br - ar, fma(h, bi - ai, S1[0]));
                        S1[1] = fma(g, bi + ai, fma(-h, br + ar, S1[1]));
                        S1[2] = fma(g, cr, fma(h, ci, S1[2]));
                        S23[0] = cf_fma(g2, cf_sub(Br, Ar), cf_fma(h2, cf_sub(Bi, Ai), S23[0]));
                        cf_parts(S23[1], y0, y1);
                        S23[1] = cf_fma(g2, cf_add(Bi, Ai), cf_make(fma(-h, s0, y0), fma(-h, s1, y1)));
                        S23[2] = cf_fma(g2, Cr, cf_fma(h2, Ci, S23[2]));
                    } else {
                        S1[0] = fma(g, bi - ai, fma(h, br - ar, S1[0]));
                        S1[1] = fma(-g, br + ar, fma(h, bi + ai, S1[1]));
                        S1[2] = fma(g, ci, fma(h, cr, S1[2]));
                        S23[0] = cf_fma(g2, cf_sub(Bi, Ai), cf_fma(h2, cf_sub(Br, Ar), S23[0]));
                        cf_parts(cf_fma(h2, cf_add(Bi, Ai), S23[1]), y0, y1);
                        S23[1] = cf_make(fma(-g, s0, y0), fma(-g, s1, y1));
                        S23[2] = cf_fma(g2, Ci, cf_fma(h2, Cr, S23[2]));
                    }
                }
                ar = cr;
                ai = ci;
                cr = br;
                ci = bi;
                h = hn;
                g = gn;
            }
        }
    };
#pragma unroll 1
    for (int n = 0; n <= n_max; n += ALT ? 2 : 1) {
        if (mixed && n == pL + 1) clear();
        pass(std::true_type{}, n);
        sums(std::integral_constant<int, 0>{}, n);
        if (!ALT) continue;
        if (n + 1 > n_max) break;
        if (mixed && n == pL) clear();
        pass(std::false_type{}, n + 1);
        sums(std::integral_constant<int, 1>{}, n + 1);
    }
    if (!active) return;
    if (pL < 0) {
        if (a.grad_sigma) a.grad_sigma[e] = 0.0;
        return;
    }
    // the sums at their scale
    float SV[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float f = d == 2 ? -2.0f : 1.0f;
        float s2, s3;
        cf_parts(S23[d], s2, s3);
        SV[0][d] = f * S1[d];
        SV[1][d] = f * s2;
        SV[2][d] = f * s3;
    }
    vjp_scatter<float>(a, e, sexp, F, 2.0f * SU, SV);
}

}  // namespace q2x
