// q2x_evaluate.cu -- far-field evaluation of expansions at target points
// (the M2P step that consumes the Q2X / M2M coefficients).
//
// Eq. (bas3) expands the Green's function in S_n^m about r*, so a box whose
// coefficients are F_n^m (Eq. (bas4), COEFF norm) has the potential
//   phi(x) = sum_{n<=p} sum_{|m|<=n} F_n^m S_n^m(x - r*)
//          = sum_n [F_n^0 S_n^0 + 2 Re sum_{m>0} F_n^m S_n^m]   (Eq. (bas2.1)),
// and raw moments M_n^m (MOMENT norm) give phi = (1/4pi) sum (-1)^n M_n^{-m} S_n^m.
// S_n^m = i^{-m} (n-m)! r^{-2n-1} T_n^m for m >= 0 (Eq. (bas1)) with
// T_n^m = r^n P_n^m(cos theta) e^{i m phi}, the solid harmonic polynomial built
// by the associated-Legendre recurrences in Cartesian form:
//   T_m^m = (-1)^m (2m-1)!! (x + iy)^m,  T_{m+1}^m = (2m+1) z T_m^m,
//   (n - m) T_n^m = (2n-1) z T_{n-1}^m - (n+m-1) r^2 T_{n-2}^m.
// Since T_n^m = P_n T_m^m with a real sequence P_n, each order's column is
// summed as Re(i^{-m} T_m^m sum_n F_n^m U_n) with U_n = (n-m)! r^{-2n-1} P_n
// from a division-free real recurrence (see eval_one).  One thread per
// target, looping over the target's expansion list (CSR).  FP64.
#include <cuda_runtime.h>

#include <cstdint>

#include "q2x.h"
#include "q2x_farfield.h"
#include "q2x_plan.h"

namespace q2x {

__global__ void q2x_evaluate_kernel(const EvalArgs a)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n_tgt) return;
    int64_t j0 = __ldg(a.tgt_off + t), j1 = __ldg(a.tgt_off + t + 1);
    if (j0 < 0 || j1 < j0 || (j1 > j0 && a.exp_idx == nullptr)) {  // an empty list set may pass NULL
        atomicOr(a.err, 8u);
        j0 = j1 = 0;
    }
    const double x = __ldg(a.tgt + t), y = __ldg(a.tgt + a.n_tgt + t), z = __ldg(a.tgt + 2 * a.n_tgt + t);
    double acc = 0.0;
#pragma unroll 1
    for (int64_t j = j0; j < j1; ++j) {
        const int64_t e = __ldg(a.exp_idx + j);
        if (e < 0 || e >= a.n_exp) {
            atomicOr(a.err, 1u);
            continue;
        }
        acc += eval_one(a.coef + e * (int64_t)a.np, a.p, a.norm, x - __ldg(a.exp_c + e),
                        y - __ldg(a.exp_c + a.n_exp + e), z - __ldg(a.exp_c + 2 * a.n_exp + e));
    }
    a.out[t] = a.accumulate ? a.out[t] + acc : acc;
}

// H = curl A at each target (Eq. (st3)): expansions with three component rows.
__global__ void q2x_evaluate_curl_kernel(const EvalArgs a)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n_tgt) return;
    int64_t j0 = __ldg(a.tgt_off + t), j1 = __ldg(a.tgt_off + t + 1);
    if (j0 < 0 || j1 < j0 || (j1 > j0 && a.exp_idx == nullptr)) {  // an empty list set may pass NULL
        atomicOr(a.err, 8u);
        j0 = j1 = 0;
    }
    const double x = __ldg(a.tgt + t), y = __ldg(a.tgt + a.n_tgt + t), z = __ldg(a.tgt + 2 * a.n_tgt + t);
    double g[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};  // g[k][j] = d A_k / d x_j
#pragma unroll 1
    for (int64_t j = j0; j < j1; ++j) {
        const int64_t e = __ldg(a.exp_idx + j);
        if (e < 0 || e >= a.n_exp) {
            atomicOr(a.err, 1u);
            continue;
        }
        grad_one(a.coef + e * (int64_t)a.np, a.n_exp * (int64_t)a.np, a.p, x - __ldg(a.exp_c + e),
                 y - __ldg(a.exp_c + a.n_exp + e), z - __ldg(a.exp_c + 2 * a.n_exp + e), g);
    }
    const double h[3] = {g[2][1] - g[1][2], g[0][2] - g[2][0], g[1][0] - g[0][1]};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double* o = a.out + d * a.n_tgt + t;
        *o = a.accumulate ? *o + h[d] : h[d];
    }
}

}  // namespace q2x

// Whether a call takes the direction path (q2x_farfield.cu).  Its three
// launches and the preparation of the expansions have to be made up for: with
// one expansion the potential at p = 12 takes 56 us against 33 at 16,384 targets,
// 60 against 107 at 65,536, 327 against 1,382 at 2^20 (p = 6: 36 against 42, p = 2:
// 29 against 18 at 65,536); the curl, whose general form is a long FP64 chain,
// 119 us against 173 at 2,200 targets already.  An expansion costs as much as 18 (p =
// 16) to 45 targets (p = 4) of one list entry; how long the lists are is not known
// here.  At p = 12 and 65,536 targets 1,000 expansions take 93 us against 107,
// 2,000 128 against 107 with one entry a target and 371 against 822 with eight
// (8,000: 343 against 107 and 596 against 822); at p = 4 and 600,000 targets 10,000
// 243 against 187.  The scratch stays below 2 GiB; *ws receives it, NULL
// where the general path has to run.
static q2x_status take_directions(q2x_plan_t plan, int p, int comps, int64_t n_exp, int64_t n_tgt, void** ws)
{
    *ws = nullptr;
    const int64_t entries = (int64_t)(p + 1) * (p + 2) / 2;
    if (p < 2 || n_exp <= 0 || n_exp > 0x7fffffffLL || n_tgt / (p < 8 ? 64 : 32) < n_exp) return Q2X_OK;
    if (n_tgt < (comps == 1 ? 3000000 : 180000) / entries) return Q2X_OK;
    const size_t bytes = q2x::far_workspace(p, comps, n_exp);
    if (bytes > ((size_t)2 << 30)) return Q2X_OK;
    return q2x_plan_scratch(plan, bytes, ws);
}

extern "C" q2x_status q2x_evaluate_curl(q2x_plan_t plan, int p, int64_t n_exp, const double* coef3,
                                        const double* exp_c, int64_t n_tgt, const double* tgt,
                                        const int64_t* tgt_off, const int64_t* exp_idx, double* out3,
                                        int accumulate)
{
    if (!plan) return q2x_fail(nullptr, Q2X_ERR_ARG, "plan is NULL");
    if (plan->norm != 0) return q2x_fail(plan, Q2X_ERR_UNSUPPORTED, "curl evaluation needs the COEFF norm");
    if (p < 0 || p > plan->p_max) return q2x_fail(plan, Q2X_ERR_RANGE, "p = %d outside 0..%d", p, plan->p_max);
    if (n_exp < 0 || n_tgt < 0) return q2x_fail(plan, Q2X_ERR_ARG, "negative size");
    if (accumulate != 0 && accumulate != 1) return q2x_fail(plan, Q2X_ERR_ARG, "accumulate must be 0 or 1");
    if (n_tgt == 0) return Q2X_OK;
    if (!tgt || !tgt_off || !out3) return q2x_fail(plan, Q2X_ERR_ARG, "NULL target array");
    if (n_exp > 0 && (!coef3 || !exp_c)) return q2x_fail(plan, Q2X_ERR_ARG, "NULL expansion array");
    cudaError_t e = cudaSetDevice(plan->device);
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "cudaSetDevice");
    q2x::EvalArgs a;
    a.p = p;
    a.np = (p + 1) * (p + 1);
    a.norm = 0;
    a.accumulate = accumulate;
    a.n_exp = n_exp;
    a.n_tgt = n_tgt;
    a.coef = coef3;
    a.exp_c = exp_c;
    a.tgt = tgt;
    a.tgt_off = tgt_off;
    a.exp_idx = exp_idx;
    a.out = out3;
    a.err = plan->d_err;
    void* ws;
    q2x_status st = take_directions(plan, p, 3, n_exp, n_tgt, &ws);
    if (st != Q2X_OK) return st;
    if (ws) {
        e = q2x::far_run(a, 3, ws, plan->stream);
        if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "far-field direction kernels");
        plan->launches += 3;
        return Q2X_OK;
    }
    q2x::q2x_evaluate_curl_kernel<<<(unsigned)((n_tgt + 127) / 128), 128, 0, plan->stream>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "q2x_evaluate_curl_kernel launch");
    plan->launches += 1;
    return Q2X_OK;
}

extern "C" q2x_status q2x_evaluate(q2x_plan_t plan, int p, int64_t n_exp, const double* coef, const double* exp_c,
                                   int64_t n_tgt, const double* tgt, const int64_t* tgt_off,
                                   const int64_t* exp_idx, double* out, int accumulate)
{
    if (!plan) return q2x_fail(nullptr, Q2X_ERR_ARG, "plan is NULL");
    if (p < 0 || p > plan->p_max) return q2x_fail(plan, Q2X_ERR_RANGE, "p = %d outside 0..%d", p, plan->p_max);
    if (n_exp < 0 || n_tgt < 0) return q2x_fail(plan, Q2X_ERR_ARG, "negative size");
    if (accumulate != 0 && accumulate != 1) return q2x_fail(plan, Q2X_ERR_ARG, "accumulate must be 0 or 1");
    if (n_tgt == 0) return Q2X_OK;
    if (!tgt || !tgt_off || !out) return q2x_fail(plan, Q2X_ERR_ARG, "NULL target array");
    if (n_exp > 0 && (!coef || !exp_c)) return q2x_fail(plan, Q2X_ERR_ARG, "NULL expansion array");
    cudaError_t e = cudaSetDevice(plan->device);
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "cudaSetDevice");
    q2x::EvalArgs a;
    a.p = p;
    a.np = (p + 1) * (p + 1);
    a.norm = plan->norm;
    a.accumulate = accumulate;
    a.n_exp = n_exp;
    a.n_tgt = n_tgt;
    a.coef = coef;
    a.exp_c = exp_c;
    a.tgt = tgt;
    a.tgt_off = tgt_off;
    a.exp_idx = exp_idx;
    a.out = out;
    a.err = plan->d_err;
    void* ws;
    q2x_status st = take_directions(plan, p, 1, n_exp, n_tgt, &ws);
    if (st != Q2X_OK) return st;
    if (ws) {
        e = q2x::far_run(a, 1, ws, plan->stream);
        if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "far-field direction kernels");
        plan->launches += 3;
        return Q2X_OK;
    }
    const int64_t grid = (n_tgt + 127) / 128;
    q2x::q2x_evaluate_kernel<<<(unsigned)grid, 128, 0, plan->stream>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "q2x_evaluate_kernel launch");
    plan->launches += 1;
    return Q2X_OK;
}
