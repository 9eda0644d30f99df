// q2x_octants.cu -- children to parents on an octree level: one translation
// a parent instead of one a child.
//
// A child's shift t = c_child - c_parent is (+-h, +-h, +-h): the mirror image
// of t0 = (h, h, h) in the axes of the bits of its octant o.  In the packed
// real coefficients a mirror in x, y or z is a diagonal of signs (R_n^m has
// the phase (i e^{i phi})^m: x -> -x conjugates it, y -> -y conjugates and
// gives (-1)^m, z -> -z gives (-1)^{n+m}), so with chi(i) the three parity
// bits of entry i
//   T_o[i][j] = s_o(i) s_o(j) T_0[i][j],   s_o(i) = (-1)^{popcount(o & chi(i))},
//   sum_o (T_o M_o)[i] = sum_j T_0[i][j] W[chi(i) ^ chi(j)][j],
//   W[c][j] = sum_o (-1)^{popcount(o & c)} M_o[j]   (a Walsh-Hadamard sum).
// It is exact algebra.  Where the corner or the size of the cube is not a short
// binary fraction, the rounded centres differ from +-h by up to 2^-53 of the
// cube, 5e-14 of h seven levels down: that rest of a child's shift is applied to
// its row first, to first order (the second is below 1e-17): 3,540 children in
// five levels 227 -> 149 us, 225 -> 84 without a rest.  T_0 is real, and half or more of it vanishes: R_k^l(t0)
// has the phase (i e^{i pi/4})^l, real for l = 0 mod 4 and imaginary for
// l = 2 mod 4, while entry (m, j) holds orders m - j and m + j only.
//
// Bound: the FP64 pipe (a warp's FP64 instruction holds it for 80 cycles), so
// the count decides.  At p = 12 a parent costs 6,500 multiply-adds and up to
// 24 x 169 additions of W (absent children skip theirs: some 8 on a surface);
// a child by the general contraction costs 12,000.  The terms are cut into one
// run of equal length a thread, entries in a transposed list, so no lane
// waits; a run's share of an entry goes to a slot in shared memory, and one
// thread an entry adds its slots in order (deterministic).
// Measured at p = 12: 3,592 children of 916 parents 129 -> 31 us (FP64 pipe
// 73 % busy), the levels above (229, 56, 8 and 1 parents) 55 + 20 + 18 + 17 ->
// 15 + 11 + 10 + 9 us, latency of loads by then; the whole pass 214 -> 69 us.
// Errors against 128-bit sums are the general path's or smaller (degrees
// weighted alike: 2.3e-16 against 3.4e-16 a level, 2.2e-15 and 2.0e-15 at the
// root).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdint>
#include <cstring>
#include <vector>

#include "q2x.h"
#include "q2x_plan.h"

namespace {

constexpr int32_t kMagic = 0x51324f43;
constexpr int kMaxChunks = 8;
constexpr int kMaxNp = (Q2X_P_MAX + 1) * (Q2X_P_MAX + 1);

struct Chunk {            // a range of rows, one CTA a parent
    int32_t row0, row1;   // entries written
    int32_t nj;           // columns they need (a prefix)
    int32_t steps;        // terms a thread, the last threads fewer
    int32_t n_terms, n_slots;
    int32_t val, code, start, first;  // byte offsets in the table
};
struct Header {
    int32_t magic, p, norm, chunks;
    Chunk c[kMaxChunks];
};

// threads of a CTA: one an entry, whole warps
__host__ __device__ inline int threads_of(int np) { return (np + 31) / 32 * 32; }

// CTAs a parent: as many as give two an SM, since the top of a tree is one
// CTA's latency; W is formed by each of them
inline int chunks_of(int p, int64_t n_dst)
{
    const int most = p < 4 ? 1 : kMaxChunks;
    return (int)std::max<int64_t>(1, std::min<int64_t>(most, 2 * 152 / std::max<int64_t>(n_dst, 1)));
}

struct Entry {
    int n, m, im;  // degree, order >= 0, imaginary part
};
inline Entry entry_of(int i)
{
    int n = 0;
    while ((n + 1) * (n + 1) <= i) ++n;
    const int m = i - n * n - n;
    return {n, m < 0 ? -m : m, m < 0 ? 1 : 0};
}
inline int parity_of(const Entry& e) { return e.im | (((e.m + e.im) & 1) << 1) | (((e.n + e.m) & 1) << 2); }

struct OctArgs {
    int p, np, norm, chunks, accumulate;
    int64_t n_src, n_dst;
    const double* src;
    const unsigned char* table;
    const int32_t* oct;
    const double* delta;  // NULL or [3][n_src]
    const int64_t* dst_off;
    double* dst;
    unsigned* err;
};

__device__ __forceinline__ double neg(double x)
{
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}

// (a, b) -> (a + b, a - b), either of them absent (zero): no addition then
__device__ __forceinline__ void butterfly(double& a, double& b, bool& ha, bool& hb)
{
    if (ha && hb) {
        const double s = a + b;
        b = a - b;
        a = s;
    } else if (hb) {
        a = b;
        b = neg(b);
    } else {
        b = a;
    }
    ha = hb = ha || hb;
}

// Re or Im of F_n^m moved by a tiny shift d, to first order: the degree-1
// harmonics R_1^0 = -z, R_1^{+-1} = (-+y + i x) / 2 on the degree below.
__device__ __noinline__ double nudge(const double* __restrict__ row, int n, int m, int im, int norm, double dx, double dy, double dz)
{
    if (n == 0) return 0.0;
    const int k0 = (n - 1) * (n - 1) + (n - 1);
    const auto re = [&](int k) { return k < 0 ? -__ldg(row + k0 - k) : k < n ? __ldg(row + k0 + k) : 0.0; };
    const auto img = [&](int k) { return k < 0 ? __ldg(row + k0 + k) : k > 0 && k < n ? __ldg(row + k0 - k) : 0.0; };
    // (k = -1 only from m = 0, where degree 0 has no order 1)
    const bool low = m > 0 || n > 1;
    const double ar = low ? re(m - 1) : 0.0, ai = low ? img(m - 1) : 0.0, br = re(m + 1), bi = img(m + 1);
    const double s = norm ? 0.5 : -0.5;  // MOMENT: R_1^1 on m - 1, R_1^-1 on m + 1; COEFF: -, the other way round
    const double y = norm ? dy : -dy;
    return im ? s * (dx * (ar + br) + y * (bi - ai)) - 2.0 * s * dz * img(m)
              : s * (y * (br - ar) - dx * (ai + bi)) - 2.0 * s * dz * re(m);
}

// REST: with delta (its registers would take a third of the CTAs off an SM)
template <bool REST>
__global__ void octants_kernel(const OctArgs a)
{
    extern __shared__ __align__(16) double smem[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int64_t d = blockIdx.x / a.chunks;
    const Header* h = reinterpret_cast<const Header*>(a.table);
    if (h->magic != kMagic || h->p != a.p || h->norm != a.norm || h->chunks != a.chunks) {
        if (tid == 0) atomicOr(a.err, 1u);  // another table: read no further
        return;
    }
    const Chunk c = h->c[blockIdx.x % a.chunks];
    // ---- the first terms of this thread's run: fetched before W is formed
    constexpr int U = 8;
    const int n = min(c.steps, c.n_terms - tid * c.steps);
    const double* val = reinterpret_cast<const double*>(a.table + c.val) + tid;
    const uint16_t* code = reinterpret_cast<const uint16_t*>(a.table + c.code) + tid;
    int slot = __ldg(reinterpret_cast<const uint16_t*>(a.table + c.start) + tid);
    double v[U], vn[U];
    unsigned cd[U], cn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        v[u] = u < n ? __ldg(val + u * nt) : 0.0;
        cd[u] = u < n ? __ldg(code + u * nt) : 0u;
    }
    int64_t s0 = __ldg(a.dst_off + d), s1 = __ldg(a.dst_off + d + 1);
    if (s0 < 0 || s1 < s0 || s1 > a.n_src || (d == 0 && s0 != 0) || (d == a.n_dst - 1 && s1 != a.n_src)) {
        if (tid == 0) atomicOr(a.err, 8u);  // bad offsets: this destination gets zeros
        s0 = s1 = 0;
    }
    // ---- W of the columns this chunk needs, one thread a column; eight
    // sources' loads in flight
    double* W = smem;  // [8][np]
    double* part = smem + 8 * a.np;
    for (int j = tid; j < c.nj; j += nt) {
        int jn = 0;
        while ((jn + 1) * (jn + 1) <= j) ++jn;
        const int jm = j - jn * jn - jn;
        unsigned present = 0;  // octants so far; their sums in this column of W
        for (int64_t s = s0; s < s1; s += 8) {
            int oct[8];
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool in = s + u < s1;
                oct[u] = in ? __ldg(a.oct + s + u) : -1;
                x[u] = in ? __ldg(a.src + (s + u) * (int64_t)a.np + j) : 0.0;
                if (REST && in) {
                    const double* d3 = a.delta + s + u;
                    x[u] += nudge(a.src + (s + u) * (int64_t)a.np, jn, jm < 0 ? -jm : jm, jm < 0, a.norm, __ldg(d3),
                                  __ldg(d3 + a.n_src), __ldg(d3 + 2 * a.n_src));
                }
                if (in && (oct[u] < 0 || oct[u] > 7) && j == 0) atomicOr(a.err, 1u);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (oct[u] >= 0 && oct[u] < 8) {
                    double* at = W + oct[u] * a.np + j;
                    *at = present >> oct[u] & 1u ? *at + x[u] : x[u];
                    present |= 1u << oct[u];
                }
        }
        double w[8];
        bool has[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            has[o] = present >> o & 1u;
            w[o] = has[o] ? W[o * a.np + j] : 0.0;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int o = 0; o < 8; ++o)
                if (!(o >> b & 1)) butterfly(w[o], w[o | 1 << b], has[o], has[o | 1 << b]);
#pragma unroll
        for (int o = 0; o < 8; ++o) W[o * a.np + j] = w[o];
    }
    __syncthreads();
    // ---- this thread's run of terms, the next eight in flight
    double acc = 0.0;
    for (int k = 0; k < n; k += U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = k + U + u;
            vn[u] = q < n ? __ldg(val + q * nt) : 0.0;
            cn[u] = q < n ? __ldg(code + q * nt) : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k + u < n) {
                acc = fma(v[u], W[cd[u] & 0xfffu], acc);
                if (cd[u] & 0x8000u) {  // the last of its entry in this run
                    part[slot++] = acc;
                    acc = 0.0;
                }
            }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = vn[u];
            cd[u] = cn[u];
        }
    }
    __syncthreads();
    // ---- entries: their slots in order
    const uint16_t* first = reinterpret_cast<const uint16_t*>(a.table + c.first);
    for (int i = c.row0 + tid; i < c.row1; i += nt) {
        const int k0 = __ldg(first + (i - c.row0)), k1 = __ldg(first + (i - c.row0) + 1);
        double v = part[k0];  // every entry has its diagonal term
        for (int k = k0 + 1; k < k1; ++k) v += part[k];
        double* out = a.dst + d * (int64_t)a.np + i;
        *out = a.accumulate ? *out + v : v;
    }
}

}  // namespace

static int64_t octant_table(int p, int norm, double h, int64_t n_dst, void* table, int64_t bytes)
{
    if (p < 0 || p > Q2X_P_MAX || (norm != 0 && norm != 1) || n_dst < 0 || !std::isfinite(h)) return -1;
    const int np = (p + 1) * (p + 1), nt = threads_of(np);
    // R_k^l(t0), l = -k..k, by the recursion of Eq. (rec2)
    std::vector<std::complex<double>> R(np);
    R[0] = 1.0;
    const std::complex<double> ixi(-0.5 * h, 0.5 * h), ieta(0.5 * h, 0.5 * h);
    for (int n = 1; n <= p; ++n)
        for (int m = -n; m <= n; ++m) {
            const int k0 = (n - 1) * (n - 1) + (n - 1);
            std::complex<double> v = 0.0;
            if (m - 1 >= -(n - 1) && m - 1 <= n - 1) v += ixi * R[k0 + m - 1];
            if (m + 1 >= -(n - 1) && m + 1 <= n - 1) v += ieta * R[k0 + m + 1];
            if (m >= -(n - 1) && m <= n - 1) v -= h * R[k0 + m];
            R[n * n + n + m] = v / (double)n;
        }
    // the part of R_k^l that does not vanish by its phase
    const auto r_of = [&](int k, int l, bool& re, bool& im) -> std::complex<double> {
        if (l < -k || l > k) return 0.0;
        const std::complex<double> v = R[k * k + k + l];
        if (l & 1) {
            re = im = true;
            return v;
        }
        if (l & 3) {
            im = true;
            return {0.0, v.imag()};
        }
        re = true;
        return {v.real(), 0.0};
    };
    // rows of T_0: (column, value) of the terms that do not vanish
    struct Term {
        uint16_t j;
        double v;
    };
    std::vector<std::vector<Term>> rows(np);
    std::vector<int> chi(np);
    std::vector<Entry> entries(np);
    for (int i = 0; i < np; ++i) {
        entries[i] = entry_of(i);
        chi[i] = parity_of(entries[i]);
    }
    int64_t total = 0;
    for (int i = 0; i < np; ++i) {
        const Entry& e = entries[i];
        rows[i].reserve((size_t)(e.n + 1) * (e.n + 1));
        for (int j = 0; j < (e.n + 1) * (e.n + 1); ++j) {
            const Entry& f = entries[j];
            const int k = e.n - f.n;
            // F^{-f.m} = (-1)^{f.m} conj F^{f.m}
            bool re = false, im = false;
            const std::complex<double> x = r_of(k, norm ? e.m - f.m : f.m - e.m, re, im);
            const std::complex<double> y =
                f.m ? r_of(k, norm ? e.m + f.m : -f.m - e.m, re, im) * ((f.m & 1) ? -1.0 : 1.0) : 0.0;
            // the entry's part of (x + y) Re F + i (x - y) Im F
            const bool real = e.im == f.im;
            if (!(real ? re : im)) continue;
            double v = !f.im ? (e.im ? (x + y).imag() : (x + y).real())
                             : (e.im ? (x - y).real() : -(x - y).imag());
            if (norm == 0 && (k & 1)) v = -v;
            rows[i].push_back({(uint16_t)j, v});
        }
        total += (int64_t)rows[i].size();
    }
    // chunks of rows with about equal numbers of terms
    const int nc = chunks_of(p, n_dst);
    Header hd{};
    hd.magic = kMagic;
    hd.p = p;
    hd.norm = norm;
    hd.chunks = nc;
    const auto align16 = [](int64_t x) { return (x + 15) / 16 * 16; };
    int64_t at = align16(sizeof(Header)), done = 0;
    for (int q = 0, row = 0; q < nc; ++q) {
        Chunk& c = hd.c[q];
        c.row0 = row;
        while (row < np && (q == nc - 1 || done + (int64_t)rows[row].size() / 2 < total * (q + 1) / nc)) {
            done += (int64_t)rows[row].size();
            c.n_terms += (int32_t)rows[row].size();
            ++row;
        }
        c.row1 = row;
        const int n = row > 0 ? entry_of(row - 1).n : 0;
        c.nj = c.row1 > c.row0 ? (n + 1) * (n + 1) : 0;
        c.steps = (c.n_terms + nt - 1) / nt;
        c.val = (int32_t)at;
        at = align16(at + (int64_t)c.steps * nt * 8);
        c.code = (int32_t)at;
        at = align16(at + (int64_t)c.steps * nt * 2);
        c.start = (int32_t)at;
        at = align16(at + (int64_t)nt * 2);
        c.first = (int32_t)at;
        at = align16(at + (int64_t)(c.row1 - c.row0 + 1) * 2);
    }
    if (!table) return at;
    if (bytes < at) return -1;
    unsigned char* base = static_cast<unsigned char*>(table);
    std::memset(base, 0, (size_t)at);
    for (int q = 0; q < nc; ++q) {
        Chunk& c = hd.c[q];
        double* val = reinterpret_cast<double*>(base + c.val);
        uint16_t* code = reinterpret_cast<uint16_t*>(base + c.code);
        uint16_t* start = reinterpret_cast<uint16_t*>(base + c.start);
        uint16_t* first = reinterpret_cast<uint16_t*>(base + c.first);
        int t = 0, slot = 0;
        for (int i = c.row0; i < c.row1; ++i) {
            first[i - c.row0] = (uint16_t)slot;
            const std::vector<Term>& r = rows[i];
            for (size_t z = 0; z < r.size(); ++z, ++t) {
                const int run = t / c.steps, k = t % c.steps;
                if (k == 0) start[run] = (uint16_t)slot;
                const bool last = z + 1 == r.size() || k + 1 == c.steps;
                val[k * nt + run] = r[z].v;
                code[k * nt + run] =
                    (uint16_t)((chi[i] ^ chi[r[z].j]) * np + r[z].j) | (uint16_t)(last ? 0x8000 : 0);
                if (last) ++slot;
            }
        }
        first[c.row1 - c.row0] = (uint16_t)slot;
        c.n_slots = slot;
    }
    std::memcpy(base, &hd, sizeof(Header));
    return at;
}

extern "C" int64_t q2x_octant_table(int p, int norm, double h, int64_t n_dst, void* table, int64_t bytes)
{
    try {
        return octant_table(p, norm, h, n_dst, table, bytes);
    } catch (...) {  // no host memory
        return -1;
    }
}

extern "C" q2x_status q2x_translate_octants(q2x_plan_t plan, int p, int64_t n_src, const double* src_coef,
                                            const void* table, const int32_t* oct, const double* delta, int64_t n_dst,
                                            const int64_t* dst_off, double* dst_coef, int accumulate)
{
    if (!plan) return q2x_fail(nullptr, Q2X_ERR_ARG, "plan is NULL");
    if (p < 0 || p > plan->p_max) return q2x_fail(plan, Q2X_ERR_RANGE, "p = %d outside 0..%d", p, plan->p_max);
    if (n_src < 0 || n_dst < 0) return q2x_fail(plan, Q2X_ERR_ARG, "negative size");
    if (accumulate != 0 && accumulate != 1) return q2x_fail(plan, Q2X_ERR_ARG, "accumulate must be 0 or 1");
    if (n_dst == 0) return Q2X_OK;
    if (n_dst > 0x7fffffffLL || n_src > ((int64_t)1 << 36)) return q2x_fail(plan, Q2X_ERR_ARG, "size too large");
    if (!dst_off || !dst_coef || !table || (n_src > 0 && (!src_coef || !oct)))
        return q2x_fail(plan, Q2X_ERR_ARG, "NULL array or table");
    cudaError_t e = cudaSetDevice(plan->device);
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "cudaSetDevice");
    OctArgs a;
    a.p = p;
    a.np = (p + 1) * (p + 1);
    a.norm = plan->norm;
    a.chunks = chunks_of(p, n_dst);
    a.accumulate = accumulate;
    a.n_src = n_src;
    a.n_dst = n_dst;
    a.src = src_coef;
    a.table = static_cast<const unsigned char*>(table);
    a.oct = oct;
    a.delta = delta;
    a.dst_off = dst_off;
    a.dst = dst_coef;
    a.err = plan->d_err;
    // W, and a slot for each entry and each run (fewer are used)
    const int nt = threads_of(a.np);
    const size_t smem = sizeof(double) * (size_t)(8 * a.np + a.np + nt);
    static_assert(sizeof(double) * (9 * kMaxNp + kMaxNp + 31) <= 48 * 1024, "shared memory without opt-in");
    const unsigned grid = (unsigned)(n_dst * a.chunks);
    if (delta)
        octants_kernel<true><<<grid, nt, smem, plan->stream>>>(a);
    else
        octants_kernel<false><<<grid, nt, smem, plan->stream>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return q2x_cuda_fail(plan, e, "q2x_translate_octants launch");
    plan->launches += 1;
    return Q2X_OK;
}
