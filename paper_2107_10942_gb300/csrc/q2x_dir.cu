// q2x_dir.cu -- the direction kernels' tables, instances and set-up (q2x_dir.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "q2x_dir.cuh"
#include "q2x_dirs_table.inc"  // written by gen_directions.py

namespace q2x {

namespace {

template <int KIND, int DENS, int OUTS>
cudaError_t dir_attr(int p, int T, size_t* smem)
{
    *smem = DirCfg<KIND, DENS, OUTS>::smem(p, T, dir_threads(p, (OUTS & 4) != 0));
    return cudaFuncSetAttribute(q2x_dir_kernel<KIND, DENS, OUTS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)*smem);
}

template <int KIND, int DENS, int OUTS>
cudaError_t dir_launch(const DirArgs& a, int T, int grid, cudaStream_t st)
{
    size_t smem;
    cudaError_t e = dir_attr<KIND, DENS, OUTS>(a.p_max, T, &smem);
    if (e != cudaSuccess) return e;
    q2x_dir_kernel<KIND, DENS, OUTS><<<grid, dir_threads(a.p_max, (OUTS & 4) != 0), smem, st>>>(a, T);
    return cudaGetLastError();
}

template <int KIND, int DENS, int OUTS>
cudaError_t dir_occupancy(int* blocks, int p, int T)
{
    size_t smem;
    cudaError_t e = dir_attr<KIND, DENS, OUTS>(p, T, &smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, q2x_dir_kernel<KIND, DENS, OUTS>,
                                                         dir_threads(p, (OUTS & 4) != 0), smem);
}

#define Q2X_DIR_FNS(K, D, O) {&dir_launch<K, D, O>, &dir_occupancy<K, D, O>}

}  // namespace

// 256 threads, 17 directions: 255 at work at p = 16.  Smaller CTAs overlap
// their phases better but map twice as many tiles to coefficients (level-9
// sphere, p = 16: 11.4 ms with 256 threads, 11.6 with 128, 12.6 with 160).
// The three sums of a vector density take three times the shared memory: 128.
int dir_threads(int, bool vec) { return vec ? 128 : 256; }

const DirFns* dir_fns()
{
    static const DirFns f[9] = {
        Q2X_DIR_FNS(KIND_SEG, DENS_CONST, 1),  Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 1),
        Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 2),  Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 3),
        Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 1), Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 2),
        Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 3), Q2X_DIR_FNS(KIND_TET, DENS_CONST, 1),
        Q2X_DIR_FNS(KIND_SEG, DENS_CONST, 4)};
    return f;
}

cudaError_t dir_setup(DirArgs& a, int kind, int dens, bool vector)
{
    const int p = a.p_max;
    void *vec, *inv, *eighth, *pw, *col;
    cudaError_t e = cudaGetSymbolAddress(&vec, g_dir_vec);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&inv, g_dir_inv);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&eighth, g_dir_eighth);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&pw, g_dir_pow);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&col, g_dir_col);
    if (e != cudaSuccess) return e;
    a.vec = static_cast<const int2*>(vec) + h_dir_vec_off[p];
    a.inv = static_cast<const int2*>(inv) + h_dir_inv_off[p];
    a.eighth = static_cast<const int2*>(eighth);
    a.pw = static_cast<const double*>(pw);
    a.col = static_cast<const double*>(col);
    a.J = p + 1;
    a.G = dir_threads(p, vector) / a.J;
    a.rnd = (long long)((1ull << 63) + (1ull << 31));
    // Bound of a level's value over the seed's (|u| < 1): the dimension's
    // binomial, for linear density (n+1)(n+2)(n+3)/2 of a half.  Seeds start at
    // 2^55 and values stay below 2^59, so that eight elements' sum fits 62
    // bits: before the degrees where the bound passes 2^4, 2^7, .. every value
    // is divided by 2^3 (the low degrees keep more bits than the highest needs).
    auto bound = [&](int n) {
        double b = n + 1;
        if (kind >= KIND_TRI) b *= (n + 2) / 2.0;
        if (kind == KIND_TET) b *= (n + 3) / 3.0;
        if (dens == DENS_LINEAR) b = std::max(b, b * (n + 3) / 2.0);
        return b;
    };
    a.seed_bits = 55;
    double most = 16.0;
    for (int v = 0; v < 4; ++v, most *= 1 << DIR_EVENT) {
        int n = 1;
        while (n <= p && bound(n) <= most) ++n;
        a.event[v] = n <= p ? n : 1 << 20;
    }
    return cudaSuccess;
}

}  // namespace q2x
