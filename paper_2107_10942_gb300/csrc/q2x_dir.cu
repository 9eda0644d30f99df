// q2x_dir.cu -- the direction kernels' tables, instances and set-up (q2x_dir.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "q2x_dir.cuh"
#include "q2x_dirs_table.inc"  // written by gen_directions.py

namespace q2x {

namespace {

// The limit on dynamic shared memory belongs to the function, for all plans and
// threads of the process, so it is the same at every set: the opt-in 227 KB
// less room for the static arrays.
constexpr int kDirSmemMax = 225 * 1024;

template <int KIND, int DENS, int OUTS, int MAX_NT>
cudaError_t dir_attr()
{
    return cudaFuncSetAttribute(q2x_dir_kernel<KIND, DENS, OUTS, MAX_NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kDirSmemMax);
}

template <int KIND, int DENS, int OUTS, int MAX_NT>
cudaError_t dir_launch(const DirArgs& a, int nt, int T, int grid, cudaStream_t st)
{
    const cudaError_t e = dir_attr<KIND, DENS, OUTS, MAX_NT>();
    if (e != cudaSuccess) return e;
    q2x_dir_kernel<KIND, DENS, OUTS, MAX_NT><<<grid, nt, DirCfg<KIND, DENS, OUTS>::smem(a.p_max, T, nt), st>>>(a, T);
    return cudaGetLastError();
}

template <int KIND, int DENS, int OUTS, int MAX_NT>
cudaError_t dir_occupancy(int* blocks, int p, int nt, int T)
{
    const cudaError_t e = dir_attr<KIND, DENS, OUTS, MAX_NT>();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, q2x_dir_kernel<KIND, DENS, OUTS, MAX_NT>, nt,
                                                         DirCfg<KIND, DENS, OUTS>::smem(p, T, nt));
}

#define Q2X_DIR_FNS(K, D, O, M) {&dir_launch<K, D, O, M>, &dir_occupancy<K, D, O, M>}
#define Q2X_DIR_ROW(M)                                                                                       \
    {Q2X_DIR_FNS(KIND_SEG, DENS_CONST, 1, M),  Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 1, M),                      \
     Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 2, M),  Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 3, M),                      \
     Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 1, M), Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 2, M),                     \
     Q2X_DIR_FNS(KIND_TRI, DENS_LINEAR, 3, M), Q2X_DIR_FNS(KIND_TET, DENS_CONST, 1, M),                      \
     Q2X_DIR_FNS(KIND_SEG, DENS_CONST, 4, M),  Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 9, M),                      \
     Q2X_DIR_FNS(KIND_TRI, DENS_CONST, 10, M)}

}  // namespace

const DirFns& dir_fns(int cls, int combo)
{
    static const DirFns f[2][11] = {Q2X_DIR_ROW(256), Q2X_DIR_ROW(128)};
    return f[cls][combo];
}

// 256 threads where two such CTAs fit an SM's shared memory (p = 16, single
// layer: 255 of them at work), else the most that do (800,000 triangles, 200 a
// leaf, both layers, p = 12: 1.67 ms with 192 threads, 2.05 with one CTA of 256);
// a vector density takes one CTA of 256 as long as that fits (2M segments, p =
// 12: 4.5 ms, two of 160 the same).  Where leaves are small a tile keeps few
// groups busy and its frames bound it, so more and smaller CTAs overlap better
// (800,000 triangles, p = 16: 13 a leaf 2.9 ms with 128 threads, 3.9 with 256; 3 a
// leaf 7.3 with 64, 13.5 with 256; p = 8: 13 a leaf 0.88 with 64, 1.90 with 256).
// The line for 128: 53 a leaf 1.15 against 1.31 ms at p = 12 and 1.86 against 2.06
// at p = 16, but 3.08 against 2.86 at p = 20, and 75 a leaf 1.26 against 1.16 at p =
// 12; 40 tetrahedra a leaf 1.14 against 1.45 at p = 10, 0.81 against 1.12 at p = 8.
DirShape dir_shape(int p, int layers, int64_t n_elem, int64_t n_leaves, int num_sms)
{
    const double mean = (double)n_elem / (double)std::max<int64_t>(n_leaves, 1);
    DirShape s{0, 256, 0};
    // accumulators, directions and about 8 groups' records of 128 bytes
    auto smem = [&](int nt) { return (size_t)(p + 1) * (16 * layers * nt + 48) + (size_t)nt / (p + 1) * 1024; };
    const size_t most = layers == 3 ? 200 * 1024 : 110 * 1024;
    while (s.nt > 128 && smem(s.nt) > most) s.nt -= 32;
    if (mean < (p > 16 ? 48.0 : p >= 10 ? 56.0 : 96.0) && layers < 3) {
        s.nt = mean < (p >= 10 ? 5.0 : 20.0) ? 64 : 128;
        s.cls = (p >= 12 && s.nt == 128) ? 0 : 1;
    }
    s.T = dir_tile_elems(p, s.nt);
    // few elements: smaller tiles, down to one element a group, so that every
    // SM has one (1,280 triangles in one leaf at p = 10: 56 tiles of one element
    // a group take 19 us less than 7 full tiles)
    const int64_t spread = n_elem / std::max(num_sms, 1);
    if (spread < s.T) s.T = (int)std::max<int64_t>(std::min(s.T, s.nt / (p + 1)), spread);
    return s;
}

int64_t dir_most_tiles(int p, int64_t n_elem, int num_sms)
{
    const int64_t T = dir_tile_elems(p, 64);
    return std::min(n_elem, std::max((n_elem + T - 1) / T, 2 * (int64_t)num_sms));
}

cudaError_t dir_tables(int p, DirTables* t)
{
    void *vec, *inv, *col;
    cudaError_t e = cudaGetSymbolAddress(&vec, g_dir_vec);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&inv, g_dir_inv);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&col, g_dir_col);
    if (e != cudaSuccess) return e;
    t->vec = static_cast<const int2*>(vec) + h_dir_vec_off[p];
    t->inv = static_cast<const int2*>(inv) + h_dir_inv_off[p];
    t->col = static_cast<const double*>(col);
    return cudaSuccess;
}

cudaError_t dir_setup(DirArgs& a, int nt)
{
    const int p = a.p_max;
    DirTables t;
    cudaError_t e = dir_tables(p, &t);
    if (e != cudaSuccess) return e;
    a.vec = t.vec;
    a.inv = t.inv;
    a.col = t.col;
    a.J = p + 1;
    a.G = nt / a.J;
    a.rnd = 1ll << 31;
    return cudaSuccess;
}

}  // namespace q2x
