// q2x_tiles.cu -- leaf tiles of one element set, built on the device: the
// tile list the single-layer FP32 path runs through the batch's persistent
// tile kernel (see q2x_batch.cuh), and its combine.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "q2x_batch.cuh"

namespace q2x {

namespace {

// inclusive warp scan of v
__device__ __forceinline__ int64_t warp_scan(int64_t v, int lane)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += u;
    }
    return v;
}

// exclusive block scan of two counts (blockDim.x == kLeafTileBlock); the
// block totals go to *tot_a, *tot_b
__device__ __forceinline__ void block_scan2(int64_t a, int64_t b, int64_t& ea, int64_t& eb, int64_t* tot_a,
                                            int64_t* tot_b)
{
    __shared__ int64_t wa[32], wb[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t ia = warp_scan(a, lane), ib = warp_scan(b, lane);
    if (lane == 31) {
        wa[wid] = ia;
        wb[wid] = ib;
    }
    __syncthreads();
    if (wid == 0) {
        const int64_t xa = warp_scan(wa[lane], lane), xb = warp_scan(wb[lane], lane);
        wa[lane] = xa - wa[lane];
        wb[lane] = xb - wb[lane];
        if (lane == 31) {
            *tot_a = xa;
            *tot_b = xb;
        }
    }
    __syncthreads();
    ea = wa[wid] + ia - a;
    eb = wb[wid] + ib - b;
}

// element range of leaf L clamped to [0, n_elem) (offsets that decrease or
// leave the range are reported by the offset check; here they only must not
// lead outside the buffers)
__device__ __forceinline__ void leaf_range(const int64_t* leaf_off, int64_t L, int64_t n_elem, int64_t& e0,
                                           int64_t& e1)
{
    e0 = __ldg(leaf_off + L);
    e1 = __ldg(leaf_off + L + 1);
    e0 = e0 < 0 ? 0 : e0 > n_elem ? n_elem : e0;
    e1 = e1 < e0 ? e0 : e1 > n_elem ? n_elem : e1;
}

// tiles of leaf L (0 if empty) and its partial rows (its tiles if it has
// several, else 0)
__device__ __forceinline__ void leaf_counts(const int64_t* leaf_off, int64_t L, int64_t T, int64_t n_elem,
                                            int64_t& nt, int64_t& ns)
{
    int64_t e0, e1;
    leaf_range(leaf_off, L, n_elem, e0, e1);
    const int64_t n = e1 - e0;
    nt = n > 0 ? (n + T - 1) / T : 0;
    ns = nt >= 2 ? nt : 0;
}

// leaf_off must be non-decreasing with leaf_off[0] = 0, leaf_off[n_leaves] = n_elem
__global__ void check_leaf_off_kernel(const int64_t* off, int64_t n_leaves, int64_t n_elem, unsigned* err)
{
    const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (L <= n_leaves && leaf_off_bad(off, L, n_leaves, n_elem)) atomicOr(err, Q2X_DEVERR_LEAF_OFF);
}

__global__ void __launch_bounds__(kLeafTileBlock) leaf_tile_count_kernel(const int64_t* leaf_off, int64_t n_leaves,
                                                                       int64_t T, LeafTileWork w)
{
    const int64_t L = (int64_t)blockIdx.x * kLeafTileBlock + threadIdx.x;
    int64_t nt = 0, ns = 0;
    if (L < n_leaves) leaf_counts(leaf_off, L, T, w.n_elem, nt, ns);
    int64_t et, es;
    block_scan2(nt, ns, et, es, w.block_tiles + blockIdx.x, w.block_slots + blockIdx.x);
    if (L < n_leaves) {
        w.tile_pre[L] = et;
        w.slot_pre[L] = es;
    }
}

// exclusive prefix of the block totals, in place (one block, chunks of
// kLeafTileBlock); the grand total of tiles to *n_tiles
__global__ void __launch_bounds__(kLeafTileBlock) leaf_tile_scan_kernel(int64_t n_blocks, LeafTileWork w)
{
    __shared__ int64_t carry[2];
    if (threadIdx.x == 0) carry[0] = carry[1] = 0;
    __syncthreads();
    for (int64_t b0 = 0; b0 < n_blocks; b0 += kLeafTileBlock) {
        const int64_t b = b0 + threadIdx.x;
        const int64_t vt = b < n_blocks ? w.block_tiles[b] : 0, vs = b < n_blocks ? w.block_slots[b] : 0;
        __shared__ int64_t tot_t, tot_s;
        int64_t et, es;
        block_scan2(vt, vs, et, es, &tot_t, &tot_s);
        if (b < n_blocks) {
            w.block_tiles[b] = carry[0] + et;
            w.block_slots[b] = carry[1] + es;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            carry[0] += tot_t;
            carry[1] += tot_s;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *w.n_tiles = carry[0] < w.max_tiles ? carry[0] : w.max_tiles;
}

// tile i of the nt tiles of leaf L (elements e0 .. e1, balanced sizes) to
// entry `at` of the list; s0 the leaf's first partial row
__device__ __forceinline__ void write_tile(const LeafTileWork& w, int64_t L, int64_t nt, int64_t i, int64_t at,
                                           int64_t s0, int64_t e0, int64_t e1, int combo, int bin)
{
    const int64_t chunk = (e1 - e0 + nt - 1) / nt;
    BatchTile t;
    t.combo = combo;
    t.bin = bin;
    t.leaf = (int32_t)L;
    t.flags = (nt == 1) ? 1 : 0;
    t.slot = (nt == 1) ? 0 : s0 + i;
    t.e_lo = e0 + i * chunk;
    t.e_hi = (t.e_lo + chunk < e1) ? t.e_lo + chunk : e1;
    if (nt > 1 && s0 + i >= w.max_slots) {  // no partial row left (bad offsets only): an empty tile
        t.flags = 1;
        t.slot = 0;
        t.e_hi = t.e_lo;
    }
    w.tiles[at] = t;
}

// one thread per leaf: its tiles (balanced sizes, at most T elements) and
// its partial-row offset
__global__ void leaf_tile_fill_kernel(const int64_t* leaf_off, int64_t n_leaves, int64_t T, int combo, int bin,
                                      LeafTileWork w)
{
    const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (L >= n_leaves) return;
    const int64_t blk = L / kLeafTileBlock;
    const int64_t t0 = w.block_tiles[blk] + w.tile_pre[L];
    const int64_t s0 = w.block_slots[blk] + w.slot_pre[L];
    int64_t nt, ns;
    leaf_counts(leaf_off, L, T, w.n_elem, nt, ns);
    const int64_t smax = w.max_slots;
    w.slot_off[L] = s0 < smax ? s0 : smax;
    if (L == n_leaves - 1) w.slot_off[n_leaves] = s0 + ns < smax ? s0 + ns : smax;
    if (nt == 0) return;
    int64_t e0, e1;
    leaf_range(leaf_off, L, w.n_elem, e0, e1);
    for (int64_t i = 0; i < nt; ++i) {
        if (t0 + i >= w.max_tiles) break;  // past the counted tiles (bad offsets only)
        write_tile(w, L, nt, i, t0 + i, s0, e0, e1, combo, bin);
    }
}

// All of the above for at most kLeafTileBlock leaves, in one launch of one
// block: the offset check, the counts and their scan, the tiles (over all
// threads, each tile's leaf by bisection of the prefix sums) and the tile
// counter's reset.  A small call's five launches took longer than its work.
__global__ void __launch_bounds__(kLeafTileBlock) leaf_tile_small_kernel(const int64_t* leaf_off, int64_t n_leaves,
                                                                       int64_t T, int combo, int bin, LeafTileWork w,
                                                                       unsigned* err)
{
    __shared__ int64_t s_pre[kLeafTileBlock + 1], tot_t, tot_s;
    const int64_t L = threadIdx.x;
    int64_t nt = 0, ns = 0;
    if (L < n_leaves) {
        leaf_counts(leaf_off, L, T, w.n_elem, nt, ns);
        const int64_t o0 = leaf_off[L], o1 = leaf_off[L + 1];
        if (o0 < 0 || o0 > w.n_elem || o1 < o0 || o1 > w.n_elem || (L == 0 && o0 != 0) ||
            (L == n_leaves - 1 && o1 != w.n_elem))
            if (err) atomicOr(err, Q2X_DEVERR_LEAF_OFF);
    }
    int64_t et, es;
    block_scan2(nt, ns, et, es, &tot_t, &tot_s);
    __syncthreads();
    s_pre[L] = et;
    const int64_t smax = w.max_slots;
    if (L < n_leaves) w.slot_off[L] = es < smax ? es : smax;
    if (L == 0) {
        s_pre[kLeafTileBlock] = tot_t;
        w.slot_off[n_leaves] = tot_s < smax ? tot_s : smax;
        *w.n_tiles = tot_t < w.max_tiles ? tot_t : w.max_tiles;
        *w.counter = 0;
    }
    __syncthreads();
    const int64_t n_tiles = tot_t < w.max_tiles ? tot_t : w.max_tiles;
    for (int64_t i = threadIdx.x; i < n_tiles; i += kLeafTileBlock) {
        int lo = 0, hi = kLeafTileBlock - 1;  // the last leaf whose first tile is at most i and that has tiles
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= i)
                lo = mid;
            else
                hi = mid - 1;
        }
        // (leaves without tiles share their successor's prefix: lo is the last of them, the one with tiles)
        int64_t e0, e1;
        leaf_range(leaf_off, lo, w.n_elem, e0, e1);
        const int64_t cnt = s_pre[lo + 1] - s_pre[lo], k = i - s_pre[lo];
        write_tile(w, lo, cnt, k, i, w.slot_off[lo], e0, e1, combo, bin);
    }
}

// One warp per (lpw leaves, every chunks-th 32 columns): each lane reads one leaf's slot and
// element ranges; the warp then handles, one after the other, the leaves that
// have work (several tiles: their partial rows summed in slot order; empty and
// not accumulating: a zero row).  It is a chain of loads, so the warps are as
// many as the chip holds (leaf_tiles_combine), and never fewer leaves than
// give that.
__global__ void leaf_tile_combine_kernel(const double* __restrict__ partial, const int64_t* __restrict__ slot_off,
                                         const int64_t* __restrict__ leaf_off, int np, int64_t n_leaves, double* coef,
                                         int accumulate, int lpw, int chunks)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t L0 = warp / chunks * lpw;
    if (L0 >= n_leaves) return;  // warp-uniform
    const int64_t L = L0 + lane;
    const int c0 = (int)(warp % chunks) * 32 + lane;
    long long s0 = 0, s1 = 0;
    bool work = false;
    if (lane < lpw && L < n_leaves) {
        s0 = slot_off[L];
        s1 = slot_off[L + 1];
        const bool empty = __ldg(leaf_off + L + 1) == __ldg(leaf_off + L);
        // a single-tile leaf wrote its own row
        work = s1 > s0 || (empty && !accumulate);
    }
    unsigned mask = __ballot_sync(0xffffffffu, work);
    while (mask) {
        const int r = __ffs(mask) - 1;
        mask &= mask - 1;
        const long long a0 = __shfl_sync(0xffffffffu, s0, r), a1 = __shfl_sync(0xffffffffu, s1, r);
        for (int c = c0; c < np; c += 32 * chunks) {
            double* at = coef + (L0 + r) * np + c;
            *at = a1 == a0 ? 0.0 : sum_rows(partial + c, a0, a1, np, accumulate, accumulate ? *at : 0.0);
        }
    }
}

}  // namespace

cudaError_t check_leaf_off(const int64_t* leaf_off, int64_t n_leaves, int64_t n_elem, unsigned* err, cudaStream_t st)
{
    check_leaf_off_kernel<<<(unsigned)((n_leaves + 1 + 255) / 256), 256, 0, st>>>(leaf_off, n_leaves, n_elem, err);
    return cudaGetLastError();
}

cudaError_t leaf_tiles_build(const int64_t* leaf_off, int64_t n_leaves, int64_t T, int combo, int bin,
                             const LeafTileWork& w, unsigned* err, int* launches, cudaStream_t st)
{
    if (n_leaves <= kLeafTileBlock) {
        leaf_tile_small_kernel<<<1, kLeafTileBlock, 0, st>>>(leaf_off, n_leaves, T, combo, bin, w, err);
        *launches = 1;
        return cudaGetLastError();
    }
    *launches = 3;
    if (err) {
        const cudaError_t e = check_leaf_off(leaf_off, n_leaves, w.n_elem, err, st);
        if (e != cudaSuccess) return e;
        *launches = 4;
    }
    const cudaError_t e = cudaMemsetAsync(w.counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    const int64_t nb = leaf_tile_blocks(n_leaves);
    leaf_tile_count_kernel<<<(unsigned)nb, kLeafTileBlock, 0, st>>>(leaf_off, n_leaves, T, w);
    leaf_tile_scan_kernel<<<1, kLeafTileBlock, 0, st>>>(nb, w);
    leaf_tile_fill_kernel<<<(unsigned)((n_leaves + 255) / 256), 256, 0, st>>>(leaf_off, n_leaves, T, combo, bin, w);
    return cudaGetLastError();
}

cudaError_t leaf_tiles_combine(const double* partial, const int64_t* slot_off, const int64_t* leaf_off, int np,
                               int64_t n_leaves, double* coef, int accumulate, cudaStream_t st)
{
    // as many warps as 152 SMs hold (64 each), then more leaves and columns a
    // warp.  Whole calls at p = 10, 32 leaves and all columns a warp -> so:
    // 1 leaf of 56 tiles 42.0 -> 27.6 us, some 50 leaves of 0.8 k triangles
    // 249 -> 113, 3 k of 0.2 k 1218 -> 1133 (FP32-mixed 309 -> 225), 12 k
    // (FP32-mixed) 892 -> 761; at 240 k leaves both are the same
    const int warps = 8;
    const int64_t cap = 152 * 64, groups = (n_leaves + 31) / 32;
    const int chunks = (int)std::min<int64_t>((np + 31) / 32, std::max<int64_t>(1, cap / groups));
    int lpw = 1;
    while (lpw < 32 && n_leaves * chunks > cap * lpw) lpw *= 2;
    const int64_t n_warps = (n_leaves + lpw - 1) / lpw * chunks;
    leaf_tile_combine_kernel<<<(unsigned)((n_warps + warps - 1) / warps), warps * 32, 0, st>>>(
        partial, slot_off, leaf_off, np, n_leaves, coef, accumulate, lpw, chunks);
    return cudaGetLastError();
}

}  // namespace q2x
