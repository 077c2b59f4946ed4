// sort_fp64.cu -- counting sort of the FP64 path's particles by cell, for grids whose
// node fields and moments do not stay in L2 (push_fp64.cu): the particles in flight
// then touch few cells, and a lane of the push walks particles of one cell.
//
// Passes over one species: a histogram of the cells whose returning atomics give
// every particle its rank inside its cell, the exclusive scan of the counts, the
// inverse permutation (slot -> source index), and a gather of one array at a time
// through one spare array (8 B per particle instead of a second copy of the
// state).  Blocks of 32 << lgw consecutive ranks are stored transposed, so that
// lane a of a warp that reads slots 32 k + a walks consecutive ranks; the last,
// partial block keeps rank order.
//
// Roofline: HBM; per particle 24 B (keys, twice) + 8 B (rank) + 8 B (permutation)
// + 20 B for each of the 5 or 6 arrays.  128^3, 2 x 67M particles: 13.4 ms a sort
// (every 16 steps of 56 ms).
#include <algorithm>

#include "pic_internal.cuh"
#include "sort_cells.cuh"

namespace pic {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(long long n) { return (int)std::max(1LL, std::min((n + kThreads - 1) / kThreads, 152LL * 32)); }

// Interior cell index of particle p (positions lie in the box; a wall particle at
// x = nx belongs to the last cell).
template <int NDIM>
__device__ __forceinline__ int cell_of(const Geom &g, const Species64 &s, long long p) {
    const int i = min((int)s.x[0][p], g.nx - 1), j = min((int)s.x[1][p], g.ny - 1);
    const int k = NDIM == 3 ? min((int)s.x[2][p], g.nz - 1) : 0;
    return (k * g.ny + j) * g.nx + i;
}

template <int NDIM>
__global__ void __launch_bounds__(kThreads) k_rank64(Geom g, Species64 s, long long n, int *counts, int *rank) {
    for (long long p = (long long)blockIdx.x * kThreads + threadIdx.x; p < n; p += (long long)gridDim.x * kThreads)
        rank[p] = atomicAdd(counts + cell_of<NDIM>(g, s, p), 1);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_blocks64(const int *counts, int *offsets, int *sums, long long n) {
    __shared__ int sh[33];
    scan_blocks_body<kScanThreads>(counts, offsets, sums, n, blockIdx.x, sh);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums64(int *sums, int nb) {
    __shared__ int sh[33];
    scan_sums_body<kScanThreads>(sums, nb, sh);
}

template <int NDIM>
__global__ void __launch_bounds__(kThreads) k_perm64(Geom g, Species64 s, long long n, const int *offsets,
                                                     const int *sums, const int *rank, int *perm, int lgw) {
    const long long full = n >> (5 + lgw) << (5 + lgw);
    for (long long p = (long long)blockIdx.x * kThreads + threadIdx.x; p < n; p += (long long)gridDim.x * kThreads) {
        const int key = cell_of<NDIM>(g, s, p);
        long long r = (long long)__ldg(offsets + key) + __ldg(sums + key / kScanTile) + rank[p];
        if (r < full) {
            const int i = (int)r & ((32 << lgw) - 1);
            r += (((i & ((1 << lgw) - 1)) << 5) + (i >> lgw)) - i;
        }
        perm[r] = (int)p;
    }
}

// dst[q] = src[perm[q]] (or perm[q] itself when src is null).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_gather64(T *__restrict__ dst, const T *__restrict__ src,
                                                       const int *__restrict__ perm, long long n) {
    const long long stride = (long long)gridDim.x * kThreads;
    for (long long q = (long long)blockIdx.x * kThreads + threadIdx.x; q < n; q += 4 * stride) {
        int p[4];
        T v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) p[a] = q + a * stride < n ? __ldg(perm + q + a * stride) : -1;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (p[a] >= 0) v[a] = src ? __ldg(src + p[a]) : (T)p[a];
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (p[a] >= 0) dst[q + a * stride] = v[a];
    }
}

}  // namespace

void launch_perm64(const Geom &g, const Species64 &s, long long n, int *counts, int *offsets, int *block_sums,
                   int *rank, int *perm, cudaStream_t st) {
    const long long ncell = (long long)g.nx * g.ny * g.nz;
    const int nb = (int)((ncell + kScanTile - 1) / kScanTile), grid = blocks_for(n), lgw = walk_lg64(n);
    cudaMemsetAsync(counts, 0, sizeof(int) * ncell, st);
    if (g.ndim == 3) k_rank64<3><<<grid, kThreads, 0, st>>>(g, s, n, counts, rank);
    else k_rank64<2><<<grid, kThreads, 0, st>>>(g, s, n, counts, rank);
    k_scan_blocks64<<<nb, kScanThreads, 0, st>>>(counts, offsets, block_sums, ncell);
    k_scan_sums64<<<1, kScanThreads, 0, st>>>(block_sums, nb);
    if (g.ndim == 3) k_perm64<3><<<grid, kThreads, 0, st>>>(g, s, n, offsets, block_sums, rank, perm, lgw);
    else k_perm64<2><<<grid, kThreads, 0, st>>>(g, s, n, offsets, block_sums, rank, perm, lgw);
}

void launch_gather64(double *dst, const double *src, const int *perm, long long n, cudaStream_t st) {
    k_gather64<double><<<blocks_for(n), kThreads, 0, st>>>(dst, src, perm, n);
}

void launch_gather_ids(int32_t *dst, const int32_t *src, const int *perm, long long n, cudaStream_t st) {
    k_gather64<int32_t><<<blocks_for(n), kThreads, 0, st>>>(dst, src, perm, n);
}

}  // namespace pic
