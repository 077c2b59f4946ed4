// sort.cu -- counting sort of the mixed-path particles by tile-major cell key.
//
// key(cell) = tile_index * cells_per_tile + index of the cell inside its tile,
// so particles end up grouped by tile and, inside a tile, by cell; the cell
// order inside a tile is then stored block-transposed (interleaved_slot).  Histogram
// of the keys, exclusive scan, and a rank pass
// that writes the inverse permutation (4 bytes per particle); the push that follows
// reads the particles through it and writes them to the other buffer, so the sort
// moves no particle itself.  The tile offsets are read from the scanned counts.
// Every phase also
// has a batched form that sorts one species of many runs in one launch.
//
// Roofline: HBM bound; per particle 4 B (histogram) + 8 B (rank) plus per key
// 3 x 4 B.  Particle counts are int32 (at most 2^31 - 1 particles per species).
#include <algorithm>

#include "pic_internal.cuh"
#include "sort_cells.cuh"

namespace pic {

namespace {

// ---- block counts of the phases of one sort ----

__host__ __device__ inline int blocks_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    const long long cap = 152LL * 32;
    return (int)(b < 1 ? 1 : (b < cap ? b : cap));
}
constexpr int kWalkThreads = 512;
__host__ __device__ inline int walk_blocks(const SortArgs &a) { return a.old_tile_start ? a.t.ntiles : blocks_for(a.n, kWalkThreads); }
inline int key_blocks(const SortArgs &a) { return blocks_for(nkeys_of(a), 256); }
// The box passes (sort_cells.cuh) take sorted sources whose tile box fits.
__host__ __device__ inline bool boxed(const SortArgs &a) { return a.old_tile_start && box_fits(a.t, a.g.ndim); }

// ---- one run: one launch per phase ----

// blockIdx.y is the species of the run.

__global__ void k_zero(const __grid_constant__ SortPack a) {
    zero_body(a.s[blockIdx.y].counts, nkeys_of(a.s[blockIdx.y]), blockIdx.x, gridDim.x);
}

// Histogram (RANK false) or rank pass; ONE: of the first species alone.
template <int NDIM, bool RANK, bool ONE>
__global__ void __launch_bounds__(kWalkThreads, 3) k_keys(const __grid_constant__ SortPack pack) {
    const SortArgs &a = pack.s[ONE ? 0 : blockIdx.y];
    const int nb = walk_blocks(a);
    if (a.n == 0 || (int)blockIdx.x >= nb) return;
    if (boxed(a)) {
        __shared__ int box[box_max<NDIM>()];
        box_body<NDIM, kWalkThreads, RANK>(a, blockIdx.x, 0, 1, box);
        return;
    }
    const SrcWalk w{a.old_tile_start, a.n, (int)blockIdx.x, nb, a.lgw_src};
    if (RANK) rank_body<NDIM, 4>(a, w, nkeys_of(a));
    else histogram_body<NDIM, 4>(a, w, nkeys_of(a));
}

__global__ void __launch_bounds__(kScanThreads) k_scan_blocks(const __grid_constant__ SortPack pack) {
    __shared__ int sh[33];
    const SortArgs &a = pack.s[blockIdx.y];
    scan_blocks_body<kScanThreads>(a.counts, a.counts, a.block_sums, nkeys_of(a), blockIdx.x, sh);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const __grid_constant__ SortPack pack) {
    __shared__ int sh[33];
    const SortArgs &a = pack.s[blockIdx.y];
    scan_sums_body<kScanThreads>(a.block_sums, scan_blocks(a), sh);
}

// Blocks of kScanTile keys.  With few blocks (kFewBlocks) the sums are not scanned by a
// launch of their own: every block adds up those before it.
constexpr int kFewBlocks = kScanThreads;
__global__ void __launch_bounds__(kScanThreads) k_scan_finish(const __grid_constant__ SortPack pack) {
    __shared__ int sh[33];
    const SortArgs &a = pack.s[blockIdx.y];
    const int b = blockIdx.x;
    int sum;
    if (gridDim.x <= kFewBlocks) {
        int v[kScanTile / kScanThreads] = {(int)threadIdx.x < b ? a.block_sums[threadIdx.x] : 0};
        sum = block_scan<kScanThreads>(v, sh);
    } else sum = a.block_sums[b];
    const long long nkeys = nkeys_of(a), k0 = (long long)b * kScanTile;
    for (long long i = k0 + threadIdx.x; i < min(k0 + kScanTile, nkeys); i += kScanThreads) scan_finish_one(a, i, sum);
    if (b == 0 && threadIdx.x == 0) a.tile_start[a.t.ntiles] = (int)a.n;
}

// Work list of the push: every tile that holds particles, cut into parts of at most
// `size` particles of all species.  list[c] = {tile, part | parts << 16}, list[count]
// for c < *count.  One block.
__global__ void __launch_bounds__(kScanThreads) k_push_parts(PushParts a) {
    __shared__ int sh[kScanThreads / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry = 0;
    for (int t0 = 0; t0 < a.ntiles; t0 += kScanThreads) {
        const int t = t0 + threadIdx.x;
        long long n = 0;
        if (t < a.ntiles)
            for (int q = 0; q < a.nspecies; ++q) n += a.tile_start[q][t + 1] - a.tile_start[q][t];
        const int parts = (int)((n + a.size - 1) / a.size);
        int incl = parts;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sh[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int w = lane < kScanThreads / 32 ? sh[lane] : 0;
            int wi = w;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            sh[lane] = wi - w;
            if (lane == 31) sh[32] = wi;
        }
        __syncthreads();
        const int at = carry + sh[warp] + incl - parts;
        for (int p = 0; p < parts && at + p < a.cap; ++p) a.list[at + p] = make_int2(t, p | parts << 16);
        carry += sh[32];
        __syncthreads();
    }
    if (threadIdx.x == 0) *a.count = carry;
}

// ---- many independent sorts (one species of every run of an ensemble): one
// launch per phase; block B belongs to sort s with prefix[s] <= B < prefix[s+1]
// of that phase's block prefix. ----

__device__ inline int find_sort(const int *prefix, int nsort, int B) {
    int lo = 0, hi = nsort;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= B) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void k_zero_multi(const SortArgs *as, const int *prefix, int nsort) {
    const int s = find_sort(prefix, nsort, blockIdx.x);
    zero_body(as[s].counts, nkeys_of(as[s]), blockIdx.x - prefix[s], prefix[s + 1] - prefix[s]);
}

template <int NDIM>
__global__ void __launch_bounds__(kWalkThreads) k_histogram_multi(const SortArgs *as, const int *prefix, int nsort) {
    const int s = find_sort(prefix, nsort, blockIdx.x);
    const SortArgs &a = as[s];
    if (a.old_tile_start && box_fits(a.t, NDIM)) {
        __shared__ int box[box_max<NDIM>()];
        box_body<NDIM, kWalkThreads, false>(a, blockIdx.x - prefix[s], 0, 1, box);
        return;
    }
    const SrcWalk w{a.old_tile_start, a.n, (int)blockIdx.x - prefix[s], prefix[s + 1] - prefix[s], a.lgw_src};
    histogram_body<NDIM, 4>(a, w, nkeys_of(a));
}

__global__ void __launch_bounds__(kScanThreads) k_scan_blocks_multi(const SortArgs *as, const int *prefix,
                                                                    int nsort) {
    __shared__ int sh[33];
    const int s = find_sort(prefix, nsort, blockIdx.x);
    const SortArgs &a = as[s];
    scan_blocks_body<kScanThreads>(a.counts, a.counts, a.block_sums, nkeys_of(a), blockIdx.x - prefix[s], sh);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums_multi(const SortArgs *as) {
    __shared__ int sh[33];
    const SortArgs &a = as[blockIdx.x];
    scan_sums_body<kScanThreads>(a.block_sums, scan_blocks(a), sh);
}

__global__ void k_scan_finish_multi(const SortArgs *as, const int *prefix, int nsort) {
    const int s = find_sort(prefix, nsort, blockIdx.x);
    scan_finish_body(as[s], nkeys_of(as[s]), blockIdx.x - prefix[s], prefix[s + 1] - prefix[s]);
}

template <int NDIM>
__global__ void __launch_bounds__(kWalkThreads) k_rank_multi(const SortArgs *as, const int *prefix, int nsort) {
    const int s = find_sort(prefix, nsort, blockIdx.x);
    const SortArgs &a = as[s];
    if (a.old_tile_start && box_fits(a.t, NDIM)) {
        __shared__ int box[box_max<NDIM>()];
        box_body<NDIM, kWalkThreads, true>(a, blockIdx.x - prefix[s], 0, 1, box);
        return;
    }
    const SrcWalk w{a.old_tile_start, a.n, (int)blockIdx.x - prefix[s], prefix[s + 1] - prefix[s], a.lgw_src};
    rank_body<NDIM, 4>(a, w, nkeys_of(a));
}

}  // namespace

size_t sort_scan_scratch(long long nkeys) { return (size_t)((nkeys + kScanTile - 1) / kScanTile + 1); }

constexpr long long kApart = 1 << 25;
int launch_sort(const SortPack &a, cudaStream_t s) {
    const SortArgs &a0 = a.s[0];
    int nw = 0;
    long long most = 0;
    for (int q = 0; q < a.n; ++q) {
        nw = std::max(nw, a.s[q].n > 0 ? walk_blocks(a.s[q]) : 0);
        most = std::max(most, a.s[q].n);
    }
    const int nb = scan_blocks(a0);
    int launches = 3;
    // one launch for all species fills the GPU better; large ones each have a launch of their
    // own, whose arguments are at fixed places (128^3, 2 x 67M particles: 1.72 against 1.86 ms a
    // sort; 64^3, 2 x 8.4M: 0.35 against 0.30; 45 x 37 x 51, 2 x 1.7M: 0.125 against 0.092)
    auto keys = [&](auto one, auto all) {
        if (nw == 0) return;
        if (most <= kApart) {
            all<<<dim3(nw, a.n), kWalkThreads, 0, s>>>(a);
            ++launches;
            return;
        }
        for (int q = 0; q < a.n; ++q) {
            SortPack p{};
            p.n = 1;
            p.s[0] = a.s[q];
            if (a.s[q].n > 0) one<<<walk_blocks(a.s[q]), kWalkThreads, 0, s>>>(p), ++launches;
        }
    };
    k_zero<<<dim3(key_blocks(a0), a.n), 256, 0, s>>>(a);
    if (a0.g.ndim == 3) keys(k_keys<3, false, true>, k_keys<3, false, false>);
    else keys(k_keys<2, false, true>, k_keys<2, false, false>);
    k_scan_blocks<<<dim3(nb, a.n), kScanThreads, 0, s>>>(a);
    if (nb > kFewBlocks) k_scan_sums<<<dim3(1, a.n), kScanThreads, 0, s>>>(a);
    k_scan_finish<<<dim3(nb, a.n), kScanThreads, 0, s>>>(a);
    if (a0.g.ndim == 3) keys(k_keys<3, true, true>, k_keys<3, true, false>);
    else keys(k_keys<2, true, true>, k_keys<2, true, false>);
    return launches + (nb > kFewBlocks ? 1 : 0);
}

void launch_push_parts(const PushParts &a, cudaStream_t s) { k_push_parts<<<1, kScanThreads, 0, s>>>(a); }

void sort_multi_prefixes(const SortArgs *h_args, int nsort, int *h_prefix) {
    int *pz = h_prefix, *pw = h_prefix + (nsort + 1), *pb = h_prefix + 2 * (nsort + 1);
    pz[0] = pw[0] = pb[0] = 0;
    for (int i = 0; i < nsort; ++i) {
        const SortArgs &a = h_args[i];
        pz[i + 1] = pz[i] + key_blocks(a);
        pw[i + 1] = pw[i] + (a.n > 0 ? walk_blocks(a) : 0);
        pb[i + 1] = pb[i] + scan_blocks(a);
    }
}

void launch_sort_multi(const SortArgs *d_args, const int *d_prefix, const int *h_prefix, int nsort, int ndim,
                       cudaStream_t s) {
    if (nsort <= 0) return;
    const int *pz = d_prefix, *pw = d_prefix + (nsort + 1), *pb = d_prefix + 2 * (nsort + 1);
    const int nz = h_prefix[nsort], nw = h_prefix[2 * (nsort + 1) - 1], nb = h_prefix[3 * (nsort + 1) - 1];
    k_zero_multi<<<nz, 256, 0, s>>>(d_args, pz, nsort);
    if (nw > 0) {
        if (ndim == 3) k_histogram_multi<3><<<nw, kWalkThreads, 0, s>>>(d_args, pw, nsort);
        else k_histogram_multi<2><<<nw, kWalkThreads, 0, s>>>(d_args, pw, nsort);
    }
    k_scan_blocks_multi<<<nb, kScanThreads, 0, s>>>(d_args, pb, nsort);
    k_scan_sums_multi<<<nsort, kScanThreads, 0, s>>>(d_args);
    k_scan_finish_multi<<<nz, 256, 0, s>>>(d_args, pz, nsort);
    if (nw > 0) {
        if (ndim == 3) k_rank_multi<3><<<nw, kWalkThreads, 0, s>>>(d_args, pw, nsort);
        else k_rank_multi<2><<<nw, kWalkThreads, 0, s>>>(d_args, pw, nsort);
    }
}

}  // namespace pic
