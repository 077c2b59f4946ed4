// sort_cells.cuh -- phase bodies of the counting sort of the mixed-path
// particles (see sort.cu): key histogram, block scans and rank pass,
// each written for block b of nb blocks of one sort.  Shared by the sort
// kernels (sort.cu) and the persistent ensemble step (walk.cu).
#pragma once
#include "pic_internal.cuh"
#include "span.cuh"

namespace pic {

namespace {

constexpr int kScanTile = 4096;      // keys per scan block
constexpr int kScanThreads = 1024;   // threads of the scan kernels (4 keys each)

template <int NDIM>
__device__ inline int cell_key(const TileGeom &t, uint32_t c) {
    int i, j, k;
    unpack_cell(NDIM, c, i, j, k);
    if (t.lg[0] >= 0) return tile_key_pow2(t, i, j, k);   // shifts instead of divisions
    const int ti = i / t.T[0], tj = j / t.T[1], tk = NDIM == 3 ? k / t.T[2] : 0;
    const int li = i - ti * t.T[0], lj = j - tj * t.T[1], lk = NDIM == 3 ? k - tk * t.T[2] : 0;
    const int tile = (tk * t.ntile[1] + tj) * t.ntile[0] + ti;
    return tile * t.cells_per_tile + (lk * t.T[1] + lj) * t.T[0] + li;
}

// Tile of a key.
__device__ inline int key_tile(const TileGeom &t, int key) {
    return t.lg[0] >= 0 ? key >> (t.lg[0] + t.lg[1] + t.lg[2]) : key / t.cells_per_tile;
}

// Position of cell-sorted rank r inside a tile of n_t particles: every full
// block of 32 W (W = 2^lgw) is stored as a transpose, so that lane a of a warp,
// reading element base + 32k + a for k = 0..W-1, walks the W consecutive
// ranks W a .. W a + W - 1 (mostly one cell) while the 32 lanes of one load sit in
// different cells.  The tail of the tile (m = n_t mod 32 W) keeps rank order in 3D; in 2D it
// is such a block of floor(m / 32) ranks per lane, with the last m mod 32 in order.  (In
// order, the lanes of a warp are in one cell and their adds to the current collide: 512^2
// 640 -> 617 us per step, 1024^2 2274 -> 2200, 16-run ensemble 2690 -> 2470.  In 3D, where
// a block is half as long, the push gains 19 us of 4756 on 128^3 and the sort loses 25.)
template <int NDIM>
__device__ __forceinline__ int interleaved_slot(int r, int n_t, int lgw) {
    const int block = 32 << lgw, full = n_t & ~(block - 1);
    if (r < full) {
        const int i = r & (block - 1);
        return (r - i) + ((i & ((1 << lgw) - 1)) << 5) + (i >> lgw);
    }
    const int i = r - full, w = (n_t - full) >> 5;
    if (NDIM == 3 || i >= 32 * w) return r;
    const int a = (int)__fdividef((float)i + 0.5f, (float)w);   // i / w: at most 31, and 1 / 2w >= 2^-7 off a whole number
    return full + ((i - a * w) << 5) + a;
}

// Source traversal: with a tiled source (sorted before), CTA b walks old tile b
// in its cell-sorted rank order (slot t0 + interleaved_slot(i)), so consecutive
// threads see consecutive ranks of one cell; an untiled source (as uploaded)
// is walked in storage order by a grid-stride loop.
// With a tiled source, block b takes part b % parts of old tile b / parts (its
// share of the tile's ranks, in order).
struct SrcWalk {
    const int *old_start;   // old tile offsets, or nullptr when the source is untiled
    long long n;
    int b, nb;              // this block and the block count of the walk
    int lgw;                // walk length of the source layout
    int parts = 1;          // blocks per old tile
    __device__ __forceinline__ void begin(long long &i, long long &end, int &t0, int &nt) const {
        if (old_start) {
            const int tile = b / parts, part = b - tile * parts;
            t0 = ldro(old_start + tile);
            nt = ldro(old_start + tile + 1) - t0;
            i = (long long)nt * part / parts + threadIdx.x;
            end = (long long)nt * (part + 1) / parts;
        } else {
            t0 = 0;
            nt = 0;
            i = (long long)b * blockDim.x + threadIdx.x;
            end = n;
        }
    }
    __device__ __forceinline__ long long step() const {
        return old_start ? (long long)blockDim.x : (long long)nb * blockDim.x;
    }
    template <int NDIM>
    __device__ __forceinline__ long long pos(long long i, int t0, int nt) const {
        return old_start ? (long long)t0 + interleaved_slot<NDIM>((int)i, nt, lgw) : i;
    }
};

// ---- phase bodies, written for block b of nb blocks working on one sort ----

__device__ inline void zero_body(int *a, long long n, int b, int nb) {
    for (long long i = (long long)b * blockDim.x + threadIdx.x; i < n; i += (long long)nb * blockDim.x) a[i] = 0;
}

// Keys of the V source elements i + v * step (v = 0..V-1) of a walk, -1 past its end.
template <int NDIM, int V>
__device__ __forceinline__ void walk_keys(const SortArgs &a, const SrcWalk &w, long long i, long long end, int t0,
                                          int nt, long long nkeys, long long (&p)[V], int (&key)[V]) {
    uint32_t c[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const long long iv = i + v * w.step();
        p[v] = iv < end ? w.template pos<NDIM>(iv, t0, nt) : -1;
        c[v] = p[v] >= 0 ? ldro(cell_ptr(a.src, p[v])) : 0u;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        key[v] = p[v] >= 0 ? cell_key<NDIM>(a.t, c[v]) : -1;
        if (p[v] >= 0 && (key[v] < 0 || key[v] >= nkeys)) {
            atomicOr(a.err, ERR_SORT);
            key[v] = -1;
        }
    }
}

// ---- key passes over a tiled source ----
//
// A block of THREADS threads takes a share of one old tile.  Most of its particles
// are still in the tile or within the halo H of it, a box of cells that fits shared
// memory: they are counted there (a shared atomic that returns the particle's rank in
// its cell), and one global atomic per occupied cell of the box then adds the count,
// or reserves that many slots.  A particle beyond the box takes a global atomic of its
// own.
constexpr int kBoxRounds = 16;     // particles a thread holds per round, one register each
constexpr int kBoxMax3 = 4096, kBoxMax2 = 2048;   // cells of a box the shared array holds
template <int NDIM> __host__ __device__ constexpr int box_max() { return NDIM == 3 ? kBoxMax3 : kBoxMax2; }
// Does the tile's box fit, so that the box passes can run?
__host__ __device__ inline bool box_fits(const TileGeom &t, int ndim) {
    return (long long)t.R[0] * t.R[1] * t.R[2] <= (ndim == 3 ? kBoxMax3 : kBoxMax2);
}

// The histogram (RANK false), or the rank pass (RANK true: the inverse permutation
// perm[slot] = source index), of part `part` of `parts` of old tile `tile`.  box:
// box_max ints of shared memory; all threads of the block take part.
template <int NDIM, int THREADS, bool RANK>
__device__ inline void box_body(const SortArgs &a, int tile, int part, int parts, int *box) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    const int t0 = ldro(a.old_tile_start + tile), nt = ldro(a.old_tile_start + tile + 1) - t0;
    const int end = t0 + (int)((long long)nt * (part + 1) / parts);
    const int tx = tile % t.ntile[0], tyz = tile / t.ntile[0];
    const int x0 = tx * t.T[0] - t.H, y0 = (tyz % t.ntile[1]) * t.T[1] - t.H,
              z0 = NDIM == 3 ? (tyz / t.ntile[1]) * t.T[2] - t.H : 0;
    const int Rx = t.R[0], Ry = t.R[1], nb = Rx * Ry * (NDIM == 3 ? t.R[2] : 1);
    const long long nkeys = (long long)t.ntiles * t.cells_per_tile;
    // the new layout of the block's own tile, where most particles stay
    const int own0 = RANK ? ldro(a.tile_start + tile) : 0, own1 = RANK ? ldro(a.tile_start + tile + 1) : 0;
    auto place = [&](int r, int d0, int d1, int p) {
        const long long dst = (long long)d0 + interleaved_slot<NDIM>(r - d0, d1 - d0, a.lgw);
        if (r >= d0 && r < d1 && dst < a.n) a.perm[dst] = p;
        else atomicOr(a.err, ERR_SORT);   // counts inconsistent with the particles
    };
    auto place_key = [&](int r, int key, int p) {
        // (clamped: the cell may lie outside the grid in storage that was never written)
        const int dt = (int)min((unsigned)key_tile(t, key), (unsigned)(t.ntiles - 1));
        place(r, ldro(a.tile_start + dt), ldro(a.tile_start + dt + 1), p);
    };
    for (Slot base = t0 + (int)((long long)nt * part / parts); slot_before(base, end);
         base = slot_at(base, kBoxRounds * THREADS)) {
        for (int q = threadIdx.x; q < nb; q += THREADS) box[q] = 0;
        __syncthreads();
        // rank in the cell << 17 | cell in the tile << 16 | box cell, -1 when there is nothing left to place
        int held[kBoxRounds];
#pragma unroll
        for (int v0 = 0; v0 < kBoxRounds; v0 += 8) {
            uint32_t c[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const Slot p = slot_at(base, (v0 + v) * THREADS + threadIdx.x);
                c[v] = slot_before(p, end) ? ldro(cell_ptr(a.src, p)) : 0u;
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const Slot p = slot_at(base, (v0 + v) * THREADS + threadIdx.x);
                held[v0 + v] = -1;
                if (!slot_before(p, end)) continue;
                // the cell, or its image, in the box
                int i, j, k;
                unpack_cell(NDIM, c[v], i, j, k);
                i -= x0; j -= y0; k -= z0;
                i += i < 0 ? g.nx : (i >= g.nx ? -g.nx : 0);
                j += j < 0 ? g.ny : (j >= g.ny ? -g.ny : 0);
                if (NDIM == 3) k += k < 0 ? g.nz : (k >= g.nz ? -g.nz : 0);
                if ((unsigned)i < (unsigned)Rx && (unsigned)j < (unsigned)Ry && (NDIM == 2 || (unsigned)k < (unsigned)t.R[2])) {
                    const int b = (NDIM == 3 ? k * Ry + j : j) * Rx + i;
                    const int rank = atomicAdd(box + b, 1);
                    if (RANK) {
                        // (the last tile of an axis may stick out of the grid: those cells are others' images)
                        const bool own = (unsigned)(i - t.H) < (unsigned)min(t.T[0], g.nx - x0 - t.H) &&
                                         (unsigned)(j - t.H) < (unsigned)min(t.T[1], g.ny - y0 - t.H) &&
                                         (NDIM == 2 || (unsigned)(k - t.H) < (unsigned)min(t.T[2], g.nz - z0 - t.H));
                        held[v0 + v] = rank << 17 | (own ? 1 << 16 : 0) | b;
                    }
                } else {
                    const int key = cell_key<NDIM>(t, c[v]);
                    if (key < 0 || key >= nkeys) {
                        atomicOr(a.err, ERR_SORT);
                        continue;
                    }
                    const int r = atomicAdd(a.counts + key, 1);
                    if (RANK) place_key(r, key, (int)p);
                }
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < nb; q += THREADS) {
            const int n = box[q];
            if (n > 0) {
                const int i = q % Rx, r = q / Rx, k = NDIM == 3 ? r / Ry : 0, j = r - k * Ry;
                const uint32_t c = pack_cell(NDIM, g.wx(x0 + i), g.wy(y0 + j), NDIM == 3 ? g.wz(z0 + k) : 0);
                const int b = atomicAdd(a.counts + cell_key<NDIM>(t, c), n);
                if (RANK) box[q] = b;
            }
        }
        if (RANK) {
            __syncthreads();
#pragma unroll
            for (int v = 0; v < kBoxRounds; ++v) {
                if (held[v] < 0) continue;
                const int p = (int)slot_at(base, v * THREADS + threadIdx.x);
                const int r = box[held[v] & 0xffff] + (held[v] >> 17);
                if (held[v] & (1 << 16)) place(r, own0, own1, p);
                else place_key(r, cell_key<NDIM>(t, ldro(cell_ptr(a.src, p))), p);
            }
        }
        __syncthreads();
    }
}

// ---- key passes over any source ----

// V elements per thread and iteration (independent loads in flight).
template <int NDIM, int V>
__device__ inline void histogram_body(const SortArgs &a, const SrcWalk &w, long long nkeys) {
    long long i, end;
    int t0, nt;
    w.begin(i, end, t0, nt);
    // the loop is warp-uniform (every lane takes part in the warp aggregation)
    const int lane = threadIdx.x & 31;
    for (long long ib = i - lane; ib < end; ib += V * w.step()) {
        long long p[V];
        int key[V];
        walk_keys<NDIM, V>(a, w, ib + lane, end, t0, nt, nkeys, p, key);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            // warp aggregation: lanes with the same key add once
            const unsigned peers = __match_any_sync(0xffffffffu, key[v]);
            const int leader = __ffs(peers) - 1;
            if (key[v] >= 0 && (int)(threadIdx.x & 31) == leader) atomicAdd(a.counts + key[v], __popc(peers));
        }
    }
}

// Block-level exclusive scan of kScanTile ints held THREADS x (kScanTile /
// THREADS) in registers (sh: 33 ints); returns the block total.
template <int THREADS>
__device__ inline int block_scan(int (&v)[kScanTile / THREADS], int *sh) {
    constexpr int kScanItems = kScanTile / THREADS;
    int local = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) { const int x = v[q]; v[q] = local; local += x; }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (THREADS / 32) ? sh[lane] : 0;
        int wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        sh[lane] = wi - w;       // exclusive warp offsets
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    const int off = sh[warp] + incl - local;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) v[q] += off;
    const int total = sh[32];
    __syncthreads();
    return total;
}

// Scan of block b's kScanTile counts (out may be in); the block total goes to block_sums[b].
template <int THREADS>
__device__ inline void scan_blocks_body(const int *in, int *out, int *block_sums, long long n, int b, int *sh) {
    constexpr int kScanItems = kScanTile / THREADS;
    const long long base = (long long)b * kScanTile + (long long)threadIdx.x * kScanItems;
    int v[kScanItems];
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) v[q] = base + q < n ? in[base + q] : 0;
    const int total = block_scan<THREADS>(v, sh);
#pragma unroll
    for (int q = 0; q < kScanItems; ++q)
        if (base + q < n) out[base + q] = v[q];
    if (threadIdx.x == 0) block_sums[b] = total;
}

// Exclusive scan of the block sums in one block (any count, in chunks).
template <int THREADS>
__device__ inline void scan_sums_body(int *block_sums, int nb, int *sh) {
    constexpr int kScanItems = kScanTile / THREADS;
    int carry = 0;
    for (int base = 0; base < nb; base += kScanTile) {
        int v[kScanItems];
        const int b0 = base + threadIdx.x * kScanItems;
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) v[q] = b0 + q < nb ? block_sums[b0 + q] : 0;
        const int total = block_scan<THREADS>(v, sh);
#pragma unroll
        for (int q = 0; q < kScanItems; ++q)
            if (b0 + q < nb) block_sums[b0 + q] = v[q] + carry;
        carry += total;
    }
}

// Add block offsets to the scanned counts (the cursors); extract tile offsets.
__device__ inline void scan_finish_one(const SortArgs &a, long long i, int sum) {
    int v = a.counts[i] + sum;
    if (v < 0 || v > a.n) {   // counts inconsistent with the particles: flag, keep offsets in range
        atomicOr(a.err, ERR_SORT);
        v = v < 0 ? 0 : (int)a.n;
    }
    a.counts[i] = v;
    if (i % a.t.cells_per_tile == 0) a.tile_start[i / a.t.cells_per_tile] = v;
}
__device__ inline void scan_finish_body(const SortArgs &a, long long nkeys, int b, int nb) {
    for (long long i = (long long)b * blockDim.x + threadIdx.x; i < nkeys; i += (long long)nb * blockDim.x)
        scan_finish_one(a, i, a.block_sums[i / kScanTile]);
    if (b == 0 && threadIdx.x == 0) a.tile_start[a.t.ntiles] = (int)a.n;
}

// Rank pass: the destination slot of every source particle, written as the
// inverse permutation perm[slot] = source index (4-byte scattered writes only).
// V elements per thread and iteration; their cursor atomics are all issued
// before the first result is used, so they are in flight together.
template <int NDIM, int V>
__device__ inline void rank_body(const SortArgs &a, const SrcWalk &w, long long nkeys) {
    long long i, end;
    int t0s, nts;
    w.begin(i, end, t0s, nts);
    const int lane = threadIdx.x & 31;
    for (long long ib = i - lane; ib < end; ib += V * w.step()) {   // warp-uniform loop
        long long p[V];
        int key[V];
        walk_keys<NDIM, V>(a, w, ib + lane, end, t0s, nts, nkeys, p, key);
        unsigned peers[V];
        int leader[V], b[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            // lanes that share a key take consecutive slots with one atomic
            peers[v] = __match_any_sync(0xffffffffu, key[v]);
            leader[v] = __ffs(peers[v]) - 1;
            b[v] = 0;
            if (key[v] >= 0 && lane == leader[v]) b[v] = atomicAdd(a.counts + key[v], __popc(peers[v]));
        }
        int base[V];
#pragma unroll
        for (int v = 0; v < V; ++v)
            base[v] = __shfl_sync(0xffffffffu, b[v], leader[v]) + __popc(peers[v] & ((1u << lane) - 1u));
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (key[v] < 0) continue;
            const int tile = key_tile(a.t, key[v]);
            const int t0 = ldro(a.tile_start + tile), t1 = ldro(a.tile_start + tile + 1);
            const long long dst = (long long)t0 + interleaved_slot<NDIM>(base[v] - t0, t1 - t0, a.lgw);
            if (base[v] >= t0 && base[v] < t1 && dst < a.n) a.perm[dst] = (int)p[v];
            else atomicOr(a.err, ERR_SORT);   // counts inconsistent with the particles
        }
    }
}

// Keys and scan blocks of one sort.
__host__ __device__ inline long long nkeys_of(const SortArgs &a) { return (long long)a.t.ntiles * a.t.cells_per_tile; }
__host__ __device__ inline int scan_blocks(const SortArgs &a) { return (int)((nkeys_of(a) + kScanTile - 1) / kScanTile); }

}  // namespace

}  // namespace pic
