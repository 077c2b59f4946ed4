// fields.cu -- Yee FDTD field kernels (App. A.3.2) and the node-averaged fields
// used by the gather (App. A.3.3).
//
// Every kernel runs one thread per padded cell, ghosts included.  A thread
// computes the update of its cell from neighbours that hold the bits of their
// interior images, so a ghost cell receives exactly the value of the interior cell
// it mirrors and the padded arrays stay periodic without a separate copy.
// Each thread reads its own cell and neighbours, and writes only its own cell,
// of arrays that are not read at neighbour positions in the same kernel, so
// no two threads race.
//
// Roofline: HBM bound.  Algorithmic bytes per cell: b advance (both halves) 6 reads +
// 6 writes; e advance 6 + 3 (J) reads, 3 writes, 3 zero-writes; node fields 6
// reads + 6 writes, in units of sizeof(Real) (J: 8 B).  Blocks of 256 cells of one
// z plane, so that a thread divides once for its coordinates.
#include <type_traits>

#include "field_cells.cuh"
#include "pic_internal.cuh"

namespace pic {

namespace {

// Calls body(cell) for the cells of the blocks dealt to this thread block.
template <typename F>
__device__ __forceinline__ void for_cells(const Geom &g, F &&body) {
    const uint32_t plane = (uint32_t)g.px * (uint32_t)g.py;
    const int per = (int)((plane + 255) / 256), n = per * g.pz;
    for (int b = blockIdx.x; b < n; b += gridDim.x) {
        const int k = b / per;
        const uint32_t q = (uint32_t)(b - k * per) * 256 + threadIdx.x;
        if (q < plane) body(CellAt(g, q, k));
    }
}

// Both half advances of b over every padded cell; with a history slot, the interior
// sums of e^2 and b^2 at t are added to it.  carry: see launch_b_advance.
template <typename R>
__global__ void __launch_bounds__(256) k_b_advance(Geom g, FieldPtrs<R> f, R h, HistRef hist, bool carry) {
    double *slot = hist.slot();
    if (slot && carry && blockIdx.x == 0 && threadIdx.x == 0 && hist.has_previous()) slot[0] = slot[-7];
    double *energy_acc = slot ? slot + 2 : nullptr;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for_cells(g, [&](const CellAt &c) { b_advance_cell<R>(g, f, h, c, energy_acc != nullptr, acc); });
    __shared__ double sh[6 * 256];
    if (energy_acc) block_accumulate<6, 256>(acc, energy_acc, sh);
}

// FP64 path: e <- e + dt curl b + J (Ampere, Eq. dyn4 with the deposited current, main
// loop steps 6, 11, 12).
template <typename R>
__global__ void __launch_bounds__(256) k_e_advance(Geom g, FieldPtrs<R> f, const R *J0, const R *J1, const R *J2, R dt) {
    for_cells(g, [&](const CellAt &c) {
        const uint32_t p = c.p, xm = c.xm(g), ym = c.ym(g), zm = c.zm(g);
        const R bx = ld(f.b[0], p), by = ld(f.b[1], p), bz = ld(f.b[2], p);
        const R curl_x = (bz - ld(f.b[2], ym)) - (by - ld(f.b[1], zm));
        const R curl_y = (bx - ld(f.b[0], zm)) - (bz - ld(f.b[2], xm));
        const R curl_z = (by - ld(f.b[1], xm)) - (bx - ld(f.b[0], ym));
        R ex = f.e[0][p] + dt * curl_x + folded_current(g, J0, c);
        R ey = f.e[1][p] + dt * curl_y + folded_current(g, J1, c);
        R ez = f.e[2][p] + dt * curl_z + folded_current(g, J2, c);
        if (g.bcx == 1 && g.wx(c.pi - g.G) == 0) { ey = R(0); ez = R(0); }   // tangential e vanishes on the wall
        f.e[0][p] = ex;
        f.e[1][p] = ey;
        f.e[2][p] = ez;
    });
}

__global__ void __launch_bounds__(256) k_e_advance_fx(Geom g, FieldPtrs<float> f, const unsigned long long *J0,
                                                      const unsigned long long *J1, const unsigned long long *J2,
                                                      unsigned long long *Z0, unsigned long long *Z1,
                                                      unsigned long long *Z2, float dt, F2 scale, long long *hist_inc) {
    // no kernel of this launch reads the counter; the next step's kernels see the new value
    if (hist_inc && blockIdx.x == 0 && threadIdx.x == 0) *hist_inc += 1;
    for_cells(g, [&](const CellAt &c) { e_fx_cell(g, f, J0, J1, J2, Z0, Z1, Z2, dt, scale, c); });
}

template <typename R, typename ZT, typename CT>
__global__ void __launch_bounds__(256) k_e_advance_smoothed(Geom g, FieldPtrs<R> f, const CT *Js, double scale, ZT *Z0,
                                                            ZT *Z1, ZT *Z2, R dt, long long *hist_inc) {
    if (hist_inc && blockIdx.x == 0 && threadIdx.x == 0) *hist_inc += 1;
    for_cells(g, [&](const CellAt &c) { e_smoothed_cell<R, ZT, CT>(g, f, Js, scale, Z0, Z1, Z2, dt, c); });
}

__global__ void __launch_bounds__(256) k_node_fields(Geom g, FieldPtrs<float> f, float4 *nfA, float2 *nfB) {
    for_cells(g, [&](const CellAt &c) { node_cell(g, f, nfA, nfB, c); });
}

__global__ void __launch_bounds__(256) k_node_fields64(Geom g, FieldPtrs<double> f, double2 *nf) {
    for_cells(g, [&](const CellAt &c) { node_cell64(g, f, nf, c); });
}

// Batched over runs: block b belongs to the run r with block_prefix[r] <= b <
// block_prefix[r+1] and updates 256 padded cells of that run.
template <int PHASE>
__global__ void __launch_bounds__(256) k_fields_multi(const FieldRunF *runs, const int *block_prefix, int nruns,
                                                      float h, float dt) {
    __shared__ __align__(16) FieldRunF r;
    __shared__ int run_sh;
    if (threadIdx.x == 0) {
        int lo = 0, hi = nruns;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (block_prefix[mid] <= (int)blockIdx.x) lo = mid; else hi = mid;
        }
        run_sh = lo;
    }
    __syncthreads();
    {
        const int *src = reinterpret_cast<const int *>(runs + run_sh);
        int *dst = reinterpret_cast<int *>(&r);
        for (int q = threadIdx.x; q < (int)(sizeof(FieldRunF) / sizeof(int)); q += blockDim.x) dst[q] = src[q];
    }
    __syncthreads();
    const long long p = (long long)(blockIdx.x - block_prefix[run_sh]) * blockDim.x + threadIdx.x;
    const bool in = p < r.g.pcells;
    const CellAt c(r.g, in ? p : 0);
    if (PHASE == FIELD_B) {
        double *slot = r.hist.slot();
        if (slot && r.carry && p == 0 && r.hist.has_previous()) slot[0] = slot[-7];
        double *energy_acc = slot ? slot + 2 : nullptr;
        double acc[6] = {0, 0, 0, 0, 0, 0};
        if (in) b_advance_cell<float>(r.g, r.f, h, c, energy_acc != nullptr, acc);
        __shared__ double sh[6 * 256];
        if (energy_acc) block_accumulate<6, 256>(acc, energy_acc, sh);
    } else if (PHASE == FIELD_NODE) {
        if (in) node_cell(r.g, r.f, r.nfA, r.nfB, c);
    } else {
        if (r.hist_inc && blockIdx.x == block_prefix[run_sh] && threadIdx.x == 0) *r.hist_inc += 1;
        if (in) {
            if (r.smooth > 0)
                e_smoothed_cell<float, unsigned long long, long long>(r.g, r.f, r.sbuf[r.smooth & 1], r.scale,
                                                                      r.Z[0], r.Z[1], r.Z[2], dt, c);
            else
                e_fx_cell(r.g, r.f, r.J[0], r.J[1], r.J[2], r.Z[0], r.Z[1], r.Z[2], dt,
                          F2{(float)r.scale, (float)(r.scale - (double)(float)r.scale)}, c);
        }
    }
}

template <typename R>
__global__ void k_add_uniform(Geom g, FieldPtrs<R> f, double e0, double e1, double e2, double b0, double b1,
                              double b2) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.pcells; p += stride) {
        int pi, pj, pk;
        padded_coords(g, p, pi, pj, pk);
        const int i = g.wx(pi - g.G);
        double v[6] = {e0, e1, e2, b0, b1, b2};
        if (g.bcx == 1 && i == 0) { v[1] = 0.0; v[2] = 0.0; v[3] = 0.0; }
        if constexpr (std::is_same<R, float>::value) {
            for (int c = 0; c < 3; ++c) {
                const double x = __dadd_rn(e_full(f, c, p), v[c]);
                const float hi = (float)x;
                f.e[c][p] = hi;
                f.el[c][p] = (float)(x - (double)hi);
            }
        } else {
            f.e[0][p] += (R)v[0]; f.e[1][p] += (R)v[1]; f.e[2][p] += (R)v[2];
        }
        f.b[0][p] += (R)v[3]; f.b[1][p] += (R)v[4]; f.b[2][p] += (R)v[5];
    }
}

inline int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    const long long cap = 152LL * 16;   // 16 resident 256-thread blocks per SM on 152 SMs
    return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}
// grid of a for_cells kernel
inline int cells_grid(const Geom &g, int per_sm) {
    const long long n = ((long long)g.px * g.py + 255) / 256 * g.pz;
    return (int)(n < 152LL * per_sm ? n : 152LL * per_sm);
}

}  // namespace

template <typename R>
void launch_b_advance(const Geom &g, FieldPtrs<R> f, R h, HistRef energy, bool carry, cudaStream_t s) {
    // (few blocks: each adds its six sums to the same addresses)
    k_b_advance<R><<<cells_grid(g, 4), 256, 0, s>>>(g, f, h, energy, carry);
}

template <typename R>
void launch_e_advance(const Geom &g, FieldPtrs<R> f, const R *const J[3], R dt, cudaStream_t s) {
    k_e_advance<R><<<cells_grid(g, 16), 256, 0, s>>>(g, f, J[0], J[1], J[2], dt);
}

void launch_node_fields(const Geom &g, FieldPtrs<float> f, float4 *nfA, float2 *nfB, cudaStream_t s) {
    k_node_fields<<<cells_grid(g, 16), 256, 0, s>>>(g, f, nfA, nfB);
}

void launch_node_fields64(const Geom &g, FieldPtrs<double> f, double2 *nf, cudaStream_t s) {
    k_node_fields64<<<cells_grid(g, 16), 256, 0, s>>>(g, f, nf);
}

void launch_fields_multi(int phase, const FieldRunF *runs_dev, const int *block_prefix_dev, int nblocks, int nruns,
                         float h, float dt, cudaStream_t s) {
    if (phase == FIELD_B) k_fields_multi<FIELD_B><<<nblocks, 256, 0, s>>>(runs_dev, block_prefix_dev, nruns, h, dt);
    else if (phase == FIELD_NODE) k_fields_multi<FIELD_NODE><<<nblocks, 256, 0, s>>>(runs_dev, block_prefix_dev, nruns, h, dt);
    else k_fields_multi<FIELD_E_FX><<<nblocks, 256, 0, s>>>(runs_dev, block_prefix_dev, nruns, h, dt);
}

void launch_e_advance_fx(const Geom &g, FieldPtrs<float> f, const unsigned long long *const J[3],
                         unsigned long long *const Jzero[3], float dt, double alpha_abs, long long *hist_inc,
                         cudaStream_t s) {
    const double scale = alpha_abs * 0x1p-36;
    const F2 sc = {(float)scale, (float)(scale - (double)(float)scale)};
    k_e_advance_fx<<<cells_grid(g, 16), 256, 0, s>>>(g, f, J[0], J[1], J[2], Jzero[0], Jzero[1], Jzero[2],
                                                           dt, sc, hist_inc);
}

template <typename R, typename ZT, typename CT>
void launch_e_advance_smoothed(const Geom &g, FieldPtrs<R> f, const CT *Js, double scale, ZT *const Jzero[3],
                               R dt, long long *hist_inc, cudaStream_t s) {
    ZT *const Z[3] = {Jzero ? Jzero[0] : nullptr, Jzero ? Jzero[1] : nullptr, Jzero ? Jzero[2] : nullptr};
    k_e_advance_smoothed<R, ZT, CT><<<cells_grid(g, 16), 256, 0, s>>>(g, f, Js, scale, Z[0], Z[1], Z[2], dt, hist_inc);
}

template <typename R>
void launch_add_uniform(const Geom &g, FieldPtrs<R> f, const double e0[3], const double b0[3], cudaStream_t s) {
    k_add_uniform<R><<<grid_for(g.pcells, 256), 256, 0, s>>>(g, f, e0[0], e0[1], e0[2], b0[0], b0[1], b0[2]);
}

template void launch_b_advance<float>(const Geom &, FieldPtrs<float>, float, HistRef, bool, cudaStream_t);
template void launch_b_advance<double>(const Geom &, FieldPtrs<double>, double, HistRef, bool, cudaStream_t);
template void launch_e_advance<double>(const Geom &, FieldPtrs<double>, const double *const[3], double, cudaStream_t);
template void launch_e_advance_smoothed<double, double, double>(const Geom &, FieldPtrs<double>, const double *,
                                                               double, double *const[3], double, long long *,
                                                               cudaStream_t);
template void launch_e_advance_smoothed<float, unsigned long long, long long>(const Geom &, FieldPtrs<float>,
                                                                              const long long *, double,
                                                                              unsigned long long *const[3], float,
                                                                              long long *, cudaStream_t);
template void launch_add_uniform<float>(const Geom &, FieldPtrs<float>, const double[3], const double[3],
                                        cudaStream_t);
template void launch_add_uniform<double>(const Geom &, FieldPtrs<double>, const double[3], const double[3],
                                         cudaStream_t);

}  // namespace pic
