// field_cells.cuh -- per-cell bodies of the Yee FDTD field updates (App.
// A.3.2), the current fold and the node-averaged fields (App. A.3.3), shared
// by the field kernels (fields.cu) and the persistent ensemble step (walk.cu).
//
// Each body updates one padded cell from its neighbours and writes only that cell
// (see fields.cu for the layout).  Ghost cells hold the bits of the interior cells
// they mirror, so a neighbour is the next padded cell, or the image one period away
// for the outermost layer: one select per axis where wrapping the coordinates took
// the kernels several times their memory time.
#pragma once
#include <type_traits>

#include "pic_internal.cuh"

namespace pic {

namespace {

// Padded coordinates of padded index p: multiply-high divisions while the
// grid has fewer than 2^32 padded cells, 64-bit division beyond.
__device__ inline void padded_coords(const Geom &g, long long p, int &pi, int &pj, int &pk) {
    if (g.pcells <= 0xffffffffLL) {
        const uint32_t n = (uint32_t)p;
        const uint32_t q = g.fpx.div(n);
        pi = (int)(n - q * (uint32_t)g.px);
        const uint32_t r = g.fpy.div(q);
        pj = (int)(q - r * (uint32_t)g.py);
        pk = (int)r;
        return;
    }
    pi = (int)(p % g.px);
    long long q = p / g.px;
    pj = (int)(q % g.py);
    pk = (int)(q / g.py);
}

// A padded cell: its coordinates, and its index modulo 2^32 (grids of more cells
// than that do not fit the device's memory).
struct CellAt {
    int pi, pj, pk;
    uint32_t p;
    __device__ __forceinline__ CellAt(const Geom &g, long long at) : p((uint32_t)at) { padded_coords(g, at, pi, pj, pk); }
    __device__ __forceinline__ CellAt(const Geom &g, int i, int j, int k)
        : pi(i), pj(j), pk(k), p(((uint32_t)k * (uint32_t)g.py + (uint32_t)j) * (uint32_t)g.px + (uint32_t)i) {}
    // cell q of plane pk
    __device__ __forceinline__ CellAt(const Geom &g, uint32_t q, int k) : pk(k) {
        pj = (int)g.fpx.div(q);
        pi = (int)(q - (uint32_t)pj * (uint32_t)g.px);
        p = (uint32_t)k * ((uint32_t)g.px * (uint32_t)g.py) + q;
    }
    __device__ __forceinline__ bool interior(const Geom &g) const {
        return (unsigned)(pi - g.G) < (unsigned)g.nx && (unsigned)(pj - g.G) < (unsigned)g.ny &&
               (unsigned)(pk - g.Gz) < (unsigned)g.nz;
    }
    // interior, and no other padded cell is its image
    __device__ __forceinline__ bool deep(const Geom &g) const {
        return pi >= 2 * g.G && pi < g.nx && pj >= 2 * g.G && pj < g.ny &&
               (g.ndim == 2 || (pk >= 2 * g.Gz && pk < g.nz));
    }
    // padded index of the neighbour below and above on each axis (or of its image)
    __device__ __forceinline__ uint32_t xm(const Geom &g) const { return p + (uint32_t)(pi > 0 ? -1 : g.nx - 1); }
    __device__ __forceinline__ uint32_t xp(const Geom &g) const { return p + (uint32_t)(pi + 1 < g.px ? 1 : 1 - g.nx); }
    __device__ __forceinline__ uint32_t ym(const Geom &g) const {
        return p + (uint32_t)(pj > 0 ? -1 : g.ny - 1) * (uint32_t)g.px;
    }
    __device__ __forceinline__ uint32_t yp(const Geom &g) const {
        return p + (uint32_t)(pj + 1 < g.py ? 1 : 1 - g.ny) * (uint32_t)g.px;
    }
    __device__ __forceinline__ uint32_t zm(const Geom &g) const {
        return p + (uint32_t)(pk > 0 ? -1 : g.nz - 1) * ((uint32_t)g.px * (uint32_t)g.py);
    }
    __device__ __forceinline__ uint32_t zp(const Geom &g) const {
        return p + (uint32_t)(pk + 1 < g.pz ? 1 : 1 - g.nz) * ((uint32_t)g.px * (uint32_t)g.py);
    }
    // index of the interior image in a compact plane
    __device__ __forceinline__ uint32_t compact(const Geom &g) const {
        return ((uint32_t)g.wz(pk - g.Gz) * (uint32_t)g.ny + (uint32_t)g.wy(pj - g.G)) * (uint32_t)g.nx +
               (uint32_t)g.wx(pi - g.G);
    }
};

template <typename R>
__device__ inline R ld(const R *a, uint32_t i) { return ldro(a + i); }

// A float as a double.  The hardware's conversion runs on the FP64 pipe (one warp
// instruction per 16 clocks); normal values take a few integer instructions.
__device__ __forceinline__ double widen(float x) {
    const int b = __float_as_int(x);
    if ((b & 0x7fffffff) == 0) return 0.0;
    if ((unsigned)(b << 1) - 0x01000000u >= 0xfe000000u) return (double)x;   // subnormal, infinite, NaN
    return __hiloint2double((b & (int)0x80000000) | (((b & 0x7fffffff) >> 3) + (896 << 20)), b << 29);
}
__device__ __forceinline__ double widen(double x) { return x; }

// Block-wide FP64 sum of NV values of THREADS threads, one atomicAdd per value per block;
// sh: NV * THREADS doubles.  Warp q sums value q of all threads: 12 FP64 instructions
// per value, where a shuffle tree per warp and value (540 a block of 256, at 16 clocks
// each) made this reduction 30 of the 36 us of the b advance at 64^3.
template <int NV, int THREADS>
__device__ inline void block_accumulate(const double (&v)[NV], double *acc, double *sh) {
    static_assert(NV <= THREADS / 32, "a warp per value");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) sh[q * THREADS + threadIdx.x] = v[q];
    __syncthreads();
    if (warp < NV) {
        double x = sh[warp * THREADS + lane];
#pragma unroll
        for (int w = 1; w < THREADS / 32; ++w) x += sh[warp * THREADS + 32 * w + lane];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) atomicAdd(acc + warp, x);
    }
}

// The two half advances of b of one step, b <- b - h curl e (Faraday, Eq. dyn3 on
// the Yee lattice): e does not change between them, so one pass forms its curl once,
// stores b at t (for the gather) in the compact planes bt and b at t + dt/2 in b.
// With energy, the sums of e^2 and b^2 at t over interior cells go to acc in FP64.
template <typename R>
__device__ __forceinline__ void b_advance_cell(const Geom &g, const FieldPtrs<R> &f, R h, const CellAt &c, bool energy,
                                               double (&acc)[6]) {
    const uint32_t p = c.p, xp = c.xp(g), yp = c.yp(g), zp = c.zp(g);
    const R ex = ld(f.e[0], p), ey = ld(f.e[1], p), ez = ld(f.e[2], p);
    const R curl_x = (ld(f.e[2], yp) - ez) - (ld(f.e[1], zp) - ey);
    const R curl_y = (ld(f.e[0], zp) - ex) - (ld(f.e[2], xp) - ez);
    const R curl_z = (ld(f.e[1], xp) - ey) - (ld(f.e[0], yp) - ex);
    // normal b vanishes on the conductor wall (App. A.4)
    const bool wall = g.bcx == 1 && g.wx(c.pi - g.G) == 0;
    R bx = f.b[0][p] - h * curl_x;
    R by = f.b[1][p] - h * curl_y;
    R bz = f.b[2][p] - h * curl_z;
    if (wall) bx = R(0);
    if (c.interior(g)) {
        const uint32_t q = c.compact(g);
        f.bt[0][q] = bx;
        f.bt[1][q] = by;
        f.bt[2][q] = bz;
        if (energy) {
            const double v[6] = {widen(ex), widen(ey), widen(ez), widen(bx), widen(by), widen(bz)};
#pragma unroll
            for (int q6 = 0; q6 < 6; ++q6) acc[q6] += v[q6] * v[q6];
        }
    }
    bx = bx - h * curl_x;
    by = by - h * curl_y;
    bz = bz - h * curl_z;
    if (wall) bx = R(0);
    f.b[0][p] = bx;
    f.b[1][p] = by;
    f.b[2][p] = bz;
}

// Padded coordinates of the images of interior coordinate i along one axis
// (n cells, ghost width G): i + G - n, i + G, i + G + n, those inside [0, n + 2G),
// in that order; returns their count.
__device__ __forceinline__ int axis_images(int i, int n, int G, int (&q)[3]) {
    int c = 0;
    if (i >= n - G) q[c++] = i + G - n;
    q[c++] = i + G;
    if (i < G) q[c++] = i + G + n;
    return c;
}

// Sum of the current over every padded image of interior cell (i,j,k), in the
// order of increasing image offset along z, y, then x.
template <typename R>
__device__ inline R folded_current(const Geom &g, const R *J, int i, int j, int k) {
    int qx[3], qy[3], qz[3];
    const int nqx = axis_images(i, g.nx, g.G, qx), nqy = axis_images(j, g.ny, g.G, qy);
    const int nqz = g.ndim == 3 ? axis_images(k, g.nz, g.Gz, qz) : (qz[0] = k + g.Gz, 1);
    R s = R(0);
    for (int c = 0; c < nqz; ++c)
        for (int b = 0; b < nqy; ++b) {
            const long long row = ((long long)qz[c] * g.py + qy[b]) * g.px;
            for (int a = 0; a < nqx; ++a) s += J[row + qx[a]];
        }
    return s;
}

template <typename R>
__device__ inline R folded_current(const Geom &g, const R *J, const CellAt &c) {
    if (c.deep(g)) return J[c.p];
    return folded_current(g, J, g.wx(c.pi - g.G), g.wy(c.pj - g.G), g.wz(c.pk - g.Gz));
}

// Mixed path: the same update with the fixed-point current (int64, units of
// 2^-36 of sgn(q) times the volume flux); scale = |alpha| 2^-36, passed as an
// FP32 pair (scale_hi + scale_lo).  e is the FP32 pair e + el (FieldPtrs),
// updated with error-free FP32 transformations (Knuth's TwoSum, and the
// FMA-based exact product): the curl of the FP32 b values, the converted
// integer current and the sum are all carried to about 2^-48 relative, so
// div e - rho~ changes by the rounding of the fluxes alone and does not drift
// with the FP32 rounding of e (a single FP32 e made the Gauss residual grow by
// about 5e-9 of max rho per step in a 128^3 thermal plasma).  The FP32 pipe
// does this at a small fraction of the cost of the same update in FP64.
// Every operation is an explicit round-to-nearest intrinsic, never contracted,
// so the single-run and the batched field kernels give bitwise the same fields.
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, err};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
// curl component (a - a_m) - (b - b_m) of four FP32 values, as a pair
__device__ __forceinline__ F2 curl_pair(float a, float a_m, float b, float b_m) {
    const F2 d1 = two_sum(a, -a_m), d2 = two_sum(b, -b_m);
    const F2 c = two_sum(d1.hi, -d2.hi);
    return {c.hi, __fadd_rn(__fsub_rn(d1.lo, d2.lo), c.lo)};
}
// an int64 as a pair of FP32 values whose sum is exact (|J| < 2^48)
__device__ __forceinline__ F2 ll_pair(long long J) {
    const float h = __ll2float_rn(J);
    return {h, __ll2float_rn(J - (long long)h)};
}
// The pair's new value (e + el) + h curl + scale J, renormalised.
__device__ __forceinline__ F2 e_pair_update(const FieldPtrs<float> &f, int c, long long p, float h, F2 curl,
                                            F2 scale, long long J) {
    const F2 hc = two_prod(h, curl.hi);
    const F2 j = ll_pair(J);
    const F2 sj = two_prod(scale.hi, j.hi);
    const float hc_lo = __fmaf_rn(h, curl.lo, hc.lo);
    const float sj_lo = __fadd_rn(sj.lo, __fadd_rn(__fmul_rn(scale.hi, j.lo), __fmul_rn(scale.lo, j.hi)));
    const F2 s1 = two_sum(f.e[c][p], hc.hi);
    const F2 s2 = two_sum(s1.hi, sj.hi);
    const float lo = __fadd_rn(__fadd_rn(__fadd_rn(f.el[c][p], hc_lo), __fadd_rn(sj_lo, s1.lo)), s2.lo);
    const float hi = __fadd_rn(s2.hi, lo);
    return {hi, __fsub_rn(lo, __fsub_rn(hi, s2.hi))};
}
__device__ __forceinline__ void e_pair_store(const FieldPtrs<float> &f, int c, long long p, F2 v) {
    f.e[c][p] = v.hi;
    f.el[c][p] = v.lo;
}

__device__ __forceinline__ void e_fx_cell(const Geom &g, const FieldPtrs<float> &f, const unsigned long long *J0,
                                          const unsigned long long *J1, const unsigned long long *J2,
                                          unsigned long long *Z0, unsigned long long *Z1, unsigned long long *Z2,
                                          float dt, F2 scale, const CellAt &c) {
    const uint32_t p = c.p, xm = c.xm(g), ym = c.ym(g), zm = c.zm(g);
    const float bx = ld(f.b[0], p), by = ld(f.b[1], p), bz = ld(f.b[2], p);
    const F2 curl_x = curl_pair(bz, ld(f.b[2], ym), by, ld(f.b[1], zm));
    const F2 curl_y = curl_pair(bx, ld(f.b[0], zm), bz, ld(f.b[2], xm));
    const F2 curl_z = curl_pair(by, ld(f.b[1], xm), bx, ld(f.b[0], ym));
    F2 ex = e_pair_update(f, 0, p, dt, curl_x, scale, (long long)folded_current(g, J0, c));
    F2 ey = e_pair_update(f, 1, p, dt, curl_y, scale, (long long)folded_current(g, J1, c));
    F2 ez = e_pair_update(f, 2, p, dt, curl_z, scale, (long long)folded_current(g, J2, c));
    if (g.bcx == 1 && g.wx(c.pi - g.G) == 0) { ey = F2{0.f, 0.f}; ez = F2{0.f, 0.f}; }
    e_pair_store(f, 0, p, ex);
    e_pair_store(f, 1, p, ey);
    e_pair_store(f, 2, p, ez);
    Z0[p] = 0ull;
    Z1[p] = 0ull;
    Z2[p] = 0ull;
}

// The same update with the smoothed current: Js holds 3 compact planes (nx*ny*nz
// each, indexed (k*ny + j)*nx + i) in the units of the path's current, which
// scale converts (1 in the FP64 path, |alpha| 2^-36 in the mixed path).
template <typename R, typename ZT, typename CT>
__device__ __forceinline__ void e_smoothed_cell(const Geom &g, const FieldPtrs<R> &f, const CT *Js, double scale,
                                                ZT *Z0, ZT *Z1, ZT *Z2, R dt, const CellAt &c) {
    const uint32_t p = c.p, xm = c.xm(g), ym = c.ym(g), zm = c.zm(g);
    const long long ncell = (long long)g.nx * g.ny * g.nz;
    const uint32_t q = c.compact(g);
    const bool wall = g.bcx == 1 && g.wx(c.pi - g.G) == 0;
    const R bx = ld(f.b[0], p), by = ld(f.b[1], p), bz = ld(f.b[2], p);
    if constexpr (std::is_same<R, float>::value) {
        // the mixed path's FP32 pair, updated as in e_fx_cell (the smoothed current is int64 fixed point)
        const F2 sc = {(float)scale, (float)(scale - (double)(float)scale)};
        const F2 curl_x = curl_pair(bz, ld(f.b[2], ym), by, ld(f.b[1], zm));
        const F2 curl_y = curl_pair(bx, ld(f.b[0], zm), bz, ld(f.b[2], xm));
        const F2 curl_z = curl_pair(by, ld(f.b[1], xm), bx, ld(f.b[0], ym));
        F2 ex = e_pair_update(f, 0, p, dt, curl_x, sc, (long long)ldro(Js + q));
        F2 ey = e_pair_update(f, 1, p, dt, curl_y, sc, (long long)ldro(Js + ncell + q));
        F2 ez = e_pair_update(f, 2, p, dt, curl_z, sc, (long long)ldro(Js + 2 * ncell + q));
        if (wall) { ey = F2{0.f, 0.f}; ez = F2{0.f, 0.f}; }
        e_pair_store(f, 0, p, ex);
        e_pair_store(f, 1, p, ey);
        e_pair_store(f, 2, p, ez);
    } else {
        const R curl_x = (bz - ld(f.b[2], ym)) - (by - ld(f.b[1], zm));
        const R curl_y = (bx - ld(f.b[0], zm)) - (bz - ld(f.b[2], xm));
        const R curl_z = (by - ld(f.b[1], xm)) - (bx - ld(f.b[0], ym));
        const R jx = (R)(scale * (double)ldro(Js + q));
        const R jy = (R)(scale * (double)ldro(Js + ncell + q));
        const R jz = (R)(scale * (double)ldro(Js + 2 * ncell + q));
        R ex = f.e[0][p] + dt * curl_x + jx;
        R ey = f.e[1][p] + dt * curl_y + jy;
        R ez = f.e[2][p] + dt * curl_z + jz;
        if (wall) { ey = R(0); ez = R(0); }
        f.e[0][p] = ex;
        f.e[1][p] = ey;
        f.e[2][p] = ez;
    }
    if constexpr (std::is_same<R, float>::value) {   // (the FP64 path has one current buffer)
        Z0[p] = ZT(0);
        Z1[p] = ZT(0);
        Z2[p] = ZT(0);
    }
}

// Staggered value read by the gather between conductor walls: a value located inside
// the conductor, or a tangential e / normal b on the wall, reads zero.
template <typename R>
__device__ inline R sval(const Geom &g, const R *a, bool compact, bool xstag, int i, int j, int k) {
    if (xstag) { if (i < 0 || i > g.nx - 1) return R(0); }
    else { if (i <= 0 || i >= g.nx) return R(0); }
    if (compact) return ldro(a + ((long long)g.wz(k) * g.ny + g.wy(j)) * g.nx + g.wx(i));
    return ldro(a + g.widx(i, j, k));
}

// Node-averaged fields (App. A.3.3) at a padded node: e over its two edge
// neighbours, b over its four face neighbours.  b is that of the compact planes bt
// when there are any (within a step), else the padded b.
template <typename R>
__device__ __forceinline__ void node_average(const Geom &g, const FieldPtrs<R> &f, const CellAt &c, R (&E)[3],
                                             R (&B)[3]) {
    const bool mid = f.bt[0] != nullptr;
    const R *const bx = mid ? f.bt[0] : f.b[0], *const by = mid ? f.bt[1] : f.b[1], *const bz = mid ? f.bt[2] : f.b[2];
    if (g.bcx == 1) {
        // node coordinate, not wrapped: the masking needs the true x
        const int i = c.pi - g.G, j = c.pj - g.G, k = c.pk - g.Gz;
        auto e = [&](int a, bool st, int ii, int jj, int kk) { return sval(g, f.e[a], false, st, ii, jj, kk); };
        auto b = [&](const R *a, bool st, int ii, int jj, int kk) { return sval(g, a, mid, st, ii, jj, kk); };
        E[0] = R(0.5) * (e(0, true, i - 1, j, k) + e(0, true, i, j, k));
        E[1] = R(0.5) * (e(1, false, i, j - 1, k) + e(1, false, i, j, k));
        E[2] = R(0.5) * (e(2, false, i, j, k - 1) + e(2, false, i, j, k));
        B[0] = R(0.25) * (b(bx, false, i, j, k) + b(bx, false, i, j - 1, k) + b(bx, false, i, j, k - 1) +
                          b(bx, false, i, j - 1, k - 1));
        B[1] = R(0.25) * (b(by, true, i, j, k) + b(by, true, i - 1, j, k) + b(by, true, i, j, k - 1) +
                          b(by, true, i - 1, j, k - 1));
        B[2] = R(0.25) * (b(bz, true, i, j, k) + b(bz, true, i - 1, j, k) + b(bz, true, i - 1, j - 1, k) +
                          b(bz, true, i, j - 1, k));
        return;
    }
    E[0] = R(0.5) * (ld(f.e[0], c.xm(g)) + ld(f.e[0], c.p));
    E[1] = R(0.5) * (ld(f.e[1], c.ym(g)) + ld(f.e[1], c.p));
    E[2] = R(0.5) * (ld(f.e[2], c.zm(g)) + ld(f.e[2], c.p));
    uint32_t q, x, y, z;   // the cell, and the way to its lower neighbours
    if (mid) {
        const int i = g.wx(c.pi - g.G), j = g.wy(c.pj - g.G), k = g.wz(c.pk - g.Gz);
        q = ((uint32_t)k * (uint32_t)g.ny + (uint32_t)j) * (uint32_t)g.nx + (uint32_t)i;
        x = (uint32_t)(i > 0 ? -1 : g.nx - 1);
        y = (uint32_t)(j > 0 ? -1 : g.ny - 1) * (uint32_t)g.nx;
        z = (uint32_t)(k > 0 ? -1 : g.nz - 1) * ((uint32_t)g.nx * (uint32_t)g.ny);
    } else {
        q = c.p;
        x = c.xm(g) - q;
        y = c.ym(g) - q;
        z = c.zm(g) - q;
    }
    B[0] = R(0.25) * (ld(bx, q) + ld(bx, q + y) + ld(bx, q + z) + ld(bx, q + y + z));
    B[1] = R(0.25) * (ld(by, q) + ld(by, q + x) + ld(by, q + z) + ld(by, q + x + z));
    B[2] = R(0.25) * (ld(bz, q) + ld(bz, q + x) + ld(bz, q + x + y) + ld(bz, q + y));
}

// Mixed path: stored as {E_x,E_y,E_z,B_x} and {B_y,B_z}.
__device__ __forceinline__ void node_cell(const Geom &g, const FieldPtrs<float> &f, float4 *nfA, float2 *nfB,
                                          const CellAt &c) {
    float E[3], B[3];
    node_average<float>(g, f, c, E, B);
    nfA[c.p] = make_float4(E[0], E[1], E[2], B[0]);
    nfB[c.p] = make_float2(B[1], B[2]);
}

// FP64 path: three planes of double2, {E_x,E_y} {E_z,B_x} {B_y,B_z}.
__device__ __forceinline__ void node_cell64(const Geom &g, const FieldPtrs<double> &f, double2 *nf, const CellAt &c) {
    const size_t p = c.p;
    double E[3], B[3];
    node_average<double>(g, f, c, E, B);
    nf[p] = make_double2(E[0], E[1]);
    nf[g.pcells + p] = make_double2(E[2], B[0]);
    nf[2 * g.pcells + p] = make_double2(B[1], B[2]);
}

}  // namespace

}  // namespace pic
