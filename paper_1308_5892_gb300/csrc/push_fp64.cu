// push_fp64.cu -- the FP64 particle kernel: gather from the node-averaged
// fields, Boris push, move and charge-conserving deposit in double precision
// (main loop steps 2, 3, 8, 9 of App. A.3.1).
//
// GB300 issues about 2 FP64 lanes per clock and SM (a warp instruction occupies
// the pipe for 16 clocks), so the kernel is bound by its count of FP64 warp
// instructions, far above HBM (96 B per 3D particle-step take 1/15 of the time).
// One thread per particle with node averages and fluxes formed per particle took
// 274 FP64 instructions a particle in 3D and kept the pipe 22% busy (scattered
// loads and atomics): 11.7 ms for 8.4M particles on 64^3 cells, theta = 1, and
// 1.13 ms for 1.5M particles on 300 x 211, theta = 0.1.  This form takes 186 (227
// warp instructions per 32 particles) and keeps the pipe 88% busy: 3.6 and 0.37 ms.
//  - node averages are formed once per node by the field kernels;
//  - cell, offset, wrap and crossing tests are made on the bits of the doubles
//    by the integer pipe (floor, compare and convert are FP64 work), and
//    reciprocals start from the FP32 units;
//  - the current is summed as moments per cell (moments64), from which
//    k_current64 forms the fluxes once per cell;
//  - the kinetic energy at u^{t-1/2} is the sum the previous step recorded;
//  - a particle that stays in its cell adds to register sums of its lane, which go
//    to memory when the lane's cell changes; one that crosses a node plane is put
//    in a queue of its warp, and paths are cut into pieces 32 at a time, with every
//    lane at work.
// Moments are added in L2 by FP64 reductions without return value (200 G/s at
// scattered addresses, measured, against about 40 G/s needed) on a padded grid whose
// ghost images are folded later, so no index is wrapped.  Grids whose node fields
// and moments exceed L2 keep the particles sorted by cell (sort_fp64.cu).
#include <algorithm>

#include "field_cells.cuh"
#include "pic_internal.cuh"

namespace pic {

namespace {

constexpr int kThreads64 = 64;
constexpr int kWarps64 = 152 * 16;   // warps resident on the GPU (128 registers a thread)
constexpr int kQueue64 = 64;      // per-warp ring of crossing particles (at most 63 wait at any time)
constexpr unsigned kFull = 0xffffffffu;

// Moments of a segment's current.  With weights w = d + D/2 the flux of a segment
// through the four x faces of its cell is s D_x [W_y W_z + (-1)^.. D_y D_z / 12],
// W in {1 - w, w} (deposit_segment): bilinear in (w_y, w_z), so the four sums over
// any particles of a cell follow from four moments, s D_x times 1, w_y, w_z and
// w_y w_z + D_y D_z / 12.  Summing moments takes 18 FP64 instructions per segment
// beyond the weights where the fluxes take 32; k_current64 forms the fluxes
// once per cell.  sink.add(v, a) and sink.add(v, a, b) add a and a * b to moment v: comp 0
// at 0 (w_y, w_z), comp 1 at 4 (w_x, w_z), comp 2 at 8 (w_x, w_y); 2D: 0 (w_y), 2 (w_x),
// 4 (w_x, w_y).
template <int NDIM, class Sink>
__device__ __forceinline__ void moments64(const double d[3], const double D[3], int sign, Sink &sink) {
    double w[3], f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        w[a] = fma(0.5, D[a], d[a]);
        f[a] = __hiloint2double(__double2hiint(D[a]) ^ sign, __double2loint(D[a]));   // s D
    }
    const double tx = D[0] * (1.0 / 12.0);
    const double cxy = fma(w[0], w[1], tx * D[1]);
    if (NDIM == 3) {
        const double ty = D[1] * (1.0 / 12.0);
        const double cxz = fma(w[0], w[2], tx * D[2]), cyz = fma(w[1], w[2], ty * D[2]);
        sink.add(0, f[0]); sink.add(1, f[0], w[1]); sink.add(2, f[0], w[2]); sink.add(3, f[0], cyz);
        sink.add(4, f[1]); sink.add(5, f[1], w[0]); sink.add(6, f[1], w[2]); sink.add(7, f[1], cxz);
        sink.add(8, f[2]); sink.add(9, f[2], w[0]); sink.add(10, f[2], w[1]); sink.add(11, f[2], cxy);
    } else {
        sink.add(0, f[0]); sink.add(1, f[0], w[1]);
        sink.add(2, f[1]); sink.add(3, f[1], w[0]);
        sink.add(4, f[2]); sink.add(5, f[2], w[0]); sink.add(6, f[2], w[1]); sink.add(7, f[2], cxy);
    }
}
template <int NDIM> __host__ __device__ constexpr int nmoments() { return NDIM == 3 ? 12 : 8; }

// Moments of a lane's segments in one cell (padded index q).
template <int NDIM>
struct CellSums64 {
    static constexpr int NV = nmoments<NDIM>();
    double x[NV];
    unsigned q;
    __device__ __forceinline__ void reset(unsigned cell) {
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = 0.0;
        q = cell;
    }
    __device__ __forceinline__ void add(int v, double a) { x[v] += a; }
    __device__ __forceinline__ void add(int v, double a, double b) { x[v] = fma(a, b, x[v]); }
    __device__ __forceinline__ void flush(double *M, size_t plane) const {
        if (q == ~0u) return;
#pragma unroll
        for (int v = 0; v < NV; ++v) atomicAdd(M + v * plane + q, x[v]);
    }
};

// The push reads node averages and adds moments, or gathers and deposits at the particle
// itself (direct): a cell's node averages and moments take 112 (2D) or 144 B beside the 96 B
// of its fields, current and diagnostics, and a grid that fills the memory has no room for
// them; and they cost by the cell, which is more than they save where particles are few
// (kDirect64Cells).  No sums are kept per lane then, and the loop over the nodes stays a loop: unrolled
// by 2, 4 and 8 it is as fast (400^3 cells with 2 particles each: 341, 340, 357 ms per step,
// looped 342).
struct MomentCells64 {
    static constexpr bool kDirect = false;
    const double2 *nf;
    double *M;
};
struct DirectCells64 {
    static constexpr bool kDirect = true;
    FieldPtrs<double> f;
    double *J;
    double scale;   // minus alpha (Ampere's law takes minus alpha times the flux)
};

// Fluxes of a segment through the faces of its cell (deposit_segment), scaled, into the
// three padded planes from J (the cell's entry of the first) on.
template <int NDIM>
__device__ __forceinline__ void fluxes64(double *J, size_t plane, unsigned sx, unsigned sxy, const double d[3],
                                         const double D[3], double scale) {
    double w0[3], w1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        w1[a] = fma(0.5, D[a], d[a]);
        w0[a] = 1.0 - w1[a];
    }
    const double ax = scale * D[0], ay = scale * D[1], az = scale * D[2];
    const double cxy = D[0] * D[1] * (1.0 / 12.0);
    double *const Jx = J, *const Jy = J + plane, *const Jz = J + 2 * plane;
    if (NDIM == 3) {
        const double cyz = D[1] * D[2] * (1.0 / 12.0), czx = D[2] * D[0] * (1.0 / 12.0);
        atomicAdd(Jx, ax * fma(w0[1], w0[2], cyz));
        atomicAdd(Jx + sx, ax * fma(w1[1], w0[2], -cyz));
        atomicAdd(Jx + sxy, ax * fma(w0[1], w1[2], -cyz));
        atomicAdd(Jx + sx + sxy, ax * fma(w1[1], w1[2], cyz));
        atomicAdd(Jy, ay * fma(w0[2], w0[0], czx));
        atomicAdd(Jy + 1, ay * fma(w0[2], w1[0], -czx));
        atomicAdd(Jy + sxy, ay * fma(w1[2], w0[0], -czx));
        atomicAdd(Jy + 1 + sxy, ay * fma(w1[2], w1[0], czx));
    } else {
        atomicAdd(Jx, ax * w0[1]);
        atomicAdd(Jx + sx, ax * w1[1]);
        atomicAdd(Jy, ay * w0[0]);
        atomicAdd(Jy + 1, ay * w1[0]);
    }
    atomicAdd(Jz, az * fma(w0[0], w0[1], cxy));
    atomicAdd(Jz + 1, az * fma(w1[0], w0[1], -cxy));
    atomicAdd(Jz + sx, az * fma(w0[0], w1[1], -cxy));
    atomicAdd(Jz + 1 + sx, az * fma(w1[0], w1[1], cxy));
}

// Reciprocal and reciprocal square root of normal x > 0 to the last bit or so: the FP32
// value of the hardware (relative error e0 < 2^-22) corrected by one third-order
// step of Householder's iteration, r (1 + e + e^2) with e = 1 - x r, and
// r (1 + e/2 + 3 e^2/8) with e = 1 - x r^2, whose remainders are below e0^3.
// 3 and 5 FP64 instructions where the library's division and 1 / sqrt take about 9
// and 17.  The exponent is handled by the integer pipe.
__device__ __forceinline__ float to_float_bits(int hi, int lo) {   // truncated mantissa, exponent in FP32's range
    return __int_as_float(((hi - (896 << 20)) << 3) | (int)((unsigned)lo >> 29));
}
__device__ __forceinline__ double from_float_bits(float f) {       // exact, f > 0 normal
    const int b = __float_as_int(f);
    return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}
__device__ __forceinline__ double rcp64(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    if ((unsigned)hi >= 0x7fd00000u) return 1.0 / x;               // result near or below the normal range, inf, NaN
    const int k = (hi & 0x7ff00000) - 0x3ff00000;                  // (exponent of x) << 20
    const double m = __hiloint2double(hi - k, lo);                 // in [1, 2)
    const double r = from_float_bits(__frcp_rn(to_float_bits(hi - k, lo)));
    const double e = fma(-m, r, 1.0);
    const double y = fma(r, fma(e, e, e), r);
    return __hiloint2double(__double2hiint(y) - k, __double2loint(y));
}
__device__ __forceinline__ double rsqrt64(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    if ((unsigned)hi >= 0x7ff00000u) return rsqrt(x);              // inf, NaN
    const int k = ((hi & 0x7fe00000) - 0x3fe00000) >> 21;          // floor((exponent + 1) / 2)
    const int mh = hi - (k << 21);                                 // mantissa times 1/2 .. 2
    const double m = __hiloint2double(mh, lo);
    const double r = from_float_bits(rsqrtf(to_float_bits(mh, lo)));
    const double e = fma(-(m * r), r, 1.0);
    const double y = fma(r * e, fma(0.375, e, 0.5), r);
    return __hiloint2double(__double2hiint(y) - (k << 20), __double2loint(y));
}

// Boris step (particle_core.cuh) with every product in a fused multiply-add.
__device__ __forceinline__ void boris64(double u[3], const double E[3], const double B[3], double qe) {
    const double m[3] = {fma(qe, E[0], u[0]), fma(qe, E[1], u[1]), fma(qe, E[2], u[2])};
    const double qb = qe * rsqrt64(fma(m[2], m[2], fma(m[1], m[1], fma(m[0], m[0], 1.0))));
    const double t[3] = {qb * B[0], qb * B[1], qb * B[2]};
    const double r = rcp64(fma(t[2], t[2], fma(t[1], t[1], fma(t[0], t[0], 1.0))));
    const double f = r + r;
    const double s[3] = {f * t[0], f * t[1], f * t[2]};
    const double p[3] = {fma(m[1], t[2], fma(-m[2], t[1], m[0])), fma(m[2], t[0], fma(-m[0], t[2], m[1])),
                         fma(m[0], t[1], fma(-m[1], t[0], m[2]))};
    u[0] = fma(p[1], s[2], fma(-p[2], s[1], fma(qe, E[0], m[0])));
    u[1] = fma(p[2], s[0], fma(-p[0], s[2], fma(qe, E[1], m[1])));
    u[2] = fma(p[0], s[1], fma(-p[1], s[0], fma(qe, E[2], m[2])));
}

// Cell and offset of a position 0 <= x < 2^20, from its bits: the integer part of
// such a double lies in the upper word.  Both are exact.
__device__ __forceinline__ void split_bits(double x, int &c, double &d) {
    const int hi = __double2hiint(x);
    const int e = (hi >> 20) - 1023;                       // x >= 0: no sign bit
    const int mask = e < 0 ? 0 : (int)(0xffffffffu << (20 - e));
    const double f = e < 0 ? 0.0 : __hiloint2double(hi & mask, 0);
    c = e < 0 ? 0 : ((hi & 0xfffff) | 0x100000) >> (20 - e);
    d = x - f;
}

// A cell index 0 <= n < 2^24 as a double, without an FP64 conversion.
__device__ __forceinline__ double int_bits(int n) { return n == 0 ? 0.0 : from_float_bits((float)n); }

template <int NDIM>
__device__ __forceinline__ void gather64(const double2 *__restrict__ nf, size_t plane, unsigned q,
                                         unsigned sx, unsigned sxy, const double d[3], double E[3], double B[3]) {
    E[0] = E[1] = E[2] = B[0] = B[1] = B[2] = 0.0;
    const double w0[3] = {1.0 - d[0], 1.0 - d[1], 1.0 - d[2]};
#pragma unroll
    for (int xi = 0; xi < (NDIM == 3 ? 2 : 1); ++xi)
#pragma unroll
        for (int eta = 0; eta < 2; ++eta)
#pragma unroll
            for (int eps = 0; eps < 2; ++eps) {
                double w = (eps ? d[0] : w0[0]) * (eta ? d[1] : w0[1]);
                if (NDIM == 3) w *= (xi ? d[2] : w0[2]);
                const double2 *p = nf + (q + eps + eta * sx + xi * sxy);
                const double2 a = __ldg(p), b = __ldg(p + plane), c = __ldg(p + 2 * plane);
                E[0] += w * a.x; E[1] += w * a.y; E[2] += w * b.x;
                B[0] += w * b.y; B[1] += w * c.x; B[2] += w * c.y;
            }
}

// The same with the averages of the cell's nodes formed on the way (c: the cell).
template <int NDIM>
__device__ __forceinline__ void gather_direct64(const Geom &g, const FieldPtrs<double> &f, const int c[3],
                                                const double d[3], double E[3], double B[3]) {
    E[0] = E[1] = E[2] = B[0] = B[1] = B[2] = 0.0;
#pragma unroll 1
    for (int q = 0; q < (NDIM == 3 ? 8 : 4); ++q) {
        const int eps = q & 1, eta = (q >> 1) & 1, xi = q >> 2;
        double w = (eps ? d[0] : 1.0 - d[0]) * (eta ? d[1] : 1.0 - d[1]);
        if (NDIM == 3) w *= xi ? d[2] : 1.0 - d[2];
        double e[3], b[3];
        node_average<double>(g, f, CellAt(g, c[0] + g.G + eps, c[1] + g.G + eta, c[2] + g.Gz + xi), e, b);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            E[a] += w * e[a];
            B[a] += w * b[a];
        }
    }
}
template <int NDIM>
__device__ __forceinline__ void gather_cell64(const Geom &g, const MomentCells64 &io, const int *, unsigned q,
                                              const double d[3], double E[3], double B[3]) {
    gather64<NDIM>(io.nf, (size_t)g.pcells, q, (unsigned)g.px, (unsigned)g.px * (unsigned)g.py, d, E, B);
}
template <int NDIM>
__device__ __forceinline__ void gather_cell64(const Geom &g, const DirectCells64 &io, const int *c, unsigned,
                                              const double d[3], double E[3], double B[3]) {
    gather_direct64<NDIM>(g, io.f, c, d, E, B);
}

// One axis of a move: start offset d, displacement D; the cell shift sa and the end
// offset da, by comparisons of the upper word (pa < 0 or -0, pa >= 1).
__device__ __forceinline__ void end_of_move(double d, double D, int &sa, double &da, int *err) {
    const double pa = d + D;
    const int hi = __double2hiint(pa);
    sa = hi < 0 ? -1 : (hi >= 0x3ff00000 ? 1 : 0);
    da = pa - __hiloint2double(hi < 0 ? (int)0xbff00000 : (hi >= 0x3ff00000 ? 0x3ff00000 : 0), 0);
    if ((unsigned)__double2hiint(da) >= 0x3ff00000u) {
        // 1 after rounding (or pa = -0): the next cell's plane.  Anything else here, and
        // a cell beyond that, is faster than one cell per step or not finite.
        if (da == 1.0 && sa < 1) {
            da = 0.0;
            sa += 1;
        } else {
            atomicOr(err, ERR_FAST_MOVE);
            da = d;
            sa = 0;
        }
    }
}

// Reductions of a segment's moments in memory (m: the cell's entry of the first plane).
struct MomentSink64 {
    double *m;
    size_t plane;
    __device__ __forceinline__ void add(int v, double a) { atomicAdd(m + v * plane, a); }
    __device__ __forceinline__ void add(int v, double a, double b) { atomicAdd(m + v * plane, a * b); }
};

// A segment in the cell of padded index `cell`, into memory.
template <int NDIM>
__device__ __forceinline__ void segment64(const MomentCells64 &io, size_t plane, unsigned cell, unsigned, unsigned,
                                          const double d[3], const double D[3], int sign) {
    MomentSink64 m{io.M + cell, plane};
    moments64<NDIM>(d, D, sign, m);
}
template <int NDIM>
__device__ __forceinline__ void segment64(const DirectCells64 &io, size_t plane, unsigned cell, unsigned sx,
                                          unsigned sxy, const double d[3], const double D[3], int) {
    fluxes64<NDIM>(io.J + cell, plane, sx, sxy, d, D, io.scale);
}

// All pieces of a path; cell: padded index of the start cell.
// The path from d0 to the end d1 in the cell shifted by s is cut at the planes it
// crosses, at most one per axis, in the order of the crossing parameters t (ties in
// axis order).  Breakpoints on the crossed axis are the plane's exact value and the
// last piece ends at d1, so the pieces sum to the stored move.  t >= 0, so the
// integer pipe compares them.
template <int NDIM, class IO>
__device__ __forceinline__ void deposit_path64(const IO &io, size_t plane, unsigned cell, unsigned sx, unsigned sxy,
                                               const double d0[3], const int s[3], const double d1[3], double dz,
                                               int sign) {
    double cur[3], dv[3];
    long long t[3];
    const long long never = 0x4000000000000000LL;   // 2.0
    const unsigned stride[3] = {1u, sx, sxy};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cur[a] = a < NDIM ? d0[a] : 0.0;
        dv[a] = 0.0;
        t[a] = never;
        if (a >= NDIM) continue;
        const double to = s[a] > 0 ? 1.0 : 0.0, from = s[a] > 0 ? 0.0 : 1.0;
        const double first = to - cur[a], cross = first + (d1[a] - from);
        dv[a] = s[a] != 0 ? cross : d1[a] - cur[a];
        const double q = fabs(first) * rcp64(fabs(cross));
        if (s[a] != 0) t[a] = cross != 0.0 ? __double_as_longlong(q) : 0LL;
    }
    double tprev = 0.0;
#pragma unroll 1
    for (;;) {
        const long long tmin = min(t[0], min(t[1], t[2]));
        const bool last = tmin == never;
        const double dt = (last ? 1.0 : __longlong_as_double(tmin)) - tprev;
        const int ax = t[0] == tmin ? 0 : (t[1] == tmin ? 1 : 2);
        double pd[3], pD[3];
        unsigned next = cell;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            pd[a] = cur[a];
            if (a >= NDIM) {
                pD[a] = dz * dt;
                continue;
            }
            const bool cut = !last && ax == a, up = s[a] > 0;
            double e = fma(dv[a], dt, cur[a]);
            if (last) e = d1[a];
            if (cut) e = up ? 1.0 : 0.0;
            pD[a] = e - cur[a];
            cur[a] = cut ? (up ? 0.0 : 1.0) : e;
            if (cut) {
                t[a] = never;
                next += up ? stride[a] : 0u - stride[a];
            }
        }
        segment64<NDIM>(io, plane, cell, sx, sxy, pd, pD, sign);
        if (last) break;
        tprev = __longlong_as_double(tmin);
        cell = next;
    }
}

// Conductor walls (App. A.4): the path to the wall and the mirrored remainder are
// deposited as two legs; x returns the end.  Slow path of the few particles at a wall.
template <int NDIM, class IO>
__device__ __noinline__ void reflect64(const Geom &g, const IO &io, const int c[3], const double d[3], const double D[3],
                                       int sign, double x[3], int *err) {
    const double xs = c[0] + d[0];
    const double wall = xs + D[0] < 0.0 ? 0.0 : (double)g.nx;
    const double t = (wall - xs) / D[0];
    double L[3] = {wall - xs, D[1] * t, D[2] * t};
    double st[3] = {xs, c[1] + d[1], c[2] + d[2]};
#pragma unroll 1
    for (int leg = 0; leg < 2; ++leg) {
        int c0[3] = {0, 0, 0}, s[3] = {0, 0, 0};
        double d0[3] = {0, 0, 0}, d1[3] = {0, 0, 0};
        for (int a = 0; a < NDIM; ++a) {
            double fl = floor(st[a]);
            // a leg that starts on a node plane and moves down starts at offset 1 of the lower cell
            if (st[a] == fl && L[a] < 0.0) fl -= 1.0;
            c0[a] = (int)fl;
            d0[a] = st[a] - fl;
            end_of_move(d0[a], L[a], s[a], d1[a], err);
            x[a] = (double)(c0[a] + s[a]) + d1[a];
        }
        // the second leg may start in the image of a cell beyond a periodic edge
        deposit_path64<NDIM>(io, (size_t)g.pcells,
                             (unsigned)g.pidx(min(max(c0[0], 0), g.nx - 1), g.wy(c0[1]), NDIM == 3 ? g.wz(c0[2]) : 0),
                             (unsigned)g.px, (unsigned)g.px * (unsigned)g.py, d0, s, d1, L[2], sign);
        for (int a = 0; a < 3; ++a) {
            st[a] += L[a];
            L[a] = a == 0 ? -(D[0] - L[0]) : D[a] - L[a];
        }
        st[0] = wall;
    }
    if (x[1] < 0.0) x[1] += g.ny;
    if (x[1] >= g.ny) x[1] -= g.ny;
    if (NDIM == 3) {
        if (x[2] < 0.0) x[2] += g.nz;
        if (x[2] >= g.nz) x[2] -= g.nz;
    }
}

// Blocks of 32 << lgw slots are dealt to the warps in turn, so that the warps in
// flight work on neighbouring blocks; lane a walks the slots base + 32 k + a, which
// after a sort are consecutive cell-sorted particles.
// KIN0: also sum the energy at u^{t-1/2} (first step after a new state).
template <int NDIM, bool WALLS, bool KIN0, class IO>
__global__ void __launch_bounds__(kThreads64, 512 / kThreads64)
    k_push_fp64(const __grid_constant__ Geom g, const __grid_constant__ IO io, Species64 sp, long long n, int lgw, double h, int sign, double dt, double m_over_me, double *kin_acc, int *err) {
    constexpr int ND = NDIM == 3 ? 6 : 5;   // doubles of a queued path: start, end (and D_z in 2D)
    __shared__ double q_val[kThreads64 / 32][ND][kQueue64];
    __shared__ uint2 q_cell[kThreads64 / 32][kQueue64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    double(*qv)[kQueue64] = q_val[warp];
    uint2 *qc = q_cell[warp];
    const unsigned sx = (unsigned)g.px, sxy = (unsigned)g.px * (unsigned)g.py;
    const size_t plane = (size_t)g.pcells;
    CellSums64<NDIM> acc;
    acc.q = ~0u;
    int qhead = 0, qcount = 0;   // warp-uniform
    double kin0 = 0.0, kin1 = 0.0;
    const double qe = h * dt * 0.5;

    // all pieces of the queued path at ring position idx
    auto drain_one = [&](int idx) {
        const uint2 cc = qc[idx];
        const int s[3] = {(int)(cc.y & 3) - 1, (int)((cc.y >> 2) & 3) - 1, (int)((cc.y >> 4) & 3) - 1};
        double d0[3] = {0, 0, 0}, d1[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < NDIM; ++a) {
            d0[a] = qv[a][idx];
            d1[a] = qv[NDIM + a][idx];
        }
        deposit_path64<NDIM>(io, plane, cc.x, sx, sxy, d0, s, d1, NDIM == 2 ? qv[4][idx] : 0.0, sign);
    };

    // (step i of a warp is unit i mod 2^lgw of its block i >> lgw)
    const long long nwarps = (long long)gridDim.x * (kThreads64 / 32);
    long long blk = (long long)blockIdx.x * (kThreads64 / 32) + warp;
    for (int k = 0;; ++k) {
        if (k >> lgw) {
            k = 0;
            blk += nwarps;
        }
        const long long base = (blk << (5 + lgw)) + 32 * k;
        if (base >= n) break;
        const long long p = base + lane;
        bool queued = false;
        double d[3] = {0, 0, 0}, d1[3] = {0, 0, 0}, D[3];
        int s[3] = {0, 0, 0};
        unsigned q = 0;
        if (p < n) {
            double u[3] = {sp.u[0][p], sp.u[1][p], sp.u[2][p]};
            int c[3] = {0, 0, 0};
#pragma unroll
            for (int a = 0; a < NDIM; ++a) split_bits(sp.x[a][p], c[a], d[a]);
            if (WALLS && c[0] >= g.nx) { c[0] = g.nx - 1; d[0] = 1.0; }
            q = ((unsigned)(c[2] + g.Gz) * (unsigned)g.py + (unsigned)(c[1] + g.G)) * (unsigned)g.px +
                (unsigned)(c[0] + g.G);
            double E[3], B[3];
            gather_cell64<NDIM>(g, io, c, q, d, E, B);
            if (KIN0) kin0 += sqrt(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) - 1.0;
            boris64(u, E, B, qe);
            const double g2 = fma(u[2], u[2], fma(u[1], u[1], fma(u[0], u[0], 1.0)));
            const double inv_gam = rsqrt64(g2);
            kin1 += fma(g2, inv_gam, -1.0);
            const double dtg = dt * inv_gam;
#pragma unroll
            for (int a = 0; a < 3; ++a) D[a] = dtg * u[a];
            bool reflect = false;
            if (WALLS) {
                const double xn = (double)c[0] + d[0] + D[0];
                reflect = xn < 0.0 || xn > (double)g.nx;
            }
            if (WALLS && reflect) {
                u[0] = -u[0];
                double x[3];
                reflect64<NDIM>(g, io, c, d, D, sign, x, err);
#pragma unroll
                for (int a = 0; a < NDIM; ++a) sp.x[a][p] = x[a];
            } else {
                const int n3[3] = {g.nx, g.ny, g.nz};
#pragma unroll
                for (int a = 0; a < NDIM; ++a) {
                    end_of_move(d[a], D[a], s[a], d1[a], err);
                    int ni = c[a] + s[a];
                    if (!(WALLS && a == 0)) ni += ni < 0 ? n3[a] : (ni >= n3[a] ? -n3[a] : 0);
                    double xo = int_bits(ni) + d1[a];
                    // rounding of the sum may reach the upper edge of the box
                    if (!(WALLS && a == 0) && ni == n3[a] - 1 && xo >= (double)n3[a]) xo = 0.0;
                    sp.x[a][p] = xo;
                }
                queued = (s[0] | s[1] | s[2]) != 0;
                if (!queued) {
                    // the end minus the start is the stored move
                    const double Dp[3] = {d1[0] - d[0], d1[1] - d[1], NDIM == 3 ? d1[2] - d[2] : D[2]};
                    if constexpr (IO::kDirect) {
                        segment64<NDIM>(io, plane, q, sx, sxy, d, Dp, sign);
                    } else {
                        if (acc.q != q) {
                            acc.flush(io.M, plane);
                            acc.reset(q);
                        }
                        moments64<NDIM>(d, Dp, sign, acc);
                    }
                }
            }
            sp.u[0][p] = u[0]; sp.u[1][p] = u[1]; sp.u[2][p] = u[2];
        }
        const unsigned m = __ballot_sync(kFull, queued);
        if (queued) {
            const int idx = (qhead + qcount + __popc(m & lt_mask)) & (kQueue64 - 1);
            qc[idx] = make_uint2(q, (unsigned)(s[0] + 1) | (unsigned)(s[1] + 1) << 2 | (unsigned)(s[2] + 1) << 4);
#pragma unroll
            for (int a = 0; a < NDIM; ++a) {
                qv[a][idx] = d[a];
                qv[NDIM + a][idx] = d1[a];
            }
            if (NDIM == 2) qv[4][idx] = D[2];
        }
        qcount += __popc(m);
        if (qcount >= 32) {
            __syncwarp();
            drain_one((qhead + lane) & (kQueue64 - 1));
            __syncwarp();
            qhead = (qhead + 32) & (kQueue64 - 1);
            qcount -= 32;
        }
    }
    __syncwarp();
    if (lane < qcount) drain_one((qhead + lane) & (kQueue64 - 1));
    if constexpr (!IO::kDirect) acc.flush(io.M, plane);
    if (kin_acc) {
        for (int o = 16; o > 0; o >>= 1) {
            if (KIN0) kin0 += __shfl_xor_sync(kFull, kin0, o);
            kin1 += __shfl_xor_sync(kFull, kin1, o);
        }
        if (lane == 0) {
            if (KIN0) atomicAdd(kin_acc, m_over_me * kin0);
            atomicAdd(kin_acc + 1, m_over_me * kin1);
        }
    }
}

// Initial staggering: u^0 -> u^{-dt/2} by one Boris step of -dt/2, no move.
template <int NDIM, class IO>
__global__ void __launch_bounds__(256) k_half_back64(const __grid_constant__ Geom g, const __grid_constant__ IO io,
                                                     Species64 sp, long long n, double qe) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        int c[3] = {0, 0, 0};
        double d[3] = {0, 0, 0}, u[3] = {sp.u[0][p], sp.u[1][p], sp.u[2][p]};
        for (int a = 0; a < NDIM; ++a) split_bits(sp.x[a][p], c[a], d[a]);
        if (g.bcx == 1 && c[0] >= g.nx) { c[0] = g.nx - 1; d[0] = 1.0; }
        double E[3], B[3];
        gather_cell64<NDIM>(g, io, c, (unsigned)g.pidx(c[0], c[1], c[2]), d, E, B);
        boris64(u, E, B, qe);
        sp.u[0][p] = u[0]; sp.u[1][p] = u[1]; sp.u[2][p] = u[2];
    }
}

// Currents from the moments: J(i,j,k) of component c sums, over the four cells that
// touch the edge, the flux the cell's moments give for that edge.  Writes the
// interior of the padded planes J (their ghosts stay zero).  One thread per cell.
template <int NDIM>
__global__ void __launch_bounds__(256) k_current64(Geom g, const double *__restrict__ M, double *J0, double *J1,
                                                   double *J2, double scale) {
    const long long ncell = (long long)g.nx * g.ny * g.nz;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < ncell; t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(t % g.nx);
        const long long r = t / g.nx;
        const int j = (int)(r % g.ny), k = (int)(r / g.ny);
        const int im = i == 0 ? g.nx - 1 : i - 1, jm = j == 0 ? g.ny - 1 : j - 1, km = k == 0 ? g.nz - 1 : k - 1;
        auto m = [&](int v, int a, int b, int c) { return folded_current(g, M + (size_t)v * g.pcells, a, b, c); };
        // four moments at v0: cell itself, its lower neighbour on axis p, on axis q, on both
        auto four = [&](int v0, int pi, int pj, int pk, int qi, int qj, int qk, int bi, int bj, int bk) {
            const double m3 = m(v0 + 3, i, j, k), m1 = m(v0 + 1, i, j, k), m2 = m(v0 + 2, i, j, k);
            return ((m(v0, i, j, k) - m1) - (m2 - m3)) + (m(v0 + 1, pi, pj, pk) - m(v0 + 3, pi, pj, pk)) +
                   (m(v0 + 2, qi, qj, qk) - m(v0 + 3, qi, qj, qk)) + m(v0 + 3, bi, bj, bk);
        };
        double Jx, Jy, Jz;
        if (NDIM == 3) {
            Jx = four(0, i, jm, k, i, j, km, i, jm, km);
            Jy = four(4, im, j, k, i, j, km, im, j, km);
            Jz = four(8, im, j, k, i, jm, k, im, jm, k);
        } else {
            Jx = (m(0, i, j, k) - m(1, i, j, k)) + m(1, i, jm, k);
            Jy = (m(2, i, j, k) - m(3, i, j, k)) + m(3, im, j, k);
            Jz = four(4, im, j, k, i, jm, k, im, jm, k);
        }
        const long long c = g.pidx(i, j, k);
        J0[c] = scale * Jx;
        J1[c] = scale * Jy;
        J2[c] = scale * Jz;
    }
}

}  // namespace

// Particles of a cell-sorted block a lane walks: up to 32 while a warp gets 16 such blocks or more.
int walk_lg64(long long n) {
    int lg = 5;
    while (lg > 0 && (n >> (5 + lg)) < 16 * kWarps64) --lg;
    return lg;
}

namespace {

template <int NDIM, bool WALLS, class IO>
void launch_dim(const Geom &g, const IO &io, Species64 sp, long long n, bool sorted, double h, int sign, double dt,
                double m_over_me, double *kin_acc, bool kin0, int *err, cudaStream_t s) {
    // The pipe is the bound, so every SM gets the same share in one wave of all resident
    // warps, and each warp as many particles as that allows (its last drain is part filled).
    const int lgw = sorted ? walk_lg64(n) : 0;
    const long long nblk = (n + (32LL << lgw) - 1) >> (5 + lgw);
    const int grid = (int)((std::min<long long>(nblk, kWarps64) + kThreads64 / 32 - 1) / (kThreads64 / 32));
    auto k = kin0 ? k_push_fp64<NDIM, WALLS, true, IO> : k_push_fp64<NDIM, WALLS, false, IO>;
    k<<<grid, kThreads64, 0, s>>>(g, io, sp, n, lgw, h, sign, dt, m_over_me, kin_acc, err);
}

template <class IO>
void launch_push(const Geom &g, const IO &io, Species64 sp, long long n, bool sorted, double h, int sign, double dt,
                 double m_over_me, double *kin_acc, bool kin0, int *err, cudaStream_t s) {
    const bool walls = g.bcx == 1;
    auto f = g.ndim == 3 ? (walls ? launch_dim<3, true, IO> : launch_dim<3, false, IO>)
                         : (walls ? launch_dim<2, true, IO> : launch_dim<2, false, IO>);
    f(g, io, sp, n, sorted, h, sign, dt, m_over_me, kin_acc, kin0, err, s);
}

}  // namespace

int moment_planes64(int ndim) { return ndim == 3 ? nmoments<3>() : nmoments<2>(); }

void launch_push_fp64(const Geom &g, const Cells64 &io, Species64 sp, long long n, bool sorted, double h, double alpha,
                      double dt, double m_over_me, double *kin_acc, bool kin0, int *err, cudaStream_t s) {
    if (n <= 0) return;
    const int sign = alpha < 0 ? (int)0x80000000 : 0;
    if (io.nf) launch_push(g, MomentCells64{io.nf, io.M}, sp, n, sorted, h, sign, dt, m_over_me, kin_acc, kin0, err, s);
    else launch_push(g, DirectCells64{io.f, io.J, -alpha}, sp, n, sorted, h, sign, dt, m_over_me, kin_acc, kin0, err, s);
}

void launch_current64(const Geom &g, const double *M, double *const J[3], double alpha_abs, cudaStream_t s) {
    const long long ncell = (long long)g.nx * g.ny * g.nz;
    const int blocks = (int)std::min<long long>((ncell + 255) / 256, 152LL * 16);
    // Ampere's law takes minus alpha times the flux
    if (g.ndim == 3) k_current64<3><<<blocks, 256, 0, s>>>(g, M, J[0], J[1], J[2], -alpha_abs);
    else k_current64<2><<<blocks, 256, 0, s>>>(g, M, J[0], J[1], J[2], -alpha_abs);
}

void launch_half_back64(const Geom &g, const Cells64 &io, Species64 sp, long long n, double h, double dt,
                        cudaStream_t s) {
    if (n <= 0) return;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152LL * 16);
    const double qe = -0.25 * h * dt;
    const MomentCells64 m{io.nf, io.M};
    const DirectCells64 d{io.f, nullptr, 0.0};
    if (g.ndim == 3) {
        if (io.nf) k_half_back64<3><<<blocks, 256, 0, s>>>(g, m, sp, n, qe);
        else k_half_back64<3><<<blocks, 256, 0, s>>>(g, d, sp, n, qe);
    } else {
        if (io.nf) k_half_back64<2><<<blocks, 256, 0, s>>>(g, m, sp, n, qe);
        else k_half_back64<2><<<blocks, 256, 0, s>>>(g, d, sp, n, qe);
    }
}

}  // namespace pic
