// mj_common.cuh -- device parts of the drifting Maxwell-Juttner loader shared
// by the exact sampler (mj.cu) and the learned sampler (mlp.cu): Philox
// streams, the tabulated marginal and its inversion, the conditional of
// Eq. finding_u, and the particle assembly kernel.
#pragma once
#include <cmath>

#include "pic_internal.cuh"

namespace pic {
namespace mjk {

// ---------------------------------------------------------------- Philox-4x32-10

struct U4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ U4 philox_round(U4 c, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    return U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
}

__device__ inline U4 philox4x32_10(U4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        c = philox_round(c, k0, k1);
    }
    return c;
}

__device__ __forceinline__ double to_unit(uint32_t hi, uint32_t lo) {
    const unsigned long long m = ((unsigned long long)(hi >> 5) << 26) + (unsigned long long)(lo >> 6);
    return ((double)m + 0.5) * 0x1p-53;
}

__device__ inline void uniforms6(unsigned long long seed, int species, long long p, double w[6]) {
    const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
    for (int call = 0; call < 3; ++call) {
        const U4 r = philox4x32_10(U4{(uint32_t)(p & 0xFFFFFFFFll), (uint32_t)((unsigned long long)p >> 32),
                                      (uint32_t)call, (uint32_t)species},
                                   k0, k1);
        w[2 * call] = to_unit(r.x, r.y);
        w[2 * call + 1] = to_unit(r.z, r.w);
    }
}

// ---------------------------------------------------------------- marginal in s = asinh(y)

// density of sigma = s - psi, up to the normalisation Z of the table:
// (1 + mu G0 cosh s) cosh s exp(-2 mu sinh^2(sigma/2)),  s = sigma + psi
struct Marg {
    double mu, G0, psi, Z;
    __host__ __device__ double g(double sig) const {
        const double cs = cosh(sig + psi);
        const double sh = sinh(0.5 * sig);
        return (1.0 + mu * G0 * cs) * cs * exp(-2.0 * mu * sh * sh) / Z;
    }
};

// 8-point Gauss-Legendre nodes and weights on [-1, 1]
__host__ __device__ inline double gl_x(int i) {
    const double x[4] = {0.1834346424956498, 0.5255324099163290, 0.7966664774136267, 0.9602898564975363};
    return i < 4 ? -x[3 - i] : x[i - 4];
}
__host__ __device__ inline double gl_w(int i) {
    const double w[4] = {0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};
    return i < 4 ? w[3 - i] : w[i - 4];
}

__host__ __device__ inline double gl_integral(const Marg &m, double a, double b) {
    const double c = 0.5 * (a + b), h = 0.5 * (b - a);
    double s = 0.0;
    for (int i = 0; i < 8; ++i) s += gl_w(i) * m.g(c + h * gl_x(i));
    return s * h;
}

struct Table {
    Marg m;
    double s0, h;       // sigma_k = s0 + k h
    int n;              // intervals
    const double *F;    // n + 1 cumulative values, F[0] = 0, F[n] = 1
    double ep, em, iZ;  // e^psi, e^-psi, 1 / Z
};

__device__ inline double inverse_marginal(const Table &t, double w) {
    int lo = 0, hi = t.n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (t.F[mid] <= w) lo = mid; else hi = mid;
    }
    const double a = t.s0 + lo * t.h;
    const double Fa = t.F[lo], Fb = t.F[lo + 1];
    double sig = a + (Fb > Fa ? (w - Fa) / (Fb - Fa) : 0.5) * t.h;
    for (int it = 0; it < 4; ++it) {
        const double F = Fa + gl_integral(t.m, a, sig);
        const double g = t.m.g(sig);
        if (!(g > 0.0)) break;
        double nxt = sig - (F - w) / g;
        nxt = fmin(fmax(nxt, a), a + t.h);
        sig = nxt;
    }
    return sinh(sig + t.m.psi);
}

// inverse_marginal with about 4 densities instead of 36, and those with two exponentials
// each: sigma starts from the cubic through the four table values around it (off by
// ~(h / width)^4 / 40 intervals), the density over at most one interval is integrated by
// the 4-point rule (relative error 6e-10 (h / width)^8 |g^(8) / g| width^8 < 1e-16 out to
// six widths of the density), and the slope of the cubic, good to (h / width)^3, serves
// for the correction: after one below 1e-8 of the interval the rest is below 1e-15.
// The full inverse is taken where the interval is above 0.06 of the width, at the ends of
// the table and where this does not settle.  Both end within a few roundings of F (in
// units of the density) and of sigma of the root; err is ten times that, for the caller
// that needs the bits (0: they are those of inverse_marginal).
__device__ inline double inverse_marginal_quick(const Table &t, double w, double &err) {
    err = 0.0;
    if (!(t.h * t.h * fmax(t.m.mu, 1.0) <= 0.0036)) return inverse_marginal(t, w);
    int lo = 0, hi = t.n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (t.F[mid] <= w) lo = mid; else hi = mid;
    }
    if (lo == 0 || lo + 2 > t.n) return inverse_marginal(t, w);
    // the cubic F(x) = d1 (x + c2 x (x - 1) + c3 (x^3 - x)) + Fa on the interval 0 <= x <= 1
    const double Fa = t.F[lo], d1 = t.F[lo + 1] - Fa;
    const float inv = 1.f / (float)d1;
    const float e0 = (float)((Fa - t.F[lo - 1]) - d1), e2 = (float)((t.F[lo + 2] - t.F[lo + 1]) - d1);
    const float c2 = -0.5f * e0 * inv, c3 = (e0 + e2) * inv * (1.f / 6.f);
    if (!(fabsf(c2) < 0.25f && fabsf(c3) < 0.1f)) return inverse_marginal(t, w);
    const double r = (w - Fa) / d1;
    float xf = (float)r, slope = 1.f;
    for (int it = 0; it < 3; ++it) {
        slope = 1.f + c2 * (2.f * xf - 1.f) + c3 * (3.f * xf * xf - 1.f);
        if (it < 2) xf -= (xf + (xf - 1.f) * xf * (c2 + c3 * (xf + 1.f)) - (float)r) / slope;
    }
    const double xd = (double)xf;
    const double x = xd - (xd + (xd - 1.0) * xd * ((double)c2 + (double)c3 * (xd + 1.0)) - r) * (double)(1.f / slope);
    const double a = t.s0 + lo * t.h, g = d1 * (double)slope / t.h;
    double sig = fmin(fmax(fma(x, t.h, a), a), a + t.h);
    const double igh = (double)(1.f / (float)g);
    for (int it = 0; it < 4; ++it) {
        const double c = 0.5 * (a + sig), hw = 0.5 * (sig - a);
        double F = 0.0;
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {   // Gauss-Legendre nodes and weights
            const double s = fma((k & 1 ? hw : -hw), (k < 2 ? 0.3399810435848563 : 0.8611363115940526), c);
            const double E = exp(0.5 * s), I = 1.0 / E, sh = 0.5 * (E - I);
            const double cs = 0.5 * (E * E * t.ep + I * I * t.em);
            F += (k < 2 ? 0.6521451548625461 : 0.3478548451374538) *
                 (fma(t.m.mu * t.m.G0, cs, 1.0) * cs * exp(-2.0 * t.m.mu * sh * sh));
        }
        const double step = (Fa + F * hw * t.iZ - w) * igh;
        sig = fmin(fmax(sig - step, a), a + t.h);
        if (fabs(step) <= 1e-8 * t.h) {
            const double y = sinh(sig + t.m.psi);
            err = (4e-15 / g + 1e-14 * (1.0 + fabs(sig) + fabs(t.m.psi))) * sqrt(1.0 + y * y);
            return y;
        }
    }
    return inverse_marginal(t, w);
}

// t = a (u - 1) >= 0 from l(a + t) = w l(a) (Eq. finding_u), written as
// log1p(t / (1 + a)) - t = log w and solved by Newton from t = -log w (the
// large-a limit); the function is concave and decreasing in t, so the steps
// converge monotonically once on the right of the root, and go on until t stands still.
// Where it alternates between two neighbouring doubles, the result is that of the 60th
// step, which follows from the parity.  (Taking those steps, which some lane of nearly
// every warp did, was half of the loader's 52 ms for 4.2M particles; see k_load_mj.)
__device__ inline double conditional_t(double a, double w) {
    const double lw = log(w);
    double t = -lw, before = -1.0;
    for (int it = 0; it < 60; ++it) {
        const double f = log1p(t / (1.0 + a)) - t - lw;
        const double fp = 1.0 / (1.0 + a + t) - 1.0;
        double nt = t - f / fp;
        if (nt < 0.0) nt = 0.5 * t;
        if (nt == before) return (it & 1) ? nt : t;   // step 60 is an even number of steps after nt's, or t's
        const bool done = fabs(nt - t) <= 1e-16 * (nt + 1e-300);
        before = t;
        t = nt;
        if (done) break;
    }
    return t;
}

// The same root with one step in FP64: Newton's in FP32 as far as they go, then Halley's.
// After one of relative size d the error is below 0.6 d^3 of t (with s = 1 / (1 + a + t),
// |f2 t / 2 f1| < 1/2 and |f3 t^2 / 6 f1| = s^2 t^2 / 3 (a + t) < 1/3 for the derivatives
// f1, f2, f3), below rounding for d <= 1e-5.  FP32 gets there unless a and t are small,
// where f cancels.
__device__ inline double conditional_t_quick(double a, double w) {
    const double lw = log(w);
    const float af = 1.f + (float)a, lf = (float)lw;
    float tf = -lf;
    for (int it = 0; it < 12; ++it) {
        const float nt = fmaxf(tf - (log1pf(tf / af) - tf - lf) / (1.f / (af + tf) - 1.f), 0.5f * tf);
        const bool done = fabsf(nt - tf) <= 1e-4f * nt;
        tf = nt;
        if (done) break;
    }
    double t = (double)tf;
    for (int it = 0; it < 4; ++it) {
        const double s = 1.0 / (1.0 + a + t), f1 = s - 1.0;
        const double f = log1p(t / (1.0 + a)) - t - lw;
        const double d = f * f1 / (f1 * f1 + 0.5 * f * s * s);
        t -= d;
        if (fabs(d) <= 1e-5 * t) return t;
    }
    return conditional_t(a, w);
}

struct LoadArgs {
    Geom g;
    int ndim;
    long long n;
    int species;
    unsigned long long seed;
    int profile;
    double L, x0;
    double theta;
    double sb0;                 // drift speed the momenta are sampled with (0 for the naive control)
    double beta0;               // drift speed of the distribution
    double nvec[3], e1[3], e2[3];
    int naive;                  // rest-frame sample boosted particle by particle
    Table tab;
    int colocate;               // positions copied from src_* arrays
    // FP64 destination
    double *x64[3], *u64[3];
    const double *cx64[3];
    // mixed destination
    SpeciesMixed mx;
    SpeciesMixed cmx;
    int mixed;
    int *err;
};

// Drift-component samplers: the exact inverse of the tabulated marginal, or
// the learned network (mlp.cu).
struct ExactPar {
    __device__ void begin() const {}
    // err > 0: a bound on the distance from inverse_marginal's value
    __device__ double operator()(const LoadArgs &a, double w, double &err) const {
        return inverse_marginal_quick(a.tab, w, err);
    }
};

// Par::begin is called by every thread of a block once, and the sampler by whole warps.
template <class Par>
__global__ void __launch_bounds__(256) k_load_mj(LoadArgs a, Par par_of) {
    par_of.begin();
    const int lane = threadIdx.x & 31;
    for (long long p0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; p0 < a.n;
         p0 += (long long)gridDim.x * blockDim.x) {
        const long long p = p0 + lane;
        double w[6];
        uniforms6(a.seed, a.species, p, w);
        // momentum along n and in the orthogonal plane
        double err, y = par_of(a, w[3], err);
        if (p >= a.n) continue;
        const double mu = 1.0 / a.theta;
        const double G0 = 1.0 / sqrt(1.0 - a.sb0 * a.sb0);
        const double Gb = 1.0 / sqrt(1.0 - a.beta0 * a.beta0);
        double sphi, cphi;
        sincospi(2.0 * w[5], &sphi, &cphi);
        double mom[3];
        // FP64 instructions bound the loader: 52 ms for 4.2M particles when every one went through
        // inverse_marginal and the full conditional_t.  Here these follow, once, only where the error
        // of the quick values could change a rounding to FP32 (one particle in about 10^5), so that
        // the FP32 momenta are those of the full ones: 5.9 ms.
        for (bool quick = true;; quick = false) {
            const double gy = sqrt(1.0 + y * y);
            const double aa = mu * G0 * gy;
            const double um1 = (quick ? conditional_t_quick(aa, w[4]) : conditional_t(aa, w[4])) / aa;   // u - 1
            const double r = sqrt(um1 * (um1 + 2.0));
            double par = y, q1 = gy * r * cphi, q2 = gy * r * sphi;
            if (a.naive) {
                // the same sample drawn at rest (its table was built with beta0 = 0), then boosted
                const double g0 = sqrt(1.0 + par * par + q1 * q1 + q2 * q2);
                par = Gb * (par + a.beta0 * g0);
            }
            for (int c = 0; c < 3; ++c) mom[c] = a.nvec[c] * par + a.e1[c] * q1 + a.e2[c] * q2;
            if (!a.mixed || !quick) break;
            const double d = (4.0 * err * (1.0 + r) + 1e-14 * (1.0 + 1.0 / aa) * gy * r) * (a.naive ? 2.0 * Gb : 1.0);
            if ((float)(mom[0] - d) == (float)(mom[0] + d) && (float)(mom[1] - d) == (float)(mom[1] + d) &&
                (float)(mom[2] - d) == (float)(mom[2] + d))
                break;
            if (err > 0.0) y = inverse_marginal(a.tab, w[3]);
        }
        // position
        double pos[3] = {0.0, 0.0, 0.0};
        if (!a.colocate) {
            pos[0] = a.g.nx * w[0];
            pos[1] = a.g.ny * w[1];
            if (a.ndim == 3) pos[2] = a.g.nz * w[2];
            if (a.profile == 1) {
                const double ta = tanh(-a.x0 / a.L), tb = tanh((a.g.nx - a.x0) / a.L);
                pos[0] = a.x0 + a.L * atanh(ta + w[0] * (tb - ta));
                pos[0] = fmin(fmax(pos[0], 0.0), (double)a.g.nx);
            }
        }
        if (!a.mixed) {
            for (int c = 0; c < 3; ++c) {
                if (a.colocate) pos[c] = a.cx64[c][p];
                a.x64[c][p] = pos[c];
                a.u64[c][p] = mom[c];
            }
            if (a.g.bcx == 0 && a.x64[0][p] >= a.g.nx) a.x64[0][p] = 0.0;
            if (a.x64[1][p] >= a.g.ny) a.x64[1][p] = 0.0;
            if (a.ndim == 3 && a.x64[2][p] >= a.g.nz) a.x64[2][p] = 0.0;
        } else {
            const float um[3] = {(float)mom[0], (float)mom[1], (float)mom[2]};
            float of[3] = {0.f, 0.f, 0.f};
            uint32_t cell;
            if (a.colocate) {
                float uc[3];
                cell = get_particle(a.ndim, a.cmx, p, of, uc);
            } else {
                int ci[3] = {0, 0, 0};
                const int n3[3] = {a.g.nx, a.g.ny, a.g.nz};
                for (int c = 0; c < a.ndim; ++c) {
                    const double f = floor(pos[c]);
                    int k = (int)f;
                    // the offset on the 2^-24 grid of the mixed path (see snap_offset)
                    float o = (float)(rint((pos[c] - f) * 16777216.0) * (1.0 / 16777216.0));
                    if (o >= 1.0f) { o = 0.0f; k += 1; }
                    if (c == 0 && a.g.bcx == 1 && k >= n3[0]) { k = n3[0] - 1; o = 1.0f; }
                    else if (k >= n3[c]) k -= n3[c];
                    ci[c] = k;
                    of[c] = o;
                }
                cell = pack_cell(a.ndim, ci[0], ci[1], ci[2]);
            }
            put_particle(a.ndim, a.mx, p, cell, of, um, __int_as_float((int)p));
            if (a.ndim == 2) a.mx.id[p] = (int32_t)p;
        }
    }
}

inline LoadArgs make_load_args(const Geom &g, int ndim, long long n, int species, unsigned long long seed, int profile,
                               double L, double x0, double theta, const double beta[3], int naive, const double *Fdev,
                               double s0, double h, int ntab, double psi, double Z, int colocate, Species64 d64,
                               Species64 c64, SpeciesMixed dmx, SpeciesMixed cmx, int mixed, int *err) {
    LoadArgs a{};
    a.g = g;
    a.ndim = ndim;
    a.n = n;
    a.species = species;
    a.seed = seed;
    a.profile = profile;
    a.L = L;
    a.x0 = x0;
    a.theta = theta;
    const double b0 = std::sqrt(beta[0] * beta[0] + beta[1] * beta[1] + beta[2] * beta[2]);
    a.beta0 = b0;
    a.sb0 = naive ? 0.0 : b0;
    double nv[3] = {0.0, 0.0, 1.0};
    if (b0 > 0) for (int c = 0; c < 3; ++c) nv[c] = beta[c] / b0;
    double av[3] = {1.0, 0.0, 0.0};
    if (!(std::fabs(nv[0]) < 0.9)) { av[0] = 0.0; av[1] = 1.0; }
    const double dot = av[0] * nv[0] + av[1] * nv[1] + av[2] * nv[2];
    double e1[3] = {av[0] - dot * nv[0], av[1] - dot * nv[1], av[2] - dot * nv[2]};
    const double ne = std::sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
    for (int c = 0; c < 3; ++c) e1[c] /= ne;
    const double e2[3] = {nv[1] * e1[2] - nv[2] * e1[1], nv[2] * e1[0] - nv[0] * e1[2], nv[0] * e1[1] - nv[1] * e1[0]};
    for (int c = 0; c < 3; ++c) { a.nvec[c] = nv[c]; a.e1[c] = e1[c]; a.e2[c] = e2[c]; }
    a.naive = naive;
    const double mu = 1.0 / theta;
    const double G0 = naive ? 1.0 : 1.0 / std::sqrt(1.0 - b0 * b0);
    a.tab.m = Marg{mu, G0, psi, Z};
    a.tab.s0 = s0;
    a.tab.h = h;
    a.tab.n = ntab;
    a.tab.F = Fdev;
    a.tab.ep = std::exp(psi);
    a.tab.em = std::exp(-psi);
    a.tab.iZ = 1.0 / Z;
    a.colocate = colocate;
    for (int c = 0; c < 3; ++c) {
        a.x64[c] = d64.x[c];
        a.u64[c] = d64.u[c];
        a.cx64[c] = c64.x[c];
    }
    a.mx = dmx;
    a.cmx = cmx;
    a.mixed = mixed;
    a.err = err;
    return a;
}


}  // namespace mjk
}  // namespace pic
