// mlp.cu -- learned inverse cumulative distribution of the drift component of
// a drifting Maxwell-Juttner distribution, used by the loader as method
// PIC_MJ_MLP in place of the table inversion of App. D.
//
// Network: 3 -> 64 -> 64 -> 64 -> 1, tanh on the hidden layers, linear output.
// Inputs  x0 = (log10 theta + 0.5) / 1.5,  x1 = 2 beta0 / 0.95 - 1,
//         x2 = probit(w) / 3   (w the uniform of the marginal, Eq. distr_y);
// output  o, and s = asinh(p_par) = psi + asinh(sqrt(theta)) o, psi = atanh(beta0).
// Parameters, flat FP32: W1[64][3] b1[64] W2[64][64] b2[64] W3[64][64] b3[64] W4[64] b4.
//
// Training, FP32 on the GPU: every step draws a fresh batch from the exact
// loader (table + Newton inversion on a 16 x 12 grid of (theta, beta0)),
// runs one fused forward + backward kernel (one thread per sample,
// activations and deltas in shared memory, per-CTA weight gradients reduced
// in shared memory and added once to global memory) and one Adam step.
// Inference: FP16 weights and activations, FP32 accumulation, 32 samples per warp
// with the two 64 x 64 layers on the tensor cores.
#include <algorithm>
#include <cmath>
#include <vector>

#include <cuda_fp16.h>

#include "mj_common.cuh"

namespace pic {

namespace {

constexpr int H = 64;
constexpr int OW1 = 0, OB1 = OW1 + H * 3, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + H * H,
              OW4 = OB3 + H, OB4 = OW4 + H;
constexpr int NP = OB4 + 1;
static_assert(NP == kMlpParams, "parameter count");
constexpr int kT = 128;          // training threads per CTA, one sample each
constexpr int kS = kT + 1;       // padded row of the feature-major activations

// smem: weights | a1 a2 a3 dA dB [H][kS] | d4 [kT]
__global__ void __launch_bounds__(kT) k_mlp_fwd_bwd(const float *__restrict__ W, const float *__restrict__ X,
                                                    const float *__restrict__ T, int n, float *grad, double *loss) {
    extern __shared__ float sm[];
    float *w = sm;
    float *a1 = w + NP + 3;
    float *a2 = a1 + H * kS;
    float *a3 = a2 + H * kS;
    float *dA = a3 + H * kS;
    float *dB = dA + H * kS;
    float *d4s = dB + H * kS;
    float *xs = d4s + kT;            // [3][kT]
    for (int q = threadIdx.x; q < NP; q += kT) w[q] = W[q];
    const int t = threadIdx.x;
    const int idx = blockIdx.x * kT + t;
    const bool valid = idx < n;
    float x0 = 0.f, x1 = 0.f, x2 = 0.f, target = 0.f;
    if (valid) {
        x0 = X[idx]; x1 = X[n + idx]; x2 = X[2 * n + idx];
        target = T[idx];
    }
    xs[t] = x0; xs[kT + t] = x1; xs[2 * kT + t] = x2;
    __syncthreads();
    // forward: each thread owns column t of the activations
    for (int j = 0; j < H; ++j)
        a1[j * kS + t] = tanhf(w[OB1 + j] + w[OW1 + 3 * j] * x0 + w[OW1 + 3 * j + 1] * x1 + w[OW1 + 3 * j + 2] * x2);
    for (int j = 0; j < H; ++j) {
        float v = w[OB2 + j];
        for (int i = 0; i < H; ++i) v += w[OW2 + H * j + i] * a1[i * kS + t];
        a2[j * kS + t] = tanhf(v);
    }
    float o = w[OB4];
    for (int j = 0; j < H; ++j) {
        float v = w[OB3 + j];
        for (int i = 0; i < H; ++i) v += w[OW3 + H * j + i] * a2[i * kS + t];
        const float a = tanhf(v);
        a3[j * kS + t] = a;
        o += w[OW4 + j] * a;
    }
    // loss = mean over the batch of (o - target)^2; backward
    const float e = valid ? (o - target) : 0.f;
    const float d4 = valid ? 2.f * e / (float)n : 0.f;
    d4s[t] = d4;
    for (int j = 0; j < H; ++j) {
        const float a = a3[j * kS + t];
        dA[j * kS + t] = d4 * w[OW4 + j] * (1.f - a * a);     // layer-3 pre-activation deltas
    }
    for (int i = 0; i < H; ++i) {
        float v = 0.f;
        for (int j = 0; j < H; ++j) v += w[OW3 + H * j + i] * dA[j * kS + t];
        const float a = a2[i * kS + t];
        dB[i * kS + t] = v * (1.f - a * a);                   // layer-2 deltas
    }
    __syncthreads();
    // W3, W2 gradients: sums over the CTA's samples
    for (int q = t; q < H * H; q += kT) {
        const int j = q / H, i = q % H;
        float g3 = 0.f, g2 = 0.f;
        for (int s = 0; s < kT; ++s) {
            g3 += dA[j * kS + s] * a2[i * kS + s];
            g2 += dB[j * kS + s] * a1[i * kS + s];
        }
        atomicAdd(grad + OW3 + q, g3);
        atomicAdd(grad + OW2 + q, g2);
    }
    if (t < H) {
        float gb3 = 0.f, gb2 = 0.f, gw4 = 0.f;
        for (int s = 0; s < kT; ++s) {
            gb3 += dA[t * kS + s];
            gb2 += dB[t * kS + s];
            gw4 += d4s[s] * a3[t * kS + s];
        }
        atomicAdd(grad + OB3 + t, gb3);
        atomicAdd(grad + OB2 + t, gb2);
        atomicAdd(grad + OW4 + t, gw4);
    }
    if (t == 0) {
        float g = 0.f;
        for (int s = 0; s < kT; ++s) g += d4s[s];
        atomicAdd(grad + OB4, g);
    }
    __syncthreads();
    // layer-1 deltas (dA is free again)
    for (int i = 0; i < H; ++i) {
        float v = 0.f;
        for (int j = 0; j < H; ++j) v += w[OW2 + H * j + i] * dB[j * kS + t];
        const float a = a1[i * kS + t];
        dA[i * kS + t] = v * (1.f - a * a);
    }
    __syncthreads();
    if (t < H) {
        float gb1 = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
        for (int s = 0; s < kT; ++s) {
            const float dl = dA[t * kS + s];
            gb1 += dl;
            g0 += dl * xs[s];
            g1 += dl * xs[kT + s];
            g2 += dl * xs[2 * kT + s];
        }
        atomicAdd(grad + OB1 + t, gb1);
        atomicAdd(grad + OW1 + 3 * t, g0);
        atomicAdd(grad + OW1 + 3 * t + 1, g1);
        atomicAdd(grad + OW1 + 3 * t + 2, g2);
    }
    double l = (double)e * (double)e;
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if ((t & 31) == 0) atomicAdd(loss, l / (double)n);
}

// Adam (Kingma and Ba 2015) with bias correction; zeroes the gradient.
__global__ void k_adam(float *W, float *g, float *m, float *v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        W[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
        g[q] = 0.f;
    }
}

__global__ void k_to_half(const float *W, __half *Wh, int n) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) Wh[q] = __float2half_rn(W[q]);
}

// ---- inference: FP16 weights and activations, FP32 accumulation ----
//
// A warp evaluates 32 samples, one per lane.  The hidden layers are products of the
// 32 x 64 activations with 64 x 64 weights: two m16 tiles of mma.m16n8k16, whose
// accumulator layout is that of the next layer's left operand, so activations stay
// in registers.  (A 64-wide layer is far too small for a tcgen05 tile, and the 192
// tanh of a sample bound the kernel, not the products.)  4.2M drift components with
// their FP64 features: one thread per sample with scalar multiply-adds 10.4 ms, this
// form 1.65 ms.

constexpr int kWS = 72;   // row stride of the staged weights (halves): the 8 rows of a fragment load hit distinct banks
struct MlpShared {
    __half w[2][H * kWS];
    float w1[H * 3], b1[H], b[2][H], w4[H], b4;
};
__device__ __forceinline__ MlpShared &mlp_shared() {
    __shared__ MlpShared sh;
    return sh;
}

// Stage the weights of the block (all threads; ends with a barrier).
__device__ inline void mlp_stage(const __half *__restrict__ W) {
    MlpShared &S = mlp_shared();
    for (int q = threadIdx.x; q < H * H; q += blockDim.x) {
        S.w[0][(q / H) * kWS + q % H] = W[OW2 + q];
        S.w[1][(q / H) * kWS + q % H] = W[OW3 + q];
    }
    for (int q = threadIdx.x; q < H * 3; q += blockDim.x) S.w1[q] = __half2float(W[OW1 + q]);
    for (int q = threadIdx.x; q < H; q += blockDim.x) {
        S.b1[q] = __half2float(W[OB1 + q]);
        S.b[0][q] = __half2float(W[OB2 + q]);
        S.b[1][q] = __half2float(W[OB3 + q]);
        S.w4[q] = __half2float(W[OW4 + q]);
    }
    if (threadIdx.x == 0) S.b4 = __half2float(W[OB4]);
    __syncthreads();
}

__device__ __forceinline__ uint32_t half_pair(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Network output of the lane's sample; all 32 lanes call it together after mlp_stage.
__device__ inline float mlp_eval_warp(float x0, float x1, float x2) {
    const MlpShared &S = mlp_shared();
    const int lane = threadIdx.x & 31, gr = lane >> 2, tg = lane & 3;
    // left operands: tile m holds samples 16 m + {gr, gr + 8}, columns 16 kt + 2 tg + {0, 1, 8, 9}
    uint32_t act[2][4][4];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        float x[2][3];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int src = 16 * m + gr + 8 * r;
            x[r][0] = __shfl_sync(0xffffffffu, x0, src);
            x[r][1] = __shfl_sync(0xffffffffu, x1, src);
            x[r][2] = __shfl_sync(0xffffffffu, x2, src);
        }
#pragma unroll
        for (int kt = 0; kt < 4; ++kt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {   // register q: row gr + 8 (q & 1), columns + 8 (q >> 1)
                const int j = 16 * kt + 2 * tg + 8 * (q >> 1);
                float v[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float *w = S.w1 + 3 * (j + e), *xr = x[q & 1];
                    v[e] = tanhf(S.b1[j + e] + w[0] * xr[0] + w[1] * xr[1] + w[2] * xr[2]);
                }
                act[m][kt][q] = half_pair(v[0], v[1]);
            }
    }
    float o[2][2] = {{0.f, 0.f}, {0.f, 0.f}};   // output sums of rows gr, gr + 8 of each tile (this lane's columns)
#pragma unroll
    for (int layer = 0; layer < 2; ++layer) {
        uint32_t next[2][4][4];
        const __half *w = S.w[layer];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int j = 8 * nt + 2 * tg;
            const float b0 = S.b[layer][j], b1 = S.b[layer][j + 1];
            float c[2][4] = {{b0, b1, b0, b1}, {b0, b1, b0, b1}};
#pragma unroll
            for (int kt = 0; kt < 4; ++kt) {
                const uint32_t *f = reinterpret_cast<const uint32_t *>(w + (8 * nt + gr) * kWS + 16 * kt + 2 * tg);
                const uint32_t f0 = f[0], f1 = f[4];
#pragma unroll
                for (int m = 0; m < 2; ++m) mma16816(c[m], act[m][kt], f0, f1);
            }
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const uint32_t h = half_pair(tanhf(c[m][2 * r]), tanhf(c[m][2 * r + 1]));
                    next[m][nt >> 1][r + 2 * (nt & 1)] = h;
                    if (layer == 1) {
                        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&h));
                        o[m][r] += S.w4[j] * a.x + S.w4[j + 1] * a.y;
                    }
                }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int kt = 0; kt < 4; ++kt)
#pragma unroll
                for (int q = 0; q < 4; ++q) act[m][kt][q] = next[m][kt][q];
    }
    // sums over the quad's columns, then every lane takes its own sample's
    float mine = 0.f;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float v = o[m][r];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            v = __shfl_sync(0xffffffffu, v, 4 * (lane & 7));
            if (lane >> 3 == 2 * m + r) mine = v;
        }
    return S.b4 + mine;
}

__device__ __forceinline__ void features(double theta, double beta0, double w, float &x0, float &x1, float &x2) {
    x0 = (float)((log10(theta) + 0.5) / 1.5);
    x1 = (float)(2.0 * beta0 / 0.95 - 1.0);
    x2 = (float)(normcdfinv(w) / 3.0);
}

// (loops over whole warps: the evaluation is a warp's)
__global__ void __launch_bounds__(256) k_mlp_infer(const __half *Wg, const float *X, int n, float *out) {
    mlp_stage(Wg);
    const int lane = threadIdx.x & 31;
    for (int i0 = blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < n; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + lane;
        const bool in = i < n;
        const float o = mlp_eval_warp(in ? X[i] : 0.f, in ? X[n + i] : 0.f, in ? X[2 * n + i] : 0.f);
        if (in) out[i] = o;
    }
}

// Training batch from the exact sampler: a random grid point (theta_k, beta_j)
// and a uniform w per sample, the exact drift component s, and the network
// target o = (s - psi) / asinh(sqrt(theta)).
struct TabSet {
    const double *F;         // ncombo x (kMjTable + 1)
    const double *par;       // ncombo x 8: mu, G0, psi, Z, s0, h, theta, beta0
    int ncombo;
};

__global__ void k_mlp_data(TabSet ts, unsigned long long seed, long long base, int n, float *X, float *T) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double u[6];
        mjk::uniforms6(seed, 7, base + i, u);
        const int k = min((int)(u[0] * ts.ncombo), ts.ncombo - 1);
        const double *p = ts.par + 8 * k;
        mjk::Table tb;
        tb.m = mjk::Marg{p[0], p[1], p[2], p[3]};
        tb.s0 = p[4];
        tb.h = p[5];
        tb.n = kMjTable;
        tb.F = ts.F + (size_t)k * (kMjTable + 1);
        const double w = fmin(fmax(u[1], 1e-7), 1.0 - 1e-7);
        const double y = mjk::inverse_marginal(tb, w);
        const double s = asinh(y);
        float x0, x1, x2;
        features(p[6], p[7], w, x0, x1, x2);
        X[i] = x0; X[n + i] = x1; X[2 * n + i] = x2;
        T[i] = (float)((s - p[2]) / asinh(sqrt(p[6])));
    }
}

// Drift component from the network, for the loader (a whole warp calls it together).
struct MlpPar {
    const __half *w;
    double psi, scale;
    __device__ void begin() const { mlp_stage(w); }
    __device__ double operator()(const mjk::LoadArgs &a, double wv, double &err) const {
        err = 0.0;
        const double wc = fmin(fmax(wv, 1e-7), 1.0 - 1e-7);
        float x0, x1, x2;
        features(a.theta, a.beta0, wc, x0, x1, x2);
        const float o = mlp_eval_warp(x0, x1, x2);
        return sinh(psi + scale * (double)o);
    }
};

// Drift component of given uniforms, exact or learned (tests and the gain measurement):
// both as the loader draws it.
__global__ void __launch_bounds__(256) k_sample_par(mjk::Table tb, MlpPar mp, int use_mlp, double theta, double beta0,
                                                    const double *wv, int n, double *y) {
    mjk::LoadArgs a{};
    a.theta = theta;
    a.beta0 = beta0;
    a.tab = tb;
    if (use_mlp) mp.begin();
    const int lane = threadIdx.x & 31;
    for (int i0 = blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < n; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + lane;
        const double w = i < n ? wv[i] : 0.5;
        double err;
        const double r = use_mlp ? mp(a, w, err) : mjk::ExactPar()(a, w, err);
        if (i < n) y[i] = r;
    }
}

}  // namespace

size_t mlp_train_smem() { return sizeof(float) * (NP + 3 + 5 * H * kS + 4 * kT); }

void launch_mlp_fwd_bwd(const float *W, const float *X, const float *T, int n, float *grad, double *loss,
                        cudaStream_t s) {
    const size_t smem = mlp_train_smem();
    cudaFuncSetAttribute(k_mlp_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_mlp_fwd_bwd<<<(n + kT - 1) / kT, kT, smem, s>>>(W, X, T, n, grad, loss);
}

void launch_adam(float *W, float *g, float *m, float *v, int step, float lr, cudaStream_t s) {
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<(NP + 255) / 256, 256, 0, s>>>(W, g, m, v, NP, lr, b1, b2, 1e-8f, c1, c2);
}

void launch_mlp_to_half(const float *W, void *Wh, cudaStream_t s) {
    k_to_half<<<(NP + 255) / 256, 256, 0, s>>>(W, (__half *)Wh, NP);
}

void launch_mlp_infer(const void *Wh, const float *X, int n, float *out, cudaStream_t s) {
    if (n <= 0) return;
    const int blocks = std::min((n + 255) / 256, 152 * 8);
    k_mlp_infer<<<blocks, 256, 0, s>>>((const __half *)Wh, X, n, out);
}

void launch_mlp_data(const double *F, const double *par, int ncombo, unsigned long long seed, long long base, int n,
                     float *X, float *T, cudaStream_t s) {
    TabSet ts{F, par, ncombo};
    const int blocks = std::min((n + 255) / 256, 152 * 8);
    k_mlp_data<<<blocks, 256, 0, s>>>(ts, seed, base, n, X, T);
}

void launch_sample_par(const double *F, double s0, double h, double psi, double Z, const void *Wh, int use_mlp,
                       double theta, double beta0, const double *w, int n, double *y, cudaStream_t s) {
    mjk::Table tb;
    const double mu = 1.0 / theta;
    const double G0 = 1.0 / std::sqrt(1.0 - beta0 * beta0);
    tb.m = mjk::Marg{mu, G0, psi, Z};
    tb.s0 = s0;
    tb.h = h;
    tb.n = kMjTable;
    tb.F = F;
    tb.ep = std::exp(psi);
    tb.em = std::exp(-psi);
    tb.iZ = 1.0 / Z;
    MlpPar mp{(const __half *)Wh, std::atanh(beta0), std::asinh(std::sqrt(theta))};
    const int blocks = std::max(1, std::min((n + 255) / 256, 152 * 16));
    k_sample_par<<<blocks, 256, 0, s>>>(tb, mp, use_mlp, theta, beta0, w, n, y);
}

void launch_load_mj_mlp(const Geom &g, int ndim, long long n, int species, unsigned long long seed, int profile,
                        double L, double x0, double theta, const double beta[3], const void *Wh, int colocate,
                        Species64 d64, Species64 c64, SpeciesMixed dmx, SpeciesMixed cmx, int mixed, int *err,
                        cudaStream_t s) {
    mjk::LoadArgs a = mjk::make_load_args(g, ndim, n, species, seed, profile, L, x0, theta, beta, 0, nullptr, 0.0, 0.0,
                                          0, 0.0, 1.0, colocate, d64, c64, dmx, cmx, mixed, err);
    MlpPar mp{(const __half *)Wh, std::atanh(a.beta0), std::asinh(std::sqrt(theta))};
    if (n <= 0) return;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152LL * 16);
    mjk::k_load_mj<MlpPar><<<blocks, 256, 0, s>>>(a, mp);
}

}  // namespace pic
