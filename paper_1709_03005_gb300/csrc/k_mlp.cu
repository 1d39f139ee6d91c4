// Learned Davidson preconditioner: a small MLP that scales the diagonal
// correction row by row (not in the paper; plain diagonal Davidson remains the
// fallback and the reference).
//
//   t_i = w(f_i) r_i / (H_ii - theta),   w = 256^tanh(o),   o = MLP(f)
//   MLP: h1 = relu(W1 f + b1), h2 = relu(W2 h1 + b2), o = w3 . h2 + b3
// with n_in = 8 features, width 64, weights rounded to FP16 in the forward
// pass (inference stores them as FP16) and FP32 accumulation.
//
// Features of row i for a Ritz value theta (all divided by 10 Eh except f1):
//   f0 = (H_ii - theta), f1 = log(|H_ii - theta| + 1e-3), f2 = 1 for an L2 row,
//   f3 = E_n - theta for a continuum row of target state n (0 for L2),
//   f4 = h_jj of its continuum orbital (0 for L2), f5 = theta - theta_0,
//   f6 = H_ii, f7 = group index / number of groups (1 for L2).
// The range [1/256, 256] lets the factor damp rows whose H_ii - theta is small
// by two orders of magnitude (a shifted denominator |d| / (|d| + delta) does
// that, and a floor of 1/4 loses its gain).  Training minimises
// sum_i (w(f_i) a_i - b_i)^2 for given targets a, b (a = 1 and b a wanted
// factor fits the factor itself); the gradient is taken by a hand-written backward
// pass whose sums run in a fixed order.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "hb_davidson.cuh"

namespace hb {

constexpr int MLP_IN = 8, MLP_W = 64;
constexpr int MLP_NPARAM = MLP_W * MLP_IN + MLP_W + MLP_W * MLP_W + MLP_W + MLP_W + 1;   // 4801

struct MlpState {
    __half *wh = nullptr;        // FP16 weights (packed like the parameters)
    float *bias = nullptr;       // FP32 copy of every parameter (biases read from here)
    float *row_info = nullptr;   // [4][n]: type, E_n, h_jj, group/n_groups
    float *w = nullptr;          // [mmax][n] factors for the current iteration
    float *feats = nullptr;      // scratch features
    int64_t n = 0;
    int mmax = 0;
    bool rows_ready = false;
};

}  // namespace hb

using namespace hb;

namespace {

constexpr float kLogR = 5.545177444479562f;   // log 256: w in [1/256, 256]

// offsets inside the packed parameter vector
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_W * MLP_IN, OFF_W2 = OFF_B1 + MLP_W, OFF_B2 = OFF_W2 + MLP_W * MLP_W,
              OFF_W3 = OFF_B2 + MLP_W, OFF_B3 = OFF_W3 + MLP_W;

__device__ __forceinline__ float q16(float x) { return __half2float(__float2half_rn(x)); }

// row features for one (row, theta)
__device__ __forceinline__ void features(float d, float theta, float theta0, const float *ri, int64_t i, int64_t n,
                                         float (&f)[MLP_IN]) {
    const float type = ri[i], En = ri[n + i], hj = ri[2 * n + i], gid = ri[3 * n + i];
    const float gap = d - theta;
    f[0] = gap * 0.1f;
    f[1] = logf(fabsf(gap) + 1e-3f);
    f[2] = type;
    f[3] = type > 0.5f ? 0.0f : (En - theta) * 0.1f;
    f[4] = hj * 0.1f;
    f[5] = (theta - theta0) * 0.1f;
    f[6] = d * 0.1f;
    f[7] = gid;
}

// forward pass with weights from shared memory; returns o, fills h1, h2
__device__ __forceinline__ float mlp_forward(const float *P, const float (&f)[MLP_IN], float (&h1)[MLP_W],
                                             float (&h2)[MLP_W]) {
#pragma unroll 4
    for (int a = 0; a < MLP_W; ++a) {
        float s = P[OFF_B1 + a];
#pragma unroll
        for (int c = 0; c < MLP_IN; ++c) s = fmaf(P[OFF_W1 + a * MLP_IN + c], f[c], s);
        h1[a] = fmaxf(s, 0.0f);
    }
#pragma unroll 2
    for (int a = 0; a < MLP_W; ++a) {
        float s = P[OFF_B2 + a];
#pragma unroll
        for (int c = 0; c < MLP_W; ++c) s = fmaf(P[OFF_W2 + a * MLP_W + c], h1[c], s);
        h2[a] = fmaxf(s, 0.0f);
    }
    float o = P[OFF_B3];
#pragma unroll
    for (int c = 0; c < MLP_W; ++c) o = fmaf(P[OFF_W3 + c], h2[c], o);
    return o;
}

// stage the parameters (weights rounded to FP16) in shared memory
__device__ __forceinline__ void stage_params(const float *params, float *P) {
    for (int t = threadIdx.x; t < MLP_NPARAM; t += blockDim.x) {
        const bool is_bias = (t >= OFF_B1 && t < OFF_W2) || (t >= OFF_B2 && t < OFF_W3) || t == OFF_B3;
        P[t] = is_bias ? params[t] : q16(params[t]);
    }
    __syncthreads();
}

// ---------------------------------------------------------------- training
// Loss and gradient in one persistent kernel.  A block takes tiles of kTile
// samples and keeps everything of a tile in shared memory: activations and
// deltas as [unit][sample] (row stride kLd, 4 mod 32 banks, so that the 128-bit
// reads of eight consecutive rows hit different banks).  The three 64 x 64
// products of a sample (forward, input gradient, weight gradient) are register
// tiles (8 samples x 4 units, or 4 x 4 weights), so the kernel runs on the FP32
// pipe: 8.7 kFMA a sample, 23 us for 65536 samples at the full rate.  The
// gradient sums stay in registers over all tiles of a block, in two levels: those
// of kFold tiles (1024 samples), then the sum of these, so that the chain of FP32
// additions does not grow with the window; each block then writes one row of
// partial sums, and a second kernel adds the rows in order.
// Measured at 65536 samples: 76 us + 6 us, against 172 + 2375 us when the
// activations went through memory and each parameter walked the samples alone.
constexpr int kTile = 128, kLd = kTile + 4, kTrainThreads = 256, kFold = 8;
constexpr int kTrainSmem = (3 * MLP_W * kLd + MLP_IN * kLd + 2 * MLP_W * MLP_W + MLP_W * MLP_IN + 3 * MLP_W + 2 * kTile) *
                           (int)sizeof(float);

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// A thread's eight samples are s0 .. s0 + 3 and s0 + 64 .. s0 + 67, so that the
// 16 threads of a unit group read and write whole rows without bank conflicts.
constexpr int kHalf = kTile / 2;

__device__ __forceinline__ void put8(float *row, int s0, const float (&v)[8]) {
    *reinterpret_cast<float4 *>(row + s0) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(row + s0 + kHalf) = make_float4(v[4], v[5], v[6], v[7]);
}

__device__ __forceinline__ void get8(const float *row, int s0, float (&v)[8]) {
    const float4 x = ld4(row + s0), y = ld4(row + s0 + kHalf);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
}

// acc[j][i] += sum_k A[k][sample i] B[k][u0 + j] over k < 64 (4 units x 8 samples)
__device__ __forceinline__ void tile_product(const float *A, const float *B, int s0, int u0, float (&acc)[4][8]) {
#pragma unroll 4
    for (int k = 0; k < MLP_W; ++k) {
        float a[8];
        get8(A + k * kLd, s0, a);
        const float4 w = ld4(B + k * MLP_W + u0);
        const float b[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[j][i] = fmaf(a[i], b[j], acc[j][i]);
    }
}

__global__ void __launch_bounds__(kTrainThreads, 1)
mlp_train_kernel(const float *__restrict__ params, const float *__restrict__ feats, const float *__restrict__ ta,
                 const float *__restrict__ tb, int64_t n, int64_t tiles, float *__restrict__ partial) {
    extern __shared__ __align__(16) float sm[];
    float *H1 = sm, *H2 = H1 + MLP_W * kLd, *D1 = H2 + MLP_W * kLd, *F = D1 + MLP_W * kLd;
    float *W2 = F + MLP_IN * kLd, *W2T = W2 + MLP_W * MLP_W, *W1 = W2T + MLP_W * MLP_W;
    float *B1 = W1 + MLP_W * MLP_IN, *B2 = B1 + MLP_W, *W3 = B2 + MLP_W, *DO = W3 + MLP_W, *ER = DO + kTile;
    const int t = threadIdx.x;
    for (int e = t; e < MLP_W * MLP_W; e += kTrainThreads) {
        const float v = q16(params[OFF_W2 + e]);
        W2[e] = v;
        W2T[(e % MLP_W) * MLP_W + e / MLP_W] = v;
    }
    for (int e = t; e < MLP_W * MLP_IN; e += kTrainThreads) W1[e] = q16(params[OFF_W1 + e]);
    if (t < MLP_W) {
        B1[t] = params[OFF_B1 + t];
        B2[t] = params[OFF_B2 + t];
        W3[t] = q16(params[OFF_W3 + t]);
    }
    const float b3 = params[OFF_B3];
    // register tile of the sample products: 16 unit groups x 16 sample groups
    const int u0 = 4 * (t / 16), s0 = 4 * (t % 16);
    // gradient sums of this thread: W2[ga + 16 i][gc + 16 j]; W1[wa][wc, wc + 1];
    // b1, b2, w3 of unit wa over samples 32 (t % 4) ..; b3 and the loss on thread t < kTile
    const int ga = t / 16, gc = t % 16, wa = t / 4, wq = t % 4;
    float g2[4][4] = {}, g1[2] = {0.0f, 0.0f}, gb1 = 0.0f, gb2 = 0.0f, gw3 = 0.0f, gb3 = 0.0f, gl = 0.0f;
    // and those of the tiles folded so far (b3 and the loss take one sample a tile and thread)
    float s2[4][4] = {}, s1[2] = {0.0f, 0.0f}, sb1 = 0.0f, sb2 = 0.0f, sw3 = 0.0f;
    auto fold = [&](float &s, float &g) {
        s += g;
        g = 0.0f;
    };
    auto fold_all = [&] {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) fold(s2[i][j], g2[i][j]);
        fold(s1[0], g1[0]);
        fold(s1[1], g1[1]);
        fold(sb1, gb1);
        fold(sb2, gb2);
        fold(sw3, gw3);
    };
    int held = 0;                              // tiles in the first level
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (held == kFold) {
            fold_all();
            held = 0;
        }
        ++held;
        const int64_t i0 = tile * kTile;
        const int valid = (int)min((int64_t)kTile, n - i0);
        __syncthreads();
        for (int e = t; e < kTile * MLP_IN; e += kTrainThreads) {
            const int s = e / MLP_IN, c = e % MLP_IN;
            F[c * kLd + s] = s < valid ? feats[i0 * MLP_IN + e] : 0.0f;
        }
        __syncthreads();
        {
            float acc[4][8];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[j][i] = B1[u0 + j];
#pragma unroll
            for (int c = 0; c < MLP_IN; ++c) {
                float f[8];
                get8(F + c * kLd, s0, f);
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[j][i] = fmaf(W1[(u0 + j) * MLP_IN + c], f[i], acc[j][i]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[j][i] = fmaxf(acc[j][i], 0.0f);
                put8(H1 + (u0 + j) * kLd, s0, acc[j]);
            }
        }
        __syncthreads();
        {
            float acc[4][8];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[j][i] = B2[u0 + j];
            tile_product(H1, W2T, s0, u0, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[j][i] = fmaxf(acc[j][i], 0.0f);
                put8(H2 + (u0 + j) * kLd, s0, acc[j]);
            }
        }
        __syncthreads();
        if (t < kTile) {
            float o = b3;
#pragma unroll 8
            for (int c = 0; c < MLP_W; ++c) o = fmaf(W3[c], H2[c * kLd + t], o);
            float dout = 0.0f;
            if (t < valid) {
                const float th = tanhf(o);
                const float w = expf(kLogR * th);
                const float a = ta[i0 + t], b = tb[i0 + t];
                const float err = w * a - b;
                gl = fmaf(err, err, gl);
                dout = 2.0f * err * a * w * kLogR * (1.0f - th * th);   // dL/do
                gb3 += dout;
            }
            DO[t] = dout;
        }
        __syncthreads();
        // w3's sums, and H2 becomes D2 in place
        {
            const float w3 = W3[wa];
#pragma unroll 4
            for (int k = 0; k < 8; ++k) {
                const int s = 4 * (wq + 4 * k);
                float4 h = ld4(H2 + wa * kLd + s);
                const float4 d = ld4(DO + s);
                gw3 = fmaf(d.x, h.x, fmaf(d.y, h.y, fmaf(d.z, h.z, fmaf(d.w, h.w, gw3))));
                h.x = (s < valid && h.x > 0.0f) ? d.x * w3 : 0.0f;
                h.y = (s + 1 < valid && h.y > 0.0f) ? d.y * w3 : 0.0f;
                h.z = (s + 2 < valid && h.z > 0.0f) ? d.z * w3 : 0.0f;
                h.w = (s + 3 < valid && h.w > 0.0f) ? d.w * w3 : 0.0f;
                gb2 += (h.x + h.y) + (h.z + h.w);
                *reinterpret_cast<float4 *>(H2 + wa * kLd + s) = h;
            }
        }
        __syncthreads();
        {
            float acc[4][8] = {};
            tile_product(H2, W2, s0, u0, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float h[8];
                get8(H1 + (u0 + j) * kLd, s0, h);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int smp = s0 + (i & 3) + kHalf * (i >> 2);
                    acc[j][i] = (smp < valid && h[i] > 0.0f) ? acc[j][i] : 0.0f;
                }
                put8(D1 + (u0 + j) * kLd, s0, acc[j]);
            }
        }
        // W2[a][c] += sum D2[a] H1[c]
#pragma unroll 2
        for (int s = 0; s < kTile; s += 4) {
            float4 d[4], h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = ld4(H2 + (ga + 16 * i) * kLd + s);
#pragma unroll
            for (int j = 0; j < 4; ++j) h[j] = ld4(H1 + (gc + 16 * j) * kLd + s);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    g2[i][j] = fmaf(d[i].w, h[j].w, fmaf(d[i].z, h[j].z, fmaf(d[i].y, h[j].y, fmaf(d[i].x, h[j].x,
                                                                                                 g2[i][j]))));
        }
        __syncthreads();
        // W1[a][c] += sum D1[a] f[c]: columns 2 wq and 2 wq + 1
#pragma unroll 2
        for (int s = 0; s < kTile; s += 4) {
            const float4 d = ld4(D1 + wa * kLd + s), f0 = ld4(F + (2 * wq) * kLd + s), f1 = ld4(F + (2 * wq + 1) * kLd + s);
            g1[0] = fmaf(d.w, f0.w, fmaf(d.z, f0.z, fmaf(d.y, f0.y, fmaf(d.x, f0.x, g1[0]))));
            g1[1] = fmaf(d.w, f1.w, fmaf(d.z, f1.z, fmaf(d.y, f1.y, fmaf(d.x, f1.x, g1[1]))));
            if (((s >> 2) & 3) == wq) gb1 += (d.x + d.y) + (d.z + d.w);
        }
    }
    fold_all();
    float *out = partial + (int64_t)blockIdx.x * (MLP_NPARAM + 1);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) out[OFF_W2 + (ga + 16 * i) * MLP_W + gc + 16 * j] = s2[i][j];
    out[OFF_W1 + wa * MLP_IN + 2 * wq] = s1[0];
    out[OFF_W1 + wa * MLP_IN + 2 * wq + 1] = s1[1];
#pragma unroll
    for (int h = 1; h < 4; h <<= 1) {
        sb1 += __shfl_xor_sync(0xffffffffu, sb1, h);
        sb2 += __shfl_xor_sync(0xffffffffu, sb2, h);
        sw3 += __shfl_xor_sync(0xffffffffu, sw3, h);
    }
    if (wq == 0) {
        out[OFF_B1 + wa] = sb1;
        out[OFF_B2 + wa] = sb2;
        out[OFF_W3 + wa] = sw3;
    }
    __syncthreads();
    if (t < kTile) {
        DO[t] = gb3;
        ER[t] = gl;
    }
    __syncthreads();
    for (int h = kTile / 2; h > 0; h >>= 1) {
        if (t < h) {
            DO[t] += DO[t + h];
            ER[t] += ER[t + h];
        }
        __syncthreads();
    }
    if (t == 0) {
        out[OFF_B3] = DO[0];
        out[MLP_NPARAM] = ER[0];
    }
}

// One warp per 32 parameters x 8 rows at a time: thread (x, y) adds rows y,
// y + 8, ... in order, then the eight sums are added in order.
__global__ void __launch_bounds__(256)
mlp_grad_reduce_kernel(const float *__restrict__ partial, int rows, float scale, float *__restrict__ grads,
                       float *__restrict__ loss_out) {
    __shared__ float sums[8][32];
    const int x = threadIdx.x % 32, y = threadIdx.x / 32;
    const int t = blockIdx.x * 32 + x;
    float s = 0.0f;
    if (t <= MLP_NPARAM)
#pragma unroll 8
        for (int c = y; c < rows; c += 8) s += partial[(int64_t)c * (MLP_NPARAM + 1) + t];
    sums[y][x] = s;
    __syncthreads();
    if (y != 0 || t > MLP_NPARAM) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) s += sums[k][x];
    if (t == MLP_NPARAM) *loss_out = s * scale;
    else grads[t] = s * scale;
}

__global__ void adam_kernel(int64_t n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void mlp_predict_kernel(const float *__restrict__ params, const float *__restrict__ feats, int64_t n,
                                   float *__restrict__ out) {
    __shared__ float P[MLP_NPARAM];
    stage_params(params, P);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float f[MLP_IN], h1[MLP_W], h2[MLP_W];
#pragma unroll
    for (int c = 0; c < MLP_IN; ++c) f[c] = feats[i * MLP_IN + c];
    out[i] = expf(kLogR * tanhf(mlp_forward(P, f, h1, h2)));
}

// ------------------------------------------------------------ inside hb_diag
// features of every row for the Ritz values theta[which[j]] -> feats[j][n][8]
__global__ void diag_features_kernel(const double *__restrict__ d, const float *__restrict__ ri, int64_t n,
                                     const double *__restrict__ theta, int q, float *__restrict__ feats) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n || j >= q) return;
    float f[MLP_IN];
    features((float)d[i], (float)theta[j], (float)theta[0], ri, i, n, f);
#pragma unroll
    for (int c = 0; c < MLP_IN; ++c) feats[((int64_t)j * n + i) * MLP_IN + c] = f[c];
}

// w[j][i] = MLP factor for row i and Ritz value theta[j] (FP16 weights)
__global__ void diag_mlp_kernel(const __half *__restrict__ wh, const float *__restrict__ params,
                                const double *__restrict__ d, const float *__restrict__ ri, int64_t n,
                                const double *__restrict__ theta, int q, float *__restrict__ w) {
    __shared__ float P[MLP_NPARAM];
    for (int t = threadIdx.x; t < MLP_NPARAM; t += blockDim.x) {
        const bool is_bias = (t >= OFF_B1 && t < OFF_W2) || (t >= OFF_B2 && t < OFF_W3) || t == OFF_B3;
        P[t] = is_bias ? params[t] : __half2float(wh[t]);
    }
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n || j >= q) return;
    float f[MLP_IN], h1[MLP_W], h2[MLP_W];
    features((float)d[i], (float)theta[j], (float)theta[0], ri, i, n, f);
    const float o = mlp_forward(P, f, h1, h2);
    float v = expf(kLogR * tanhf(o));
    if (!isfinite(v)) v = 1.0f;
    w[(int64_t)j * n + i] = v;
}

// row_info from the build: type, E_n, h_jj, group id
__global__ void row_info_kernel(int64_t row0, int ns, int cn, int cf, int n_to, int n_orb, const double *__restrict__ h,
                                const double *__restrict__ E, float gid, int64_t n, float *__restrict__ ri) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)ns * cn) return;
    const int st = (int)(t / cn), j = (int)(t % cn);
    const int64_t i = row0 + t;
    const int orb = n_to + cf + j;
    ri[i] = 0.0f;
    ri[n + i] = (float)E[st * ns + st];
    ri[2 * n + i] = (float)h[(int64_t)orb * n_orb + orb];
    ri[3 * n + i] = gid;
}

}  // namespace

// ------------------------------------------------------------------- host
static int mlp_fail(hb_ctx *ctx, int code, const std::string &m) {
    if (ctx) ctx->err = m;
    return code;
}

static int ensure_rows(hb_ctx *ctx, MlpState &M, DiagWork *w, cudaStream_t s) {
    const int64_t n = ctx->dim;
    if (M.n != n || !M.row_info) {
        dfree(ctx, M.row_info);
        M.row_info = nullptr;
        if (dmalloc_n(ctx, &M.row_info, (size_t)4 * n) != cudaSuccess) return HB_ERR_OOM;
        M.n = n;
        M.rows_ready = false;
    }
    if (M.rows_ready) return HB_OK;
    // L2 rows: type 1, group id 1; continuum rows per group from the last build
    std::vector<float> init(4 * n, 0.0f);
    for (int64_t i = ctx->Dc; i < n; ++i) { init[i] = 1.0f; init[3 * n + i] = 1.0f; }
    cudaMemcpyAsync(M.row_info, init.data(), sizeof(float) * 4 * n, cudaMemcpyHostToDevice, s);
    for (auto &P : ctx->gps) {
        if (!P.same) continue;
        const GroupInfo &G = ctx->groups[P.g];
        const int64_t cnt = (int64_t)G.ns * G.cn;
        row_info_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(
            G.row_off, G.ns, G.cn, G.cf, ctx->n_to, ctx->n_orb, ctx->h, P.E,
            ctx->n_groups > 1 ? (float)P.g / (float)ctx->n_groups : 0.0f, n, M.row_info);
    }
    cudaStreamSynchronize(s);
    M.rows_ready = true;
    (void)w;
    return HB_OK;
}

int hb::mlp_weights_for(hb_ctx *ctx, DiagWork *w, const double *theta, int nr, float **out, cudaStream_t s) {
    *out = nullptr;
    MlpState *M = (MlpState *)ctx->mlp;
    if (!M || !M->wh) return mlp_fail(ctx, HB_ERR_UNSUPPORTED, "no preconditioner network");
    if (ensure_rows(ctx, *M, w, s) != HB_OK) return HB_ERR_OOM;
    if (M->mmax < nr || !M->w) {
        dfree(ctx, M->w);
        M->w = nullptr;
        if (dmalloc_n(ctx, &M->w, (size_t)nr * ctx->dim) != cudaSuccess) return HB_ERR_OOM;
        M->mmax = nr;
    }
    // theta is already on the device in w->theta (hb_diag copies it before the call)
    dim3 g((unsigned)((ctx->dim + 127) / 128), nr);
    diag_mlp_kernel<<<g, 128, 0, s>>>(M->wh, M->bias, w->d, M->row_info, ctx->dim, w->theta, nr, M->w);
    if (cudaGetLastError() != cudaSuccess) return HB_ERR_CUDA;
    (void)theta;
    *out = M->w;
    return HB_OK;
}

void hb::release_mlp(hb_ctx *ctx) {
    MlpState *M = (MlpState *)ctx->mlp;
    if (!M) return;
    for (void *p : {(void *)M->wh, (void *)M->bias, (void *)M->row_info, (void *)M->w, (void *)M->feats})
        dfree(ctx, p);
    delete M;
    ctx->mlp = nullptr;
}

extern "C" int hb_mlp_param_count(int32_t n_in, int32_t width) {
    return (n_in == MLP_IN && width == MLP_W) ? MLP_NPARAM : -1;
}

extern "C" int hb_mlp_set(hb_ctx *ctx, const hb_mlp_weights *wt) {
    if (!ctx || !wt) return mlp_fail(ctx, HB_ERR_INVALID_ARG, "NULL argument");
    if (wt->n_in != MLP_IN || wt->width != MLP_W)
        return mlp_fail(ctx, HB_ERR_UNSUPPORTED, "the preconditioner network has 8 inputs and width 64");
    if (!wt->w1 || !wt->b1 || !wt->w2 || !wt->b2 || !wt->w3 || !wt->b3)
        return mlp_fail(ctx, HB_ERR_INVALID_ARG, "NULL weight array");
    std::vector<float> p(MLP_NPARAM);
    std::memcpy(&p[OFF_W1], wt->w1, sizeof(float) * MLP_W * MLP_IN);
    std::memcpy(&p[OFF_B1], wt->b1, sizeof(float) * MLP_W);
    std::memcpy(&p[OFF_W2], wt->w2, sizeof(float) * MLP_W * MLP_W);
    std::memcpy(&p[OFF_B2], wt->b2, sizeof(float) * MLP_W);
    std::memcpy(&p[OFF_W3], wt->w3, sizeof(float) * MLP_W);
    std::memcpy(&p[OFF_B3], wt->b3, sizeof(float));
    for (float x : p)
        if (!std::isfinite(x)) return mlp_fail(ctx, HB_ERR_INVALID_ARG, "non-finite weights");
    std::vector<__half> ph(MLP_NPARAM);
    for (int i = 0; i < MLP_NPARAM; ++i) ph[i] = __float2half_rn(p[i]);
    MlpState *M = (MlpState *)ctx->mlp;
    if (!M) { M = new MlpState(); ctx->mlp = M; }
    if (!M->wh && dmalloc_n(ctx, &M->wh, (size_t)MLP_NPARAM) != cudaSuccess) return HB_ERR_OOM;
    if (!M->bias && dmalloc_n(ctx, &M->bias, (size_t)MLP_NPARAM) != cudaSuccess) return HB_ERR_OOM;
    if (cudaMemcpy(M->wh, ph.data(), sizeof(__half) * MLP_NPARAM, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(M->bias, p.data(), sizeof(float) * MLP_NPARAM, cudaMemcpyHostToDevice) != cudaSuccess)
        return mlp_fail(ctx, HB_ERR_CUDA, "uploading weights");
    M->rows_ready = false;
    return HB_OK;
}

// One row of partial sums per block of the training kernel: a block per SM, and
// no more than there are tiles.
static int64_t train_tiles(int64_t n) { return (n + kTile - 1) / kTile; }
constexpr int kTrainMaxBlocks = 256;

extern "C" int64_t hb_mlp_workspace_bytes(int64_t n) {
    return (int64_t)sizeof(float) * std::min<int64_t>(std::max<int64_t>(train_tiles(n), 1), kTrainMaxBlocks) *
           (MLP_NPARAM + 1);
}

extern "C" int hb_mlp_loss_grad(const float *params, const float *feats, const float *a, const float *b, int64_t n,
                                float *grads, float *loss, void *work, void *stream) {
    if (!params || !feats || !a || !b || !grads || !loss || !work || n <= 0) return HB_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem) != cudaSuccess)
        return HB_ERR_CUDA;
    const int64_t tiles = train_tiles(n);
    const int blocks = (int)std::min<int64_t>(tiles, std::min(sms, kTrainMaxBlocks));
    float *partial = (float *)work;
    mlp_train_kernel<<<blocks, kTrainThreads, kTrainSmem, s>>>(params, feats, a, b, n, tiles, partial);
    mlp_grad_reduce_kernel<<<(MLP_NPARAM + 1 + 31) / 32, 256, 0, s>>>(partial, blocks, 1.0f / (float)n, grads, loss);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ERR_CUDA;
}

extern "C" int hb_mlp_adam(int64_t n_param, float *params, const float *grads, float *m, float *v, int32_t step,
                           float lr, void *stream) {
    if (!params || !grads || !m || !v || step < 1) return HB_ERR_INVALID_ARG;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    adam_kernel<<<(unsigned)((n_param + 255) / 256), 256, 0, (cudaStream_t)stream>>>(n_param, params, grads, m, v, lr,
                                                                                      b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ERR_CUDA;
}

// Adam training over a device data set: the samples are taken in consecutive
// windows of `batch` (wrapping around), one loss-and-gradient pass and one
// update per step, the loss of the last step in *last_loss (host).  Scratch
// (gradients, moments, workspace) is allocated and freed by the call.
// The Adam loop of both training entry points; the scratch comes from `mem`
// (a context's memory) or from cudaMalloc when mem is null.
static int mlp_train_loop(hb_ctx *mem, float *params, const float *feats, const float *a, const float *b, int64_t n,
                          int64_t batch, int32_t steps, float lr, float *last_loss, void *stream) {
    if (!params || !feats || !a || !b || n <= 0 || batch <= 0 || steps < 1 || !(lr > 0.0f))
        return HB_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t bs = batch < n ? batch : n;
    float *g = nullptr, *m = nullptr, *v = nullptr, *loss = nullptr;
    void *work = nullptr;
    auto alloc = [&](void **p, size_t bytes) {
        return mem ? dmalloc(mem, p, bytes) : cudaMalloc(p, bytes);
    };
    cudaError_t e = alloc((void **)&g, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = alloc((void **)&m, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = alloc((void **)&v, sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = alloc((void **)&loss, sizeof(float));
    if (e == cudaSuccess) e = alloc(&work, (size_t)hb_mlp_workspace_bytes(bs));
    if (e == cudaSuccess) e = cudaMemsetAsync(m, 0, sizeof(float) * MLP_NPARAM, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(v, 0, sizeof(float) * MLP_NPARAM, s);
    int rc = e == cudaSuccess ? HB_OK : HB_ERR_OOM;
    int64_t off = 0;
    for (int32_t step = 1; step <= steps && rc == HB_OK; ++step) {
        const int64_t cnt = off + bs <= n ? bs : n - off;
        rc = hb_mlp_loss_grad(params, feats + off * MLP_IN, a + off, b + off, cnt, g, loss, work, stream);
        if (rc == HB_OK) rc = hb_mlp_adam(MLP_NPARAM, params, g, m, v, step, lr, stream);
        off += cnt;
        if (off >= n) off = 0;
    }
    if (rc == HB_OK && last_loss) {
        e = cudaMemcpyAsync(last_loss, loss, sizeof(float), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = HB_ERR_CUDA;
    }
    cudaStreamSynchronize(s);
    for (void *p : {(void *)g, (void *)m, (void *)v, (void *)loss, work}) {
        if (mem) dfree(mem, p);
        else if (p) cudaFree(p);
    }
    return rc;
}

extern "C" int hb_mlp_train_params(float *params, const float *feats, const float *a, const float *b, int64_t n,
                                   int64_t batch, int32_t steps, float lr, float *last_loss, void *stream) {
    return mlp_train_loop(nullptr, params, feats, a, b, n, batch, steps, lr, last_loss, stream);
}

extern "C" int hb_mlp_train(hb_ctx *ctx, const hb_mlp_dataset *d, float *params, hb_stats *st, void *stream) {
    if (!ctx || !d || !params) return mlp_fail(ctx, HB_ERR_INVALID_ARG, "NULL argument");
    float last = 0.0f;
    int rc = mlp_train_loop(ctx, params, d->feats, d->a, d->b, d->n, d->batch, d->steps, d->lr, &last, stream);
    if (rc != HB_OK) return mlp_fail(ctx, rc, "training failed (arguments, memory or launch)");
    // the trained network becomes the context's preconditioner network
    std::vector<float> p(MLP_NPARAM);
    if (cudaMemcpy(p.data(), params, sizeof(float) * MLP_NPARAM, cudaMemcpyDeviceToHost) != cudaSuccess)
        return mlp_fail(ctx, HB_ERR_CUDA, "reading the trained parameters");
    hb_mlp_weights w{MLP_IN, MLP_W, &p[OFF_W1], &p[OFF_B1], &p[OFF_W2], &p[OFF_B2], &p[OFF_W3], &p[OFF_B3]};
    rc = hb_mlp_set(ctx, &w);
    if (rc != HB_OK) return rc;
    if (st) {
        memset(st, 0, sizeof(*st));
        st->iterations = d->steps;
        st->mlp_loss = last;
    }
    return HB_OK;
}

extern "C" int hb_mlp_predict(const float *params, const float *feats, int64_t n, float *out, void *stream) {
    if (!params || !feats || !out || n <= 0) return HB_ERR_INVALID_ARG;
    mlp_predict_kernel<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(params, feats, n, out);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ERR_CUDA;
}

extern "C" int hb_diag_features(hb_ctx *ctx, const hb_blocks *H, const double *theta, int32_t q, float *feats,
                                void *stream) {
    if (!ctx || !H || !theta || q < 1 || !feats) return mlp_fail(ctx, HB_ERR_INVALID_ARG, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = ensure_diag_work(ctx, H, std::max(q, 1), s);
    if (rc != HB_OK) return rc;
    DiagWork *w = (DiagWork *)ctx->diag;
    fill_diag(ctx, H, w, s);   // the diagonal of H from the blocks
    MlpState *M = (MlpState *)ctx->mlp;
    if (!M) { M = new MlpState(); ctx->mlp = M; }
    rc = ensure_rows(ctx, *M, w, s);
    if (rc != HB_OK) return rc;
    double *th = nullptr;
    if (dmalloc_n(ctx, &th, (size_t)q) != cudaSuccess) return HB_ERR_OOM;
    cudaMemcpyAsync(th, theta, sizeof(double) * q, cudaMemcpyHostToDevice, s);
    dim3 g((unsigned)((ctx->dim + 255) / 256), q);
    diag_features_kernel<<<g, 256, 0, s>>>(w->d, M->row_info, ctx->dim, th, q, feats);
    cudaStreamSynchronize(s);
    dfree(ctx, th);
    return cudaGetLastError() == cudaSuccess ? HB_OK : HB_ERR_CUDA;
}
