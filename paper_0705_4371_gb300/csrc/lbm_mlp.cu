// lbm_mlp.cu -- learned form: training data for the network that
// warm-starts the energy Newton solve, and its training on the GPU.
//
//   lb_energy_dataset  moments -> energy-constrained multipliers mu by Newton
//                      (FP32 iterations, FP64 finish to 1e-12; Sec. 3.3),
//                      with the network's features and corrections mu - mu0
//   lb_mlp_normalise   input standardisation and output scales from a data set
//   lb_mlp_forward     the network on a batch (the kernels' own evaluation)
//   lb_mlp_grad        mean squared error and its gradient (deterministic)
//   lb_mlp_adam        one Adam update
//   lb_mlp_train       epochs of mini-batch Adam
//
// The forward pass of training is the inference routine (BF16 tensor cores,
// FP32 accumulation), so the network is trained on exactly the arithmetic
// that later evaluates it.  The backward pass runs in FP32 on the BF16
// weights and activations the forward pass used (gradients pass straight
// through the roundings); per-block partial sums are reduced in a fixed
// order, so every result is reproducible bit for bit.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_device.cuh"
#include "lbm_energy.cuh"
#include "lbm_internal.h"
#include "lbm_mlp.cuh"

using namespace lbm;

namespace {

constexpr int kGradRows = 32;                    // samples a block takes at a time
constexpr int kGradThreads = 256;
constexpr int kLd = kMlpHid + 4;                 // activation row: 16-byte aligned, rows on different banks
constexpr int kPartial = kMlpTrainable + 1;      // per-block gradient sums and the loss
constexpr int kPartialLd = (kPartial + 3) / 4 * 4;   // a block's row of them (16-byte aligned)
constexpr int kReduceThreads = 256;
// Adam's constants; 1 - b is stored as its own correctly rounded FP32 value
// (1.0f - 0.999f differs from 0.001 by 1.3e-5 relative)
constexpr double kAdamB1d = 0.9, kAdamB2d = 0.999;
constexpr float kAdamB1 = 0.9f, kAdamB2 = 0.999f, kAdam1mB1 = 0.1f, kAdam1mB2 = 0.001f, kAdamEps = 1e-8f;

int fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    set_last_error(buf);
    return code;
}

#define CK(x)                                                                                     \
    do {                                                                                          \
        cudaError_t e_ = (x);                                                                     \
        if (e_ != cudaSuccess)                                                                    \
            return fail(e_ == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA, "%s: %s", #x, \
                        cudaGetErrorString(e_));                                                  \
    } while (0)

// ---------------------------------------------------------------------------
// Training data: for sample i, the moments (rho, rho u, 2E) with
// 2E = escale_i x (2E of the isothermal entropic equilibrium, Sec. 4.2),
// the multipliers mu of ln(f*_j / W_j) = mu . (1, v_x, v_y, |v|^2) by the
// energy Newton solve from the polynomial start point, the features
// (rho, u_x, u_y, 2E/rho - |u|^2) and the corrections mu - mu0.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_energy_dataset(const double* __restrict__ rho,
                                                         const double* __restrict__ ux,
                                                         const double* __restrict__ uy,
                                                         const double* __restrict__ escale, long long n,
                                                         float* __restrict__ feat, float* __restrict__ dmu,
                                                         double* __restrict__ mu,
                                                         unsigned long long* __restrict__ stats) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    NewtonCount nc = {0, 0, 0, 0};
    if (i < n) {
        const double r = rho[i], u = ux[i], v = uy[i];
        // second moment of the isothermal product form (Sec. 4.2) per axis:
        // (2 sqrt(1 + 3 u^2) - 1) / 3
        const double sx = sqrt(fma(3.0 * u, u, 1.0)), sy = sqrt(fma(3.0 * v, v, 1.0));
        const double th = escale[i] * (2.0 / 3.0) * (sx + sy - 1.0);
        double fs[9], mu3[3];
        energy_solve(r, u, v, th, 0.0f, fs, nc, 4e-15f, mu3);
        const double m[4] = {log(fs[0] / D2Q9::w(0)), mu3[0], mu3[1], mu3[2]};
        const double m0[4] = {log(r) - 1.5 * (u * u + v * v), 3.0 * u, 3.0 * v, 0.0};
        const double f[4] = {r, u, v, th - u * u - v * v};
#pragma unroll
        for (int j = 0; j < 4; j++) {
            feat[i * 4 + j] = (float)f[j];
            dmu[i * 4 + j] = (float)(m[j] - m0[j]);
            if (mu) mu[i * 4 + j] = m[j];
        }
    }
    if (stats) {
        unsigned long long v4[4] = {nc.it32, nc.it64, nc.sites, nc.fails};
#pragma unroll
        for (int j = 0; j < 4; j++) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v4[j] += __shfl_xor_sync(0xffffffffu, v4[j], o);
        }
        if ((threadIdx.x & 31) == 0 && v4[2] > 0)
            for (int j = 0; j < 4; j++) atomicAdd(stats + j, v4[j]);
    }
}

// ---------------------------------------------------------------------------
// Standardisation of the features (mean, 1 / standard deviation) and the
// output scales (root mean square of mu - mu0) from a data set; one block,
// FP64 sums in a fixed order.
// ---------------------------------------------------------------------------
// Bound by the FP64 pipe (24 FP64 operations per sample at two per SM and
// clock), so the sums are spread over the whole GPU: a block sums a fixed
// set of samples and a second launch adds the blocks' sums in their order.
// 2^18 samples: 2105 us on one block of 1024 threads, 43 us on these.
constexpr int kNormThreads = 256;
constexpr int kNormBlocks = 608;                 // four blocks per SM
constexpr int kNormSums = 12;

__global__ void __launch_bounds__(kNormThreads) k_mlp_norm_sums(const float* __restrict__ feat,
                                                                 const float* __restrict__ dmu, long long n,
                                                                 double* __restrict__ sums) {
    __shared__ double red[kNormSums][kNormThreads / 32];
    double acc[kNormSums];
#pragma unroll
    for (int j = 0; j < kNormSums; j++) acc[j] = 0.0;
    for (long long i = (long long)blockIdx.x * kNormThreads + threadIdx.x; i < n;
         i += (long long)gridDim.x * kNormThreads) {
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const double f = feat[i * 4 + j], d = dmu[i * 4 + j];
            acc[j] += f;
            acc[4 + j] = fma(f, f, acc[4 + j]);
            acc[8 + j] = fma(d, d, acc[8 + j]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < kNormSums; j++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        if (lane == 0) red[j][warp] = acc[j];
    }
    __syncthreads();
    if (threadIdx.x < kNormSums) {
        double s = 0.0;
        for (int w = 0; w < kNormThreads / 32; w++) s += red[threadIdx.x][w];
        sums[(size_t)blockIdx.x * kNormSums + threadIdx.x] = s;
    }
}

__global__ void __launch_bounds__(32 * kNormSums) k_mlp_norm_finish(float* __restrict__ p,
                                                                    const double* __restrict__ sums, int blocks,
                                                                    long long n) {
    __shared__ double red[kNormSums];
    const int lane = threadIdx.x & 31, j = threadIdx.x >> 5;   // warp j adds sum j
    double s = 0.0;
    for (int b = lane; b < blocks; b += 32) s += sums[(size_t)b * kNormSums + j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[j] = s;
    __syncthreads();
    if (threadIdx.x < 4) {
        const int c = threadIdx.x;
        const double mean = red[c] / (double)n;
        const double var = red[4 + c] / (double)n - mean * mean;
        const double sd = var > 0.0 ? sqrt(var) : 0.0;
        const double rms = sqrt(red[8 + c] / (double)n);
        p[kMlpMean + c] = (float)mean;
        p[kMlpIstd + c] = sd > 0.0 ? (float)(1.0 / sd) : 1.0f;
        p[kMlpOscale + c] = rms > 0.0 ? (float)rms : 1.0f;
    }
}

// ---------------------------------------------------------------------------
// The network on a batch: y[i][0..3] for features feat[i][0..3].
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_mlp_forward(const float* __restrict__ p,
                                                     const float* __restrict__ feat, long long n,
                                                     float* __restrict__ y) {
    __shared__ MlpSmem ms;
    mlp_fill(ms, p);
    __syncthreads();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < n;
    unsigned p01 = 0u, p23 = 0u;
    if (valid) mlp_inputs(ms, feat[i * 4], feat[i * 4 + 1], feat[i * 4 + 2], feat[i * 4 + 3], p01, p23);
    float out[kMlpOut];
    mlp_warp_forward(ms, p01, p23, out);
    if (valid)
        for (int j = 0; j < kMlpOut; j++) y[i * 4 + j] = out[j];
}

// ---------------------------------------------------------------------------
// Loss gradient.  A block of 256 threads takes groups of 32 samples: forward
// pass (two warps, one 16-sample tile each, capturing the BF16 activations),
// backward pass and the block's sums over its samples of every trainable
// entry's gradient and of the squared errors, which stay in registers (a
// thread owns 4 x 4 entries of W2 and at most five others) until the block's
// last group.  Samples i0 .. i0 + n - 1; targets (mu - mu0) / out_scale;
// inv_count = 1 / (4 x batch size) (the loss is the mean over the batch and
// the four outputs).
// A batch of a few thousand samples is far too small to fill the GPU's
// arithmetic (33 M multiply-adds each way): what bounds a step is the chain
// fill - forward - backward - sums - reduction.  Groups of 32 samples put a
// batch of 4096 on 128 SMs, and the register tiles (2 x 4 of dz1, 4 x 4 of
// dW2) take one shared-memory access per four multiply-adds.
// ---------------------------------------------------------------------------
// Groups of a batch of n > 0 samples (no sum that exceeds an int).
__host__ __device__ constexpr int grad_groups(int n) { return (n - 1) / kGradRows + 1; }
static_assert(grad_groups(1) == 1 && grad_groups(kGradRows) == 1 && grad_groups(kGradRows + 1) == 2 &&
              grad_groups(0x7fffffff) == 1 << 26, "groups of the smallest and largest batches");

struct __align__(16) GradSmem {
    float w2[kMlpHid][kMlpHid];        // BF16-rounded W2, W3 as floats
    float w3[kMlpOut][kMlpHid];
    float h1[kGradRows][kLd], h2[kGradRows][kLd];
    float dz1[kGradRows][kLd], dz2[kGradRows][kLd];
    float x[kGradRows][kMlpIn], dy[kGradRows][kMlpOut], tg[kGradRows][kMlpOut];
    unsigned xp[kGradRows][2];         // standardised inputs as BF16 pairs
    float loss[kGradRows];
    MlpSmem ms;
};

// A thread's share of the block's sums: entries (4 ng + a, 4 kg + b) of dW2
// (kg = tid mod 16, ng = tid / 16), and in ex
//   tid < 64:         dW1[tid][0..3], db1[tid]
//   64 <= tid < 128:  dW3[0..3][tid - 64], db2[tid - 64]
//   128 <= tid < 132: db3[tid - 128];  tid = 132: the squared errors.
struct GradAcc {
    float w2[4][4];
    float ex[5];
};

// The block's copy of the parameters (global memory written by other blocks
// of the same launch in training: read through L2).
__device__ __forceinline__ void grad_fill(GradSmem& s, const float* __restrict__ p) {
    const int tid = threadIdx.x;
    // W2 once, for both uses: fragment (nt, ks, lane) holds four weights
#pragma unroll
    for (int e = tid; e < 8 * 4 * 32; e += kGradThreads) {
        const int nt = e >> 7, ks = (e >> 5) & 3, lane = e & 31, g = lane >> 2, tig = lane & 3;
        const int n = 8 * nt + g, k = 16 * ks + 2 * tig;
        const float* row = p + kMlpW2 + n * kMlpHid + k;
        const unsigned lo = bf16_pack(__ldcg(row), __ldcg(row + 1)), hi = bf16_pack(__ldcg(row + 8), __ldcg(row + 9));
        s.ms.w2[nt][ks][lane] = make_uint2(lo, hi);
        s.w2[n][k] = bf16_lo(lo);
        s.w2[n][k + 1] = bf16_hi(lo);
        s.w2[n][k + 8] = bf16_lo(hi);
        s.w2[n][k + 9] = bf16_hi(hi);
    }
    {
        const int nt = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3;
        const float* w = p + kMlpW1 + (8 * nt + g) * kMlpIn + 2 * (tig & 1);
        s.ms.w1[nt][lane] = tig < 2 ? bf16_pack(__ldcg(w), __ldcg(w + 1)) : 0u;
    }
    if (tid < 128) {
        const int ks = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3;
        uint2 f = make_uint2(0u, 0u);
        if (g < kMlpOut) {
            const int k = 16 * ks + 2 * tig;
            const float* row = p + kMlpW3 + g * kMlpHid + k;
            f = make_uint2(bf16_pack(__ldcg(row), __ldcg(row + 1)), bf16_pack(__ldcg(row + 8), __ldcg(row + 9)));
            s.w3[g][k] = bf16_lo(f.x);
            s.w3[g][k + 1] = bf16_hi(f.x);
            s.w3[g][k + 8] = bf16_lo(f.y);
            s.w3[g][k + 9] = bf16_hi(f.y);
        }
        s.ms.w3[ks][lane] = f;
    } else if (tid < 192) {
        s.ms.b1[tid - 128] = __ldcg(p + kMlpB1 + tid - 128);
    } else {
        s.ms.b2[tid - 192] = __ldcg(p + kMlpB2 + tid - 192);
    }
    if (tid < 8) s.ms.b3[tid] = tid < kMlpOut ? __ldcg(p + kMlpB3 + tid) : 0.0f;
    if (tid < kMlpIn) {
        s.ms.mean[tid] = p[kMlpMean + tid];
        s.ms.istd[tid] = p[kMlpIstd + tid];
        s.ms.oscale[tid] = p[kMlpOscale + tid];
    }
}

// Features and targets of a group's samples: thread t < 128 holds component
// t mod 4 of sample t / 4 (zero beyond the batch).
struct GradIn {
    float f, d;
};
__device__ __forceinline__ GradIn grad_load(const float* __restrict__ feat, const float* __restrict__ dmu,
                                            long long i0, int n, int group) {
    GradIn in = {0.0f, 0.0f};
    const int i = group * kGradRows + (int)(threadIdx.x >> 2);
    if (threadIdx.x < 4 * kGradRows && i < n) {
        in.f = feat[(i0 + i) * 4 + (threadIdx.x & 3)];
        in.d = dmu[(i0 + i) * 4 + (threadIdx.x & 3)];
    }
    return in;
}

// One group of samples, added to the thread's sums (every thread calls; the
// shared state of the previous group must no longer be needed).
__device__ __forceinline__ void grad_group(GradSmem& s, GradIn in, int valid, float inv_count, GradAcc& acc) {
    const int tid = threadIdx.x;
    if (tid < 4 * kGradRows) {
        // (f - mean) * inv_std in FP32, rounded to BF16 by pairs, as mlp_inputs
        const int c = tid & 3, r = tid >> 2;
        const float v = r < valid ? (in.f - s.ms.mean[c]) * s.ms.istd[c] : 0.0f;
        const unsigned b = bf16_pack(v, __shfl_down_sync(0xffffffffu, v, 1));
        s.x[r][c] = bf16_lo(b);
        if (!(c & 1)) s.xp[r][c >> 1] = b;
        s.tg[r][c] = r < valid ? in.d / s.ms.oscale[c] : 0.0f;
    }
    __syncthreads();
    if (tid < 2 * 32) {
        const int m = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3, r0 = 16 * m + g;
        const unsigned a0 = tig < 2 ? s.xp[r0][tig] : 0u, a1 = tig < 2 ? s.xp[r0 + 8][tig] : 0u;
        float y[4];
        mlp_tile_forward<true>(s.ms, a0, a1, y, r0, &s.h1[0][0], &s.h2[0][0], kLd);
        if (tig < 2) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int r = r0 + (j >> 1) * 8, o = 2 * tig + (j & 1);
                const float d = r < valid ? y[j] - s.tg[r][o] : 0.0f;
                s.tg[r][o] = d * d;
                s.dy[r][o] = 2.0f * d * inv_count;
            }
        }
    }
    __syncthreads();
    // dz2 = (dy W3) where z2 > 0
    {
        const int k = tid & 63;
        const float w0 = s.w3[0][k], w1 = s.w3[1][k], w2 = s.w3[2][k], w3 = s.w3[3][k];
#pragma unroll
        for (int r = tid >> 6; r < kGradRows; r += kGradThreads / 64) {
            const float4 d = *reinterpret_cast<const float4*>(s.dy[r]);
            const float a = fmaf(d.w, w3, fmaf(d.z, w2, fmaf(d.y, w1, d.x * w0)));
            s.dz2[r][k] = s.h2[r][k] > 0.0f ? a : 0.0f;
        }
    }
    if (tid < kGradRows) s.loss[tid] = (s.tg[tid][0] + s.tg[tid][1]) + (s.tg[tid][2] + s.tg[tid][3]);
    __syncthreads();
    // dz1 = (dz2 W2) where z1 > 0: rows r, r + 16, columns c .. c + 3
    {
        const int c = 4 * (tid & 15), r = tid >> 4;
        float a[2][4] = {};
#pragma unroll 4
        for (int k = 0; k < kMlpHid; k += 4) {
            const float4 d0 = *reinterpret_cast<const float4*>(&s.dz2[r][k]);
            const float4 d1 = *reinterpret_cast<const float4*>(&s.dz2[r + 16][k]);
            const float e0[4] = {d0.x, d0.y, d0.z, d0.w}, e1[4] = {d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 w = *reinterpret_cast<const float4*>(&s.w2[k + q][c]);
                a[0][0] = fmaf(e0[q], w.x, a[0][0]);
                a[0][1] = fmaf(e0[q], w.y, a[0][1]);
                a[0][2] = fmaf(e0[q], w.z, a[0][2]);
                a[0][3] = fmaf(e0[q], w.w, a[0][3]);
                a[1][0] = fmaf(e1[q], w.x, a[1][0]);
                a[1][1] = fmaf(e1[q], w.y, a[1][1]);
                a[1][2] = fmaf(e1[q], w.z, a[1][2]);
                a[1][3] = fmaf(e1[q], w.w, a[1][3]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const float4 z = *reinterpret_cast<const float4*>(&s.h1[r + 16 * h][c]);
            *reinterpret_cast<float4*>(&s.dz1[r + 16 * h][c]) =
                make_float4(z.x > 0.0f ? a[h][0] : 0.0f, z.y > 0.0f ? a[h][1] : 0.0f, z.z > 0.0f ? a[h][2] : 0.0f,
                            z.w > 0.0f ? a[h][3] : 0.0f);
        }
    }
    // dW2 += dz2^T h1 over the group's samples, in sample order
    {
        const int k = 4 * (tid & 15), n = 4 * (tid >> 4);
#pragma unroll 8
        for (int q = 0; q < kGradRows; q++) {
            const float4 dz = *reinterpret_cast<const float4*>(&s.dz2[q][n]);
            const float4 h = *reinterpret_cast<const float4*>(&s.h1[q][k]);
            const float dn[4] = {dz.x, dz.y, dz.z, dz.w}, hk[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int b = 0; b < 4; b++) acc.w2[a][b] = fmaf(dn[a], hk[b], acc.w2[a][b]);
        }
    }
    __syncthreads();
    if (tid < 128) {
        // 0..63: dW1 and db1 from dz1 and x; 64..127: dW3 and db2 from h2, dy, dz2
        const int j = tid & 63;
        const bool first = tid < 64;
#pragma unroll 8
        for (int q = 0; q < kGradRows; q++) {
            const float v = first ? s.dz1[q][j] : s.h2[q][j];
            const float4 u = *reinterpret_cast<const float4*>(first ? s.x[q] : s.dy[q]);
            acc.ex[0] = fmaf(v, u.x, acc.ex[0]);
            acc.ex[1] = fmaf(v, u.y, acc.ex[1]);
            acc.ex[2] = fmaf(v, u.z, acc.ex[2]);
            acc.ex[3] = fmaf(v, u.w, acc.ex[3]);
            acc.ex[4] += first ? v : s.dz2[q][j];
        }
    } else if (tid < 128 + kMlpOut) {
        for (int q = 0; q < kGradRows; q++) acc.ex[0] += s.dy[q][tid - 128];
    } else if (tid == 128 + kMlpOut) {
        for (int q = 0; q < kGradRows; q++) acc.ex[0] += s.loss[q];
    }
    __syncthreads();
}

__device__ __forceinline__ void grad_zero(GradAcc& acc) {
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) acc.w2[a][b] = 0.0f;
#pragma unroll
    for (int j = 0; j < 5; j++) acc.ex[j] = 0.0f;
}

// The thread's sums to the block's row of partial[blocks][kPartialLd].
__device__ __forceinline__ void grad_store(const GradAcc& acc, float* __restrict__ out) {
    const int tid = threadIdx.x, k = 4 * (tid & 15), n = 4 * (tid >> 4);
#pragma unroll
    for (int a = 0; a < 4; a++)
        *reinterpret_cast<float4*>(out + kMlpW2 + (n + a) * kMlpHid + k) =
            make_float4(acc.w2[a][0], acc.w2[a][1], acc.w2[a][2], acc.w2[a][3]);
    if (tid < 64) {
#pragma unroll
        for (int j = 0; j < 4; j++) out[kMlpW1 + tid * kMlpIn + j] = acc.ex[j];
        out[kMlpB1 + tid] = acc.ex[4];
    } else if (tid < 128) {
#pragma unroll
        for (int j = 0; j < 4; j++) out[kMlpW3 + j * kMlpHid + tid - 64] = acc.ex[j];
        out[kMlpB2 + tid - 64] = acc.ex[4];
    } else if (tid < 128 + kMlpOut) {
        out[kMlpB3 + tid - 128] = acc.ex[0];
    } else if (tid == 128 + kMlpOut) {
        out[kMlpTrainable] = acc.ex[0];
    }
}

// Sums of one batch's samples by blocks 0 .. gridDim.x - 1 (groups of 32
// samples in turn).
__global__ void __launch_bounds__(kGradThreads) k_mlp_grad(const float* __restrict__ p,
                                                           const float* __restrict__ feat,
                                                           const float* __restrict__ dmu, int n, float inv_count,
                                                           float* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& s = *reinterpret_cast<GradSmem*>(smem_raw);
    grad_fill(s, p);
    __syncthreads();
    GradAcc acc;
    grad_zero(acc);
    for (int g = blockIdx.x; g < grad_groups(n); g += gridDim.x)
        grad_group(s, grad_load(feat, dmu, 0, n, g), n - g * kGradRows, inv_count, acc);
    grad_store(acc, partial + (size_t)blockIdx.x * kPartialLd);
}

// Gradient and loss from the block partials, added in block order.
__global__ void __launch_bounds__(kReduceThreads) k_mlp_reduce(const float* __restrict__ partial, int nblk,
                                                               float* __restrict__ grad, float* loss_out,
                                                               float loss_scale) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const bool loss = e == kMlpParams;
    float g = 0.0f;
    if (e < kMlpTrainable || loss) {
        const float* at = partial + (loss ? kMlpTrainable : e);
#pragma unroll 16
        for (int b = 0; b < nblk; b++) g += at[(size_t)b * kPartialLd];
    }
    if (e < kMlpParams) grad[e] = g;
    else if (loss && loss_out) *loss_out = g * loss_scale;
}

// ---------------------------------------------------------------------------
// Training: every optimiser step of a chunk in one cooperative launch.  A
// step is the blocks' gradient sums of its batch, a grid barrier, the
// reduction with the Adam update (Kingma and Ba, 2015),
//   m <- b1 m + (1 - b1) g,  v <- b2 v + (1 - b2) g^2,
//   p <- p - lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps),
// of the entries the block owns (their p, m, v stay in its shared memory),
// and a second barrier before the next step reads the parameters.  Against
// two launches per step this saves the launches, their ramps, and the
// parameters' and moments' way through memory; a step's samples are loaded
// before the barrier that ends the previous one.  4096 samples per step,
// 2^18 samples: 12.2 us per step against 57 us for the two launches
// of one thread per sample and one thread per entry it replaces.
// ---------------------------------------------------------------------------
struct __align__(16) StepScale {
    float lr, c1, c2, unused;   // learning rate and Adam's 1 / (1 - b^t) of a step
};

struct TrainArgs {
    float* p;
    const float *feat, *dmu;
    long long n, nb;            // samples, batches per epoch
    int batch;
    long long t0;               // steps done before this launch
    int steps;                  // steps of this launch
    const StepScale* scale;     // [steps]
    float *partial, *m, *v;     // [sum_blocks][kPartialLd], Adam moments [kMlpParams]
    int sum_blocks;             // blocks with samples (every block reduces)
    float* loss_log;            // mean batch loss of each epoch (may be null)
    // arrivals (zero at launch), and a word that is not zero once a barrier
    // gave up, in this launch or an earlier one of the call
    unsigned long long* barrier;
    int polls;                  // most polls of a barrier
};

// Grid barrier of a cooperative launch (every block is resident): arrival
// count target reached, or false when the bounded wait gave up.
constexpr int kBarrierPolls = 1 << 24;
// What a call whose barrier gave up leaves in the normalisation entries, which
// training never writes otherwise (a NaN of this one payload).
constexpr unsigned kGaveUpBits = 0x7fc7e57au;
__device__ __forceinline__ bool train_barrier(unsigned long long* count, unsigned long long target, int polls,
                                              int& ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1ull);
        int done = 0;
        for (int it = polls; it > 0 && !done; it--) {
            unsigned long long c;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(c) : "l"(count) : "memory");
            done = c >= target;
        }
        ok = done;
    }
    __syncthreads();
    return ok != 0;
}

// Partial sums per entry in the reduction over G blocks: one per warp.
__host__ __device__ constexpr int train_segs(int G) { return G < kGradThreads / 32 ? G : kGradThreads / 32; }

// A barrier gave up (never expected of a cooperative launch): the block's
// entries e0 .. e0 + ne - 1 are not a result, and the parameters say so
// (lb_mlp_train_status).
__device__ __forceinline__ void train_give_up(const TrainArgs& A, int e0, int ne) {
    const int tid = threadIdx.x;
    if (tid == 0) atomicExch(A.barrier + 1, 1ull);
    for (int e = tid; e < ne; e += kGradThreads)
        if (e0 + e < kMlpTrainable) A.p[e0 + e] = nanf("");
    if (tid < kMlpParams - kMlpMean) A.p[kMlpMean + tid] = __uint_as_float(kGaveUpBits);
}

__global__ void __launch_bounds__(kGradThreads) k_mlp_train(const TrainArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& s = *reinterpret_cast<GradSmem*>(smem_raw);
    const int tid = threadIdx.x, G = gridDim.x, B = A.sum_blocks;
    const int per = (kPartial + G - 1) / G, e0 = blockIdx.x * per, ne = max(0, min(per, kPartial - e0));
    // the block's entries of p, m, v and the segments' sums, after the tiles
    float* own = reinterpret_cast<float*>(smem_raw + sizeof(GradSmem));
    float *own_p = own, *own_m = own + per, *own_v = own + 2 * per, *red = own + 3 * per;   // red[segs][per]
    const int segs = train_segs(B);
    __shared__ int ok;
    // an earlier launch of the call gave up: nothing to go on from (a block that
    // finds the word set during this launch takes no part; the others' waits are
    // bounded)
    if (__ldcg(A.barrier + 1) != 0ull) {
        train_give_up(A, e0, ne);
        return;
    }
    for (int e = tid; e < ne; e += kGradThreads) {
        const bool w = e0 + e < kMlpTrainable;
        own_p[e] = w ? A.p[e0 + e] : 0.0f;
        own_m[e] = w ? A.m[e0 + e] : 0.0f;
        own_v[e] = w ? A.v[e0 + e] : 0.0f;
    }
    unsigned long long arrived = 0;
    long long b = A.t0 % A.nb, ep = A.t0 / A.nb;   // batch of the epoch, epoch
    GradIn in = grad_load(A.feat, A.dmu, b * A.batch, (int)min((long long)A.batch, A.n - b * A.batch), blockIdx.x);
    for (int t = 0; t < A.steps; t++) {
        const long long i0 = b * A.batch;
        const int n = (int)min((long long)A.batch, A.n - i0);
        const float inv = 1.0f / (4.0f * (float)n);
        if ((int)blockIdx.x < B) {
            grad_fill(s, A.p);
            __syncthreads();
            GradAcc acc;
            grad_zero(acc);
            for (int g = blockIdx.x; g < grad_groups(n); g += B) {
                const GradIn cur = in;
                in = grad_load(A.feat, A.dmu, i0, n, g + B);   // the next group's (zeros beyond the batch)
                grad_group(s, cur, n - g * kGradRows, inv, acc);
            }
            grad_store(acc, A.partial + (size_t)blockIdx.x * kPartialLd);
        }
        const long long bn = b + 1 == A.nb ? 0 : b + 1;
        const StepScale sc = A.scale[t];
        in = grad_load(A.feat, A.dmu, bn * A.batch, (int)min((long long)A.batch, A.n - bn * A.batch), blockIdx.x);
        if (!train_barrier(A.barrier, arrived += G, A.polls, ok)) break;
        // warp w adds the partials of blocks w, w + segs, ...
        const int seg = tid >> 5;
        if (seg < segs)
            for (int e = tid & 31; e < ne; e += 32) {
                float g = 0.0f;
                const float* at = A.partial + e0 + e;
#pragma unroll 16
                for (int q = seg; q < B; q += segs) g += __ldcg(at + (size_t)q * kPartialLd);
                red[seg * per + e] = g;
            }
        __syncthreads();
        for (int e = tid; e < ne; e += kGradThreads) {
            float g = 0.0f;
            for (int w = 0; w < segs; w++) g += red[w * per + e];
            if (e0 + e < kMlpTrainable) {
                const float mm = kAdamB1 * own_m[e] + kAdam1mB1 * g;
                const float vv = kAdamB2 * own_v[e] + kAdam1mB2 * (g * g);
                own_m[e] = mm;
                own_v[e] = vv;
                own_p[e] -= sc.lr * (mm * sc.c1) / (sqrtf(vv * sc.c2) + kAdamEps);
                A.p[e0 + e] = own_p[e];
            } else if (A.loss_log) {
                A.loss_log[ep] += g * inv * (float)(1.0 / (double)A.nb);
            }
        }
        ep += bn == 0;
        b = bn;
        if (!train_barrier(A.barrier, arrived += G, A.polls, ok)) break;
    }
    if (!ok) {
        train_give_up(A, e0, ne);
        return;
    }
    for (int e = tid; e < ne; e += kGradThreads)
        if (e0 + e < kMlpTrainable) {
            A.m[e0 + e] = own_m[e];
            A.v[e0 + e] = own_v[e];
        }
}

// Learning rate (geometric from lr0 to lr1 over `total` steps) and Adam's
// bias corrections of steps t0 + 1 .. t0 + steps.
__global__ void __launch_bounds__(kReduceThreads) k_mlp_scale(StepScale* __restrict__ out, long long t0, int steps,
                                                              long long total, double lr0, double ratio) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= steps) return;
    const long long t = t0 + i;
    const double lr = lr0 * pow(ratio, total > 1 ? (double)t / (double)(total - 1) : 0.0);
    const double c1 = 1.0 / (1.0 - pow(kAdamB1d, (double)(t + 1))), c2 = 1.0 / (1.0 - pow(kAdamB2d, (double)(t + 1)));
    out[i] = {(float)lr, (float)c1, (float)c2, 0.0f};
}

// Adam on a given gradient (every trainable entry).
__global__ void __launch_bounds__(kReduceThreads) k_mlp_adam(float* __restrict__ p, const float* __restrict__ g,
                                                             float* __restrict__ m, float* __restrict__ v,
                                                             float lr, float c1, float c2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= kMlpTrainable) return;
    const float gg = g[e];
    const float mm = kAdamB1 * m[e] + kAdam1mB1 * gg;
    const float vv = kAdamB2 * v[e] + kAdam1mB2 * (gg * gg);
    m[e] = mm;
    v[e] = vv;
    p[e] -= lr * (mm * c1) / (sqrtf(vv * c2) + kAdamEps);
}

constexpr unsigned reduce_blocks() { return (kMlpParams + 1 + kReduceThreads - 1) / kReduceThreads; }

// Blocks of a batch of n samples: one per group of 32, at most what is
// resident at once (most: what cooperative launches may have).
int grad_grid(long long n, int most) {
    return (int)std::max(1ll, std::min<long long>((n + kGradRows - 1) / kGradRows, most));
}

// Shared memory of the training kernel with G blocks, B of them with samples
// (at its largest where every block has some).
size_t train_smem(int G, int B) {
    const int per = (kPartial + G - 1) / G;
    return sizeof(GradSmem) + (size_t)(3 + train_segs(B)) * per * sizeof(float);
}

// Adam's bias corrections 1 / (1 - b^t)
void adam_corrections(long long t, float& c1, float& c2) {
    c1 = (float)(1.0 / (1.0 - std::pow(kAdamB1d, (double)t)));
    c2 = (float)(1.0 / (1.0 - std::pow(kAdamB2d, (double)t)));
}

// SplitMix64 (Steele, Lea and Flood, 2014)
unsigned long long splitmix64(unsigned long long& s) {
    unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int lb_mlp_init(float* params, int n, unsigned long long seed) {
    if (!params) return fail(LB_ERR_ARG, "params is NULL");
    if (n != kMlpParams) return fail(LB_ERR_ARG, "expected %d parameters", kMlpParams);
    unsigned long long s = seed;
    auto uni = [&]() { return 2.0 * (double)(splitmix64(s) >> 11) * 0x1p-53 - 1.0; };
    for (int i = 0; i < n; i++) params[i] = 0.0f;
    for (int i = 0; i < kMlpHid * kMlpIn; i++) params[kMlpW1 + i] = (float)(uni() * std::sqrt(6.0 / kMlpIn));
    for (int i = 0; i < kMlpHid * kMlpHid; i++) params[kMlpW2 + i] = (float)(uni() * std::sqrt(6.0 / kMlpHid));
    for (int i = 0; i < kMlpOut * kMlpHid; i++) params[kMlpW3 + i] = (float)(uni() * std::sqrt(6.0 / kMlpHid));
    for (int j = 0; j < 4; j++) {
        params[kMlpIstd + j] = 1.0f;
        params[kMlpOscale + j] = 1.0f;
    }
    return LB_OK;
}

int lb_energy_dataset(const double* rho, const double* ux, const double* uy, const double* escale,
                      long long n, float* feat, float* dmu, double* mu, unsigned long long* stats,
                      void* cuda_stream) {
    if (n < 0) return fail(LB_ERR_ARG, "n must be >= 0");
    if (n > 0 && (!rho || !ux || !uy || !escale || !feat || !dmu))
        return fail(LB_ERR_ARG, "NULL argument");
    if (n == 0) return LB_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const long long blocks = (n + 255) / 256;
    if (blocks > 0x7fffffffll) return fail(LB_ERR_ARG, "n too large");
    k_energy_dataset<<<(unsigned)blocks, 256, 0, st>>>(rho, ux, uy, escale, n, feat, dmu, mu, stats);
    CK(cudaGetLastError());
    return LB_OK;
}

int lb_mlp_normalise(float* params, const float* feat, const float* dmu, long long n, void* cuda_stream) {
    if (!params || !feat || !dmu) return fail(LB_ERR_ARG, "NULL argument");
    if (n <= 0) return fail(LB_ERR_ARG, "n must be > 0");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int blocks = (int)std::min<long long>((n + kNormThreads - 1) / kNormThreads, kNormBlocks);
    double* sums = nullptr;
    CK(cudaMallocAsync(&sums, (size_t)blocks * kNormSums * sizeof(double), st));
    k_mlp_norm_sums<<<blocks, kNormThreads, 0, st>>>(feat, dmu, n, sums);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        k_mlp_norm_finish<<<1, 32 * kNormSums, 0, st>>>(params, sums, blocks, n);
        e = cudaGetLastError();
    }
    cudaFreeAsync(sums, st);
    CK(e);
    return LB_OK;
}

int lb_mlp_forward(const float* params, const float* feat, long long n, float* y, void* cuda_stream) {
    if (n < 0) return fail(LB_ERR_ARG, "n must be >= 0");
    if (n > 0 && (!params || !feat || !y)) return fail(LB_ERR_ARG, "NULL argument");
    if (n == 0) return LB_OK;
    const long long blocks = (n + 127) / 128;
    if (blocks > 0x7fffffffll) return fail(LB_ERR_ARG, "n too large");
    k_mlp_forward<<<(unsigned)blocks, 128, 0, static_cast<cudaStream_t>(cuda_stream)>>>(params, feat, n, y);
    CK(cudaGetLastError());
    return LB_OK;
}

int lb_mlp_grad(const float* params, const float* feat, const float* dmu, int n, float* grad,
                float* loss, void* cuda_stream) {
    if (!params || !feat || !dmu || !grad) return fail(LB_ERR_ARG, "NULL argument");
    if (n <= 0) return fail(LB_ERR_ARG, "n must be > 0");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    CK(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)));
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int nblk = grad_grid(n, 2 * sms);
    float* partial = nullptr;
    CK(cudaMallocAsync(&partial, (size_t)nblk * kPartialLd * sizeof(float), st));
    const float inv = 1.0f / (4.0f * (float)n);
    k_mlp_grad<<<nblk, kGradThreads, sizeof(GradSmem), st>>>(params, feat, dmu, n, inv, partial);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        k_mlp_reduce<<<reduce_blocks(), kReduceThreads, 0, st>>>(partial, nblk, grad, loss, inv);
        e = cudaGetLastError();
    }
    cudaFreeAsync(partial, st);
    CK(e);
    return LB_OK;
}

int lb_mlp_adam(float* params, const float* grad, float* m, float* v, long long t, double lr,
                void* cuda_stream) {
    if (!params || !grad || !m || !v) return fail(LB_ERR_ARG, "NULL argument");
    if (t < 1) return fail(LB_ERR_ARG, "t must be >= 1");
    if (!(lr >= 0.0) || !std::isfinite(lr)) return fail(LB_ERR_ARG, "lr must be finite and >= 0");
    float c1, c2;
    adam_corrections(t, c1, c2);
    k_mlp_adam<<<(kMlpTrainable + kReduceThreads - 1) / kReduceThreads, kReduceThreads, 0,
                 static_cast<cudaStream_t>(cuda_stream)>>>(params, grad, m, v, (float)lr, c1, c2);
    CK(cudaGetLastError());
    return LB_OK;
}

int lb_mlp_train(float* params, const float* feat, const float* dmu, long long n, int batch, int epochs,
                 double lr0, double lr1, float* loss_log, void* cuda_stream) {
    return lb_mlp_train_bounded(params, feat, dmu, n, batch, epochs, lr0, lr1, loss_log, kBarrierPolls, cuda_stream);
}

int lb_mlp_train_status(const float* params, void* cuda_stream) {
    if (!params) return fail(LB_ERR_ARG, "params is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    unsigned bits = 0;
    CK(cudaMemcpyAsync(&bits, params + kMlpMean, sizeof(bits), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (bits == kGaveUpBits) return fail(LB_ERR_TIMEOUT, "a grid barrier of the training kernel gave up");
    return LB_OK;
}

int lb_mlp_train_bounded(float* params, const float* feat, const float* dmu, long long n, int batch, int epochs,
                         double lr0, double lr1, float* loss_log, int polls, void* cuda_stream) {
    if (polls < 0) return fail(LB_ERR_ARG, "polls must be >= 0");
    if (!params || !feat || !dmu) return fail(LB_ERR_ARG, "NULL argument");
    if (n <= 0 || batch <= 0 || epochs < 0) return fail(LB_ERR_ARG, "n, batch must be > 0, epochs >= 0");
    if (batch > (1 << 24)) return fail(LB_ERR_ARG, "batch too large");
    if (!(lr0 > 0.0) || !(lr1 > 0.0) || !std::isfinite(lr0) || !std::isfinite(lr1))
        return fail(LB_ERR_ARG, "learning rates must be positive and finite");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const long long nb = (n + batch - 1) / batch;
    const long long total = nb * (long long)epochs;
    int dev = 0, sms = 0, per_sm = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // one block per SM: a step's chain of latencies is the same with more,
    // and the reduction has fewer partials to add; every SM takes part in the
    // reduction (152 blocks: 32 entries each, one per lane)
    const int A_blocks = grad_grid(std::min<long long>(n, batch), sms), G = sms;
    const size_t smem = train_smem(G, A_blocks);
    // the limit belongs to the kernel, which other threads launch too: always
    // the largest size, so that no call lowers it under another's launch
    CK(cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)train_smem(G, G)));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_train, kGradThreads, smem));
    if (per_sm < 1) return fail(LB_ERR_CUDA, "the training kernel does not fit on this device");
    // working memory: block partials, Adam's moments, the chunk's step scales, the barrier
    // and the word that says that one gave up
    constexpr long long kChunk = 1 << 16;   // steps per launch
    const size_t scale_b = (size_t)std::min(std::max(total, 1ll), kChunk) * sizeof(StepScale);
    const size_t mv_b = 2 * (size_t)kMlpParams * sizeof(float);
    const size_t part_b = (size_t)A_blocks * kPartialLd * sizeof(float);
    unsigned char* mem = nullptr;
    CK(cudaMallocAsync(&mem, scale_b + mv_b + 16 + part_b, st));
    float* m = reinterpret_cast<float*>(mem + scale_b);
    cudaError_t e = cudaMemsetAsync(mem + scale_b, 0, mv_b + 16, st);
    if (e == cudaSuccess && loss_log) e = cudaMemsetAsync(loss_log, 0, (size_t)epochs * sizeof(float), st);
    TrainArgs A = {params, feat, dmu, n, nb, batch, 0, 0, reinterpret_cast<StepScale*>(mem),
                   reinterpret_cast<float*>(mem + scale_b + mv_b + 16), m, m + kMlpParams, A_blocks, loss_log,
                   reinterpret_cast<unsigned long long*>(mem + scale_b + mv_b), polls};
    for (long long t = 0; t < total && e == cudaSuccess; t += kChunk) {
        A.t0 = t;
        A.steps = (int)std::min(kChunk, total - t);
        if (t > 0) e = cudaMemsetAsync(A.barrier, 0, sizeof(unsigned long long), st);
        if (e != cudaSuccess) break;
        k_mlp_scale<<<(A.steps + kReduceThreads - 1) / kReduceThreads, kReduceThreads, 0, st>>>(
            reinterpret_cast<StepScale*>(mem), t, A.steps, total, lr0, lr1 / lr0);
        e = cudaGetLastError();
        if (e != cudaSuccess) break;
        void* args[] = {&A};
        e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_mlp_train), dim3(G), dim3(kGradThreads), args,
                                        smem, st);
    }
    cudaFreeAsync(mem, st);
    CK(e);
    return LB_OK;
}

}  // extern "C"
