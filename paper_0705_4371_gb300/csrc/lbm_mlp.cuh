// lbm_mlp.cuh -- the 4-64-64-4 network that warm-starts the energy Newton
// solve (learned form).  Inputs: the site's features (rho, u_x, u_y,
// theta = 2E/rho - |u|^2), standardised; outputs: the scaled corrections
// (mu - mu0) / out_scale of the four Lagrange multipliers of
// ln(f*_i / W_i) = mu . (1, v_x, v_y, |v|^2) (Sec. 3.3) about the
// polynomial start point mu0 = (ln rho - 3/2 |u|^2, 3 u_x, 3 u_y, 0).
// ReLU hidden layers.
//
// Parameters: one FP32 vector (the master copy)
//   W1[64][4] b1[64] W2[64][64] b2[64] W3[4][64] b3[4] mean[4] inv_std[4]
//   out_scale[4]
// Evaluation is one warp per 32 sites on the tensor cores
// (mma.sync m16n8k16, BF16 operands, FP32 accumulation): the standardised
// inputs, the weights and the hidden activations are rounded to BF16 (round
// to nearest even), biases are added in FP32 (they initialise the
// accumulators).  The hidden layer's output fragments are re-packed in
// registers as the next layer's input fragments, so the activations never
// leave the registers.
#pragma once

#include <cstdint>

namespace lbm {

constexpr int kMlpIn = 4, kMlpHid = 64, kMlpOut = 4;
constexpr int kMlpW1 = 0;
constexpr int kMlpB1 = kMlpW1 + kMlpHid * kMlpIn;      // 256
constexpr int kMlpW2 = kMlpB1 + kMlpHid;               // 320
constexpr int kMlpB2 = kMlpW2 + kMlpHid * kMlpHid;     // 4416
constexpr int kMlpW3 = kMlpB2 + kMlpHid;               // 4480
constexpr int kMlpB3 = kMlpW3 + kMlpOut * kMlpHid;     // 4736
constexpr int kMlpMean = kMlpB3 + kMlpOut;             // 4740
constexpr int kMlpIstd = kMlpMean + kMlpIn;            // 4744
constexpr int kMlpOscale = kMlpIstd + kMlpIn;          // 4748
constexpr int kMlpParams = kMlpOscale + kMlpOut;       // 4752
constexpr int kMlpTrainable = kMlpMean;                // entries below this are trained

// The network's weights in mma fragment order (BF16 pairs), biases and
// normalisation, in shared memory.  [n-tile][k-step][lane] for W2,
// [k-step][lane] for W3 (outputs 4..7 of its n-tile are zero), [n-tile][lane]
// for W1 (its k-step has inputs 0..3; inputs 4..15 are zero).
struct MlpSmem {
    unsigned w1[8][32];
    uint2 w2[8][4][32];
    uint2 w3[4][32];
    float b1[kMlpHid], b2[kMlpHid], b3[8];
    float mean[kMlpIn], istd[kMlpIn], oscale[kMlpOut];
};

// Two FP32 values to a BF16 pair (round to nearest even); lo in the low half.
__device__ __forceinline__ unsigned bf16_pack(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
// The same after ReLU (max(x, 0)).
__device__ __forceinline__ unsigned bf16_pack_relu(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float bf16_lo(unsigned u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(unsigned u) { return __uint_as_float(u & 0xffff0000u); }

// D = A B + D, m16n8k16, BF16 A (row) and B (col), FP32 accumulators.
__device__ __forceinline__ void mma_bf16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                         unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Block-cooperative fill of the shared copy from the FP32 parameter vector
// (the caller synchronises before use).
__device__ __forceinline__ void mlp_fill(MlpSmem& s, const float* __restrict__ p) {
    const int tid = threadIdx.x, nt_ = blockDim.x;
    for (int e = tid; e < 8 * 32; e += nt_) {
        const int nt = e >> 5, lane = e & 31, g = lane >> 2, tig = lane & 3;
        const int n = 8 * nt + g, k = 2 * tig;
        s.w1[nt][lane] = tig < 2 ? bf16_pack(p[kMlpW1 + n * kMlpIn + k], p[kMlpW1 + n * kMlpIn + k + 1])
                                 : 0u;
    }
    for (int e = tid; e < 8 * 4 * 32; e += nt_) {
        const int nt = e >> 7, ks = (e >> 5) & 3, lane = e & 31, g = lane >> 2, tig = lane & 3;
        const float* row = p + kMlpW2 + (8 * nt + g) * kMlpHid + 16 * ks + 2 * tig;
        s.w2[nt][ks][lane] = make_uint2(bf16_pack(row[0], row[1]), bf16_pack(row[8], row[9]));
    }
    for (int e = tid; e < 4 * 32; e += nt_) {
        const int ks = e >> 5, lane = e & 31, g = lane >> 2, tig = lane & 3;
        if (g < kMlpOut) {
            const float* row = p + kMlpW3 + g * kMlpHid + 16 * ks + 2 * tig;
            s.w3[ks][lane] = make_uint2(bf16_pack(row[0], row[1]), bf16_pack(row[8], row[9]));
        } else {
            s.w3[ks][lane] = make_uint2(0u, 0u);
        }
    }
    for (int e = tid; e < kMlpHid; e += nt_) {
        s.b1[e] = p[kMlpB1 + e];
        s.b2[e] = p[kMlpB2 + e];
    }
    for (int e = tid; e < 8; e += nt_) s.b3[e] = e < kMlpOut ? p[kMlpB3 + e] : 0.0f;
    for (int e = tid; e < kMlpIn; e += nt_) {
        s.mean[e] = p[kMlpMean + e];
        s.istd[e] = p[kMlpIstd + e];
        s.oscale[e] = p[kMlpOscale + e];
    }
}

// Standardised features (FP32: (f - mean) * inv_std) rounded to two BF16
// pairs (inputs 0, 1 and 2, 3).
__device__ __forceinline__ void mlp_inputs(const MlpSmem& s, float f0, float f1, float f2, float f3,
                                           unsigned& p01, unsigned& p23) {
    p01 = bf16_pack((f0 - s.mean[0]) * s.istd[0], (f1 - s.mean[1]) * s.istd[1]);
    p23 = bf16_pack((f2 - s.mean[2]) * s.istd[2], (f3 - s.mean[3]) * s.istd[3]);
}

// Forward pass of one 16-row tile (rows r0 = g and r0 + 8 of the fragment
// layout, g = lane / 4): a0, a1 the standardised inputs 2 tig, 2 tig + 1 of
// the two rows (zero for tig >= 2).  yc: output 2 tig + j of row r0 in
// register j, of row r0 + 8 in register 2 + j (lanes with tig < 2).  Every
// lane of the warp must call it.  CAP: also store the hidden activations
// (BF16 values, after ReLU) of the two rows at h1, h2 (rows of stride ld).
template <bool CAP>
__device__ __forceinline__ void mlp_tile_forward(const MlpSmem& s, unsigned a0, unsigned a1, float* yc,
                                                 int r0 = 0, float* h1 = nullptr, float* h2 = nullptr, int ld = 0) {
    const int lane = threadIdx.x & 31, tig = lane & 3, r1 = r0 + 8;
    // layer 1; its n-tiles 2j, 2j+1 form k-step j of layer 2
    unsigned A2[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; nt++) {
        const float bl = s.b1[8 * nt + 2 * tig], bh = s.b1[8 * nt + 2 * tig + 1];
        float c[4] = {bl, bh, bl, bh};
        mma_bf16(c, a0, a1, 0u, 0u, s.w1[nt][lane], 0u);
        const unsigned u0 = bf16_pack_relu(c[0], c[1]), u1 = bf16_pack_relu(c[2], c[3]);
        A2[nt >> 1][(nt & 1) * 2 + 0] = u0;
        A2[nt >> 1][(nt & 1) * 2 + 1] = u1;
        if constexpr (CAP) {
            const int col = 8 * nt + 2 * tig;
            h1[r0 * ld + col] = bf16_lo(u0);
            h1[r0 * ld + col + 1] = bf16_hi(u0);
            h1[r1 * ld + col] = bf16_lo(u1);
            h1[r1 * ld + col + 1] = bf16_hi(u1);
        }
    }
    // layers 2 and 3: W of layer 2's accumulators at a time take their k-steps
    // side by side (each k-step of one waits for its previous one; all eight
    // where a block's two warps are alone with the chain, CAP), and each pair
    // of layer-2 n-tiles is one layer-3 k-step
    constexpr int W = CAP ? 8 : 2;
    yc[0] = yc[2] = s.b3[2 * tig];
    yc[1] = yc[3] = s.b3[2 * tig + 1];
#pragma unroll
    for (int n0 = 0; n0 < 8; n0 += W) {
        float c[W][4];
#pragma unroll
        for (int q = 0; q < W; q++) {
            const int col = 8 * (n0 + q) + 2 * tig;
            c[q][0] = c[q][2] = s.b2[col];
            c[q][1] = c[q][3] = s.b2[col + 1];
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int q = 0; q < W; q++) {
                const uint2 b = s.w2[n0 + q][j][lane];
                mma_bf16(c[q], A2[j][0], A2[j][1], A2[j][2], A2[j][3], b.x, b.y);
            }
#pragma unroll
        for (int q = 0; q < W; q += 2) {
            unsigned A3[4];
#pragma unroll
            for (int hh = 0; hh < 2; hh++) {
                const unsigned u0 = bf16_pack_relu(c[q + hh][0], c[q + hh][1]);
                const unsigned u1 = bf16_pack_relu(c[q + hh][2], c[q + hh][3]);
                A3[2 * hh] = u0;
                A3[2 * hh + 1] = u1;
                if constexpr (CAP) {
                    const int col = 8 * (n0 + q + hh) + 2 * tig;
                    h2[r0 * ld + col] = bf16_lo(u0);
                    h2[r0 * ld + col + 1] = bf16_hi(u0);
                    h2[r1 * ld + col] = bf16_lo(u1);
                    h2[r1 * ld + col + 1] = bf16_hi(u1);
                }
            }
            const uint2 b = s.w3[(n0 + q) / 2][lane];
            mma_bf16(yc, A3[0], A3[1], A3[2], A3[3], b.x, b.y);
        }
    }
}

// Forward pass of the network for the warp's 32 sites, lane l holding site
// l: inputs (p01, p23) from mlp_inputs, outputs y[0..3].  Every lane of the
// warp must call it (lanes without a site pass zeros and ignore y).
__device__ __forceinline__ void mlp_warp_forward(const MlpSmem& s, unsigned p01, unsigned p23, float* y) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int m = 0; m < 2; m++) {
        // rows r0, r1 of this 16-site tile; input columns 2 tig, 2 tig + 1
        const int r0 = 16 * m + g, r1 = r0 + 8;
        const unsigned x0lo = __shfl_sync(FULL, p01, r0), x0hi = __shfl_sync(FULL, p23, r0);
        const unsigned x1lo = __shfl_sync(FULL, p01, r1), x1hi = __shfl_sync(FULL, p23, r1);
        const unsigned a0 = tig == 0 ? x0lo : (tig == 1 ? x0hi : 0u);
        const unsigned a1 = tig == 0 ? x1lo : (tig == 1 ? x1hi : 0u);
        float yc[4];
        mlp_tile_forward<false>(s, a0, a1, yc);
        // output j of tile row r sits in lane 4 (r mod 8) + j / 2, register
        // (j mod 2) (+2 for rows 8..15): bring it to lane 16 m + r
#pragma unroll
        for (int j = 0; j < kMlpOut; j++) {
            const int src = 4 * (lane & 7) + (j >> 1);
            const float lo = __shfl_sync(FULL, yc[j & 1], src);
            const float hi = __shfl_sync(FULL, yc[2 + (j & 1)], src);
            if ((lane >> 4) == m) y[j] = (lane & 8) ? hi : lo;
        }
    }
}

// The network as the collide kernels hold it: the biases also as
// accumulator fragments (quad t of n-tile nt: columns 8 nt + 2 t, + 1 of both
// row halves).
struct MlpSmemQ : MlpSmem {
    float4 q1[8][4], q2[8][4];
};

__device__ __forceinline__ void mlp_fill_quads(MlpSmemQ& s, const float* __restrict__ p) {
    for (int e = threadIdx.x; e < 32; e += blockDim.x) {
        const int nt = e >> 2, t = e & 3, c = 8 * nt + 2 * t;
        s.q1[nt][t] = make_float4(p[kMlpB1 + c], p[kMlpB1 + c + 1], p[kMlpB1 + c], p[kMlpB1 + c + 1]);
        s.q2[nt][t] = make_float4(p[kMlpB2 + c], p[kMlpB2 + c + 1], p[kMlpB2 + c], p[kMlpB2 + c + 1]);
    }
}

// D = A B + C, as mma_bf16, with an accumulator input of its own.
__device__ __forceinline__ void mma_bf16_from(float* d, float4 c, unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                              unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c.x), "f"(c.y), "f"(c.z), "f"(c.w));
}

// Warm start of the energy Newton solve for the warp's 32 sites (lane l: one
// site's rho, u, 2E): the energy multiplier mu_3 of the network's prediction
// (mu_1 and mu_2 follow from it in closed form).  Lanes without a valid site
// and predictions that are not finite or implausibly large (some |mu| > 8)
// get the polynomial start, 0.  Every lane of the warp must call it.
// Bound by the tensor pipe: 88 MMAs per warp at 8.7 cycles each per SM
// quarter.  Both 16-site tiles of the warp take every weight fragment as it
// is read (one shared-memory read for two MMAs), the biases enter as the first
// MMA's accumulators without a move, and the routine is out of line: inlined
// in the update twice it spilled 860 bytes per thread.  2048 x 1024: the
// network's share of a step 119 -> 62 us.
static __device__ __noinline__ float mlp_start(const MlpSmemQ& s, float rho, float ux, float uy, float e2, bool valid) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = lane >> 2, tig = lane & 3;
    unsigned p01 = 0u, p23 = 0u;
    if (valid) mlp_inputs(s, rho, ux, uy, e2 / rho - ux * ux - uy * uy, p01, p23);
    unsigned a[2][2];   // input columns 2 tig, 2 tig + 1 of rows g and g + 8 of tile m
#pragma unroll
    for (int m = 0; m < 2; m++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int r = 16 * m + 8 * h + g;
            const unsigned lo = __shfl_sync(FULL, p01, r), hi = __shfl_sync(FULL, p23, r);
            a[m][h] = tig == 0 ? lo : (tig == 1 ? hi : 0u);
        }
    unsigned A2[2][4][4];
#pragma unroll
    for (int nt = 0; nt < 8; nt++) {
        const unsigned w = s.w1[nt][lane];
        const float4 b = s.q1[nt][tig];
#pragma unroll
        for (int m = 0; m < 2; m++) {
            float c[4];
            mma_bf16_from(c, b, a[m][0], a[m][1], 0u, 0u, w, 0u);
            A2[m][nt >> 1][(nt & 1) * 2 + 0] = bf16_pack_relu(c[0], c[1]);
            A2[m][nt >> 1][(nt & 1) * 2 + 1] = bf16_pack_relu(c[2], c[3]);
        }
    }
    float yc[2][4];
#pragma unroll
    for (int m = 0; m < 2; m++) {
        yc[m][0] = yc[m][2] = s.b3[2 * tig];
        yc[m][1] = yc[m][3] = s.b3[2 * tig + 1];
    }
#pragma unroll
    for (int jp = 0; jp < 4; jp++) {
        unsigned A3[2][4];
#pragma unroll
        for (int hh = 0; hh < 2; hh++) {
            const int nt = 2 * jp + hh;
            const float4 b = s.q2[nt][tig];
            float c[2][4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint2 w = s.w2[nt][j][lane];
#pragma unroll
                for (int m = 0; m < 2; m++) {
                    if (j == 0) mma_bf16_from(c[m], b, A2[m][j][0], A2[m][j][1], A2[m][j][2], A2[m][j][3], w.x, w.y);
                    else mma_bf16(c[m], A2[m][j][0], A2[m][j][1], A2[m][j][2], A2[m][j][3], w.x, w.y);
                }
            }
#pragma unroll
            for (int m = 0; m < 2; m++) {
                A3[m][2 * hh] = bf16_pack_relu(c[m][0], c[m][1]);
                A3[m][2 * hh + 1] = bf16_pack_relu(c[m][2], c[m][3]);
            }
        }
        const uint2 w = s.w3[jp][lane];
#pragma unroll
        for (int m = 0; m < 2; m++) mma_bf16(yc[m], A3[m][0], A3[m][1], A3[m][2], A3[m][3], w.x, w.y);
    }
    // outputs 1 .. 3 to the site's lane, as in mlp_warp_forward
    float y[kMlpOut];
#pragma unroll
    for (int j = 1; j < kMlpOut; j++) {
        const int src = 4 * (lane & 7) + (j >> 1);
#pragma unroll
        for (int m = 0; m < 2; m++) {
            const float lo = __shfl_sync(FULL, yc[m][j & 1], src);
            const float hi = __shfl_sync(FULL, yc[m][2 + (j & 1)], src);
            if ((lane >> 4) == m) y[j] = (lane & 8) ? hi : lo;
        }
    }
    const float c0 = 3.0f * ux + s.oscale[1] * y[1], c1 = 3.0f * uy + s.oscale[2] * y[2], c2 = s.oscale[3] * y[3];
    return valid && fabsf(c0) <= 8.0f && fabsf(c1) <= 8.0f && fabsf(c2) <= 8.0f ? c2 : 0.0f;   // (false for NaN)
}

}  // namespace lbm
