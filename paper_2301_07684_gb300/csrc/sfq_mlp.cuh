// sfq_mlp.cuh -- what the translation units of the learned surrogate share: the object, the
// network's layout, features and activations, and the forward pass of one sample on the CUDA
// cores (its two kernels are compiled apart, in parallel: each unrolls the whole network).
#pragma once
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "sfq_internal.h"
#include "sfq_kernels.cuh"

struct sfq_mlp {
    sfq_ctx *ctx;
    int kind;                         // 0: photon emission (Eq. again), 1: pair creation (Eq. again_pp)
    float *params, *m, *v;            // binary32 master parameters, Adam moments
    uint8_t *flags;                   // fallback cells (NCELL bytes)
    float *cell_err;                  // per-cell calibration error (NCELL floats)
    int64_t adam_t;
    int calibrated;
};

namespace sfq {
namespace mlp {

constexpr int H = 64;
constexpr int NP = 8577;
constexpr int NPS = 8592;          // row stride of the gradient partials (16-byte aligned rows)
constexpr int O_W1 = 0, O_B1 = 128, O_W2 = 192, O_B2 = 4288, O_W3 = 4352, O_B3 = 8448, O_W4 = 8512, O_B4 = 8576;
constexpr float C_CHI = -1.1512925464970229f;    // (ln 1e-3 + ln 100) / 2
constexpr float S_CHI = 5.7564627324851140f;     // (ln 100 - ln 1e-3) / 2
constexpr float L_SCALE = 0.125f;
constexpr float CHI_LO = 1e-3f, CHI_HI = 100.0f;
constexpr int NCX = 64, NCU = 64, NCELL = NCX * NCU;   // calibration cells in (ln chi, u)

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float qz(float x, bool q) { return q ? bf16r(x) : x; }
__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.0f + __expf(-z)); }
// SiLU of the inference paths (tensor-core kernel, SIMT reference and calibration) with one
// special-function instruction: z sigma(z) = h (1 + tanh h), h = z / 2, from
// sigma(z) = (1 + tanh(z/2)) / 2.  tanh.approx.f32 has a relative error below 2^-10.987
// (PTX ISA), which is below the bfloat16 rounding the activations then get (2^-9).
// `h` is passed in: the callers form it as 0.5 z + 0.5 b in one fma from halved biases.
__device__ __forceinline__ float silu_h(float h) {
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(h));
    return fmaf(h, t, h);
}
__device__ __forceinline__ float dsilu(float z) {
    const float s = __fdividef(1.0f, 1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}
// What distinguishes the two samplers the network can stand for.  Photon emission: input
// u = r, chi in [1e-3, 100], sampler variable ln w-bar.  Pair creation: input u = |r'| =
// |2r - 1|, chi in [0.1, 100], sampler variable ln(-ln y) with y = 1 - v-bar (Eq.
// again_pp): -ln y ~ v-bar ~ u as u -> 0, so both variables minus ln u stay smooth at
// u -> 0, and y = exp(-u e^network) never exceeds 1.  The network output is always the
// sampler variable minus ln u.
struct Kind {
    float c_chi, inv_s_chi, chi_lo, chi_hi;
    int pair;
};
constexpr float P_C_CHI = 1.1512925464970229f;      // (ln 0.1 + ln 100) / 2
constexpr float P_S_CHI = 3.4538776394910684f;      // (ln 100 - ln 0.1) / 2
constexpr float P_CHI_LO = 0.1f, P_CHI_HI = 100.0f;
inline Kind kind_of(int pair) {
    return pair ? Kind{P_C_CHI, 1.0f / P_S_CHI, P_CHI_LO, P_CHI_HI, 1} : Kind{C_CHI, 1.0f / S_CHI, CHI_LO, CHI_HI, 0};
}
__device__ __forceinline__ void features(const Kind &K, float chi, float u, float &x1, float &x2) {
    x1 = (logf(chi) - K.c_chi) * K.inv_s_chi;
    x2 = -log1pf(-u) * L_SCALE - 1.0f;
}
// network output + offset = the sampler's variable (ln w-bar or ln(-ln y))
__device__ __forceinline__ float out_offset(const Kind &, float u) { return logf(u); }
__device__ __forceinline__ int cell_of(const Kind &K, float chi, float u) {
    const float t = (logf(chi) - logf(K.chi_lo)) * (float)NCX / (logf(K.chi_hi) - logf(K.chi_lo));
    int cx = (int)t, cu = (int)(u * (float)NCU);
    cx = cx < 0 ? 0 : (cx >= NCX ? NCX - 1 : cx);
    cu = cu < 0 ? 0 : (cu >= NCU ? NCU - 1 : cu);
    return cx * NCU + cu;
}

// ---------------------------------------------------------------------------------------
// SIMT forward of one sample with the weights in shared memory (calibration and the
// reference inference path).  Same rounding as the tensor-core kernel.
struct SimtW {
    float w1[H * 2], b1[H], w2[H * H], b2[H], w3[H * H], b3[H], w4[H], b4;
};
__device__ __forceinline__ void stage_simt(SimtW &W, const float *P) {
    for (int e = threadIdx.x; e < H * H; e += blockDim.x) {
        W.w2[e] = bf16r(P[O_W2 + e]);
        W.w3[e] = bf16r(P[O_W3 + e]);
    }
    for (int e = threadIdx.x; e < H; e += blockDim.x) {
        W.w1[2 * e] = bf16r(P[O_W1 + 2 * e]);
        W.w1[2 * e + 1] = bf16r(P[O_W1 + 2 * e + 1]);
        W.b1[e] = P[O_B1 + e];
        W.b2[e] = P[O_B2 + e];
        W.b3[e] = P[O_B3 + e];
        W.w4[e] = bf16r(P[O_W4 + e]);
    }
    if (threadIdx.x == 0) W.b4 = P[O_B4];
}
__device__ __forceinline__ float forward_simt(const SimtW &W, const Kind &K, float chi, float u) {
    float x1, x2;
    features(K, chi, u, x1, x2);
    float a[H], b[H];
#pragma unroll
    for (int j = 0; j < H; ++j)
        a[j] = bf16r(silu_h(0.5f * fmaf(W.w1[2 * j], x1, fmaf(W.w1[2 * j + 1], x2, W.b1[j]))));
    // layers 2 and 3: the products summed in binary32 (the tensor cores' order differs), then
    // h = (sum + b) / 2 as the tensor-core epilogue forms it
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < H; ++k) acc = fmaf(a[k], W.w2[j * H + k], acc);
        b[j] = bf16r(silu_h(fmaf(0.5f, acc, 0.5f * W.b2[j])));
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < H; ++k) acc = fmaf(b[k], W.w3[j * H + k], acc);
        a[j] = bf16r(silu_h(fmaf(0.5f, acc, 0.5f * W.b3[j])));
    }
    float y = W.b4;
#pragma unroll
    for (int k = 0; k < H; ++k) y = fmaf(a[k], W.w4[k], y);
    return y;
}

cudaError_t launch_predict(const float *P, const Kind &K, int64_t n, const float *chi, const float *u, float *lnw,
                           int grid, cudaStream_t s);
cudaError_t launch_calibrate(const float *P, const Kind &K, const float *inv, float tol_u, uint8_t *flags,
                             float *cell_err, cudaStream_t s);
cudaError_t launch_plain_targets(const float *inv, const Kind &K, int64_t n, const float *chi, const float *u,
                                 float *lnw, int grid, cudaStream_t s);

}  // namespace mlp
}  // namespace sfq
