// Calibration of the surrogate against the plain fitted sampler, and that sampler's values as
// training targets (sfq_mlp_calibrate, sfq_mlp_plain_targets).
#include "sfq_mlp.cuh"

namespace sfq {
namespace mlp {

// ---------------------------------------------------------------------------------------
// Calibration: per cell, the largest |u_net - u| implied by the network's ln w-bar against
// the plain sampler's, |d ln w| / (d ln w / du), over 8 x 8 points of the cell.
// The plain fitted sampler's variable: ln w-bar (photon) or ln(-ln y) (pair, u = |r'|).
__device__ __forceinline__ float plain_lnw(const Kind &K, const float *inv, float chi, float u) {
    bool oor = false;
    if (K.pair) {
        // -ln y from v-bar = 1 - y where y is near 1; where 1 - y falls below the binary32
        // table's resolution (|r'| below about 1e-5) the variable is unresolved: NaN
        const float y = pair_y<float>(inv, chi, u, oor);
        const float v = 1.0f - y;
        if (!(v >= 1.52587890625e-05f)) return __int_as_float(0x7fffffff);    // 2^-16
        return logf(y < 0.5f ? -logf(y) : -log1pf(-v));
    }
    const float s = photon_s<float>(inv, chi, u, oor);
    return (logf(2.0f * s) - logf(3.0f * chi)) * (1.0f / 3.0f);
}
__global__ void __launch_bounds__(64) calibrate_kernel(const float *__restrict__ P, const Kind K,
                                                       const float *__restrict__ inv, float tol_u,
                                                       uint8_t *__restrict__ flags, float *__restrict__ cell_err) {
    __shared__ SimtW W;
    __shared__ float red[64];
    stage_simt(W, P);
    __syncthreads();
    const int cell = blockIdx.x, cx = cell / NCU, cu = cell % NCU;
    const int pa = threadIdx.x >> 3, pb = threadIdx.x & 7;
    const float lo = logf(K.chi_lo), span = logf(K.chi_hi) - logf(K.chi_lo);
    const float chi = expf(lo + span * ((float)cx + ((float)pa + 0.5f) * 0.125f) / (float)NCX);
    const float u = ((float)cu + ((float)pb + 0.5f) * 0.125f) / (float)NCU;
    const float ln_net = forward_simt(W, K, chi, u) + out_offset(K, u);
    const float ln_p = plain_lnw(K, inv, chi, u);
    const float h = 1.0f / (float)(NCU * 64);
    // |d ln w / du| (both sampler variables rise with u)
    const float dlnw_du = fabsf(plain_lnw(K, inv, chi, u + h) - plain_lnw(K, inv, chi, u - h)) / (2.0f * h);
    float e = fabsf(ln_net - ln_p) / fmaxf(dlnw_du, 1e-30f);
    if (!(e == e)) e = 1e30f;
    red[threadIdx.x] = e;
    __syncthreads();
    for (int o = 32; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cell_err[cell] = red[0];
        flags[cell] = red[0] > tol_u ? 1 : 0;
    }
}

// ln w-bar of the plain fitted sampler (training targets without the oracle).
__global__ void plain_targets_kernel(const float *__restrict__ inv, const Kind K, int64_t n,
                                     const float *__restrict__ chi, const float *__restrict__ u,
                                     float *__restrict__ lnw) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        lnw[i] = plain_lnw(K, inv, chi[i], u[i]);
}

cudaError_t launch_calibrate(const float *P, const Kind &K, const float *inv, float tol_u, uint8_t *flags,
                             float *cell_err, cudaStream_t s) {
    calibrate_kernel<<<NCELL, 64, 0, s>>>(P, K, inv, tol_u, flags, cell_err);
    return cudaGetLastError();
}
cudaError_t launch_plain_targets(const float *inv, const Kind &K, int64_t n, const float *chi, const float *u,
                                 float *lnw, int grid, cudaStream_t s) {
    plain_targets_kernel<<<grid, 256, 0, s>>>(inv, K, n, chi, u, lnw);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace sfq
