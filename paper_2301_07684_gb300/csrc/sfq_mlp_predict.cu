// The surrogate's forward pass on the CUDA cores (sfq_mlp_predict_lnw).
#include "sfq_mlp.cuh"

namespace sfq {
namespace mlp {

__global__ void __launch_bounds__(128) predict_kernel(const float *__restrict__ P, const Kind K, int64_t n,
                                                      const float *__restrict__ chi, const float *__restrict__ u,
                                                      float *__restrict__ lnw) {
    __shared__ SimtW W;
    stage_simt(W, P);
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float uu = u[i];
        lnw[i] = forward_simt(W, K, chi[i], uu) + out_offset(K, uu);
    }
}

cudaError_t launch_predict(const float *P, const Kind &K, int64_t n, const float *chi, const float *u, float *lnw,
                           int grid, cudaStream_t s) {
    predict_kernel<<<grid, 128, 0, s>>>(P, K, n, chi, u, lnw);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace sfq
