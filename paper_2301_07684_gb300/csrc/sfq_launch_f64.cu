// Launchers of the plain binary64 path.
#include "sfq_launch.cuh"

namespace sfq {
cudaError_t launch_rate_f64(const RateLaunch &L, bool pair) { return launch_rate_t<double>(L, pair); }
cudaError_t launch_sample_f64(const SampleLaunch &L, bool pair) { return launch_sample_t<double>(L, pair); }
cudaError_t launch_uniforms_f64(int64_t n, const uint64_t *id, uint32_t step, uint32_t tag, uint64_t seed, void *u,
                                cudaStream_t s, int grid, int block) {
    return launch_uniforms_t<double>(n, id, step, tag, seed, u, s, grid, block);
}
cudaError_t launch_step_f64(const StepLaunch &L) {
    return L.ctx->inv_tr > 0 ? launch_step_trunc_f64(L) : launch_step_t<double, false>(L);
}
cudaError_t prepare_step_f64() {
    const cudaError_t e = prepare_step_t<double, false>();
    return e == cudaSuccess ? prepare_step_trunc_f64() : e;
}
cudaError_t launch_fused_f64(const StepLaunch &L, uint32_t nsteps) {
    return L.ctx->inv_tr > 0 ? launch_fused_trunc_f64(L, nsteps) : launch_fused_t<double, false>(L, nsteps);
}
cudaError_t launch_push_f64(const StepLaunch &L, double dt) { return launch_push_t<double>(L, dt); }
}  // namespace sfq
