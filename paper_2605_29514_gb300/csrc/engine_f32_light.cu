// Complex64 instantiations of the round and adjoint kernels with 256 threads and two
// CTAs per SM.
#define STN_CTA_THREADS 256
#include "engine_kernels.cuh"

namespace stn {

cudaError_t launch_round_light_f32(const EngineParams &p, int grid, int sms, cudaStream_t s) {
  return launch_round_t<float>(p, grid, sms, s);
}

cudaError_t launch_adjoint_light_f32(const EngineParams &p, double *grad, int grid, cudaStream_t s) {
  return launch_adjoint_t<float>(p, grad, grid, s);
}

int round_light_elems_f32(int n, int W) { return svd_elems_for<float>(n, W); }

}  // namespace stn
