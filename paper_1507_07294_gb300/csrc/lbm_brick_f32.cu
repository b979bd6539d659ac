// The resident-brick kernel (lbm_brick.cuh) for FP32 populations.
#include "lbm_brick.cuh"

namespace lbm {

const void* brick_kernel_f32(int mode, int var, bool pair, bool in_place) {
  return brick_kernel<kF32>(mode, var, pair, in_place);
}

cudaError_t state_sums_f32(const float* state, const float* phi, const Geometry& geo, double* partial,
                           double* out, const double* word, int* count, cudaStream_t st) {
  return state_sums<kF32>(state, phi, geo, partial, out, word, count, st);
}

}  // namespace lbm
