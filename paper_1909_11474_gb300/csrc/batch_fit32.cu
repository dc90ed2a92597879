// batch_fit32.cu -- the batched fitness kernels in FP32, minimal form, in a translation unit of its own so that the kernels compile side by side.
#include "batch_launch.cuh"

namespace tsf {

template cudaError_t launch_bucket<float, false, true>(const BatchParams &, const Bucket &, bool, cudaStream_t);

cudaError_t preload_fitness32() {
  cudaError_t e = touch_variant<16, 4, false, 3, float, kNW, true>();
  if (e == cudaSuccess) e = touch_variant<kPT, 4, false, 2, float, 12, true>();
  if (e == cudaSuccess) e = touch_variants32<true>();
  return e;
}

TSF_DEBUG_TAKE(debug_take_fit32)

}  // namespace tsf
