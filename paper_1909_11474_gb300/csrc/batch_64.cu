// batch_64.cu -- the batched kernels in FP64, minimal form, in a translation unit of its own so that the kernels compile side by side.
#include "batch_launch.cuh"

namespace tsf {

template cudaError_t launch_bucket<double, false, true>(const BatchParams &, const Bucket &, bool, cudaStream_t);
template cudaError_t launch_bucket<double, false, false>(const BatchParams &, const Bucket &, bool, cudaStream_t);

cudaError_t preload_batch64() {
  cudaError_t e = touch_variants64<true>();
  if (e == cudaSuccess) e = touch_variants64<false>();
  return e;
}

TSF_DEBUG_TAKE(debug_take_64)

}  // namespace tsf
