// batch_eval32.cu -- the batched evaluation and gradient kernels in FP32, minimal form, in a translation unit of its own so that the kernels compile side by side.
#include "batch_launch.cuh"

namespace tsf {

template cudaError_t launch_bucket<float, false, false>(const BatchParams &, const Bucket &, bool, cudaStream_t);

cudaError_t preload_eval32() { return touch_variants32<false>(); }

TSF_DEBUG_TAKE(debug_take_eval32)

}  // namespace tsf
