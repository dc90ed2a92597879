// batch_gen64.cu -- the batched kernels in FP64, Tersoff form, in a translation unit of its own so that the kernels compile side by side.
#include "batch_launch.cuh"

namespace tsf {

template cudaError_t launch_bucket<double, true, true>(const BatchParams &, const Bucket &, bool, cudaStream_t);
template cudaError_t launch_bucket<double, true, false>(const BatchParams &, const Bucket &, bool, cudaStream_t);

TSF_DEBUG_TAKE(debug_take_gen64)

}  // namespace tsf
