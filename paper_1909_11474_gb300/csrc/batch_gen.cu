// batch_gen.cu -- the batched kernels in FP32, Tersoff form (Eq. 8 angular function, free S in Eq. 11-14), in a translation unit of its own so that the kernels compile side by side.
#include "batch_launch.cuh"

namespace tsf {

template cudaError_t launch_bucket<float, true, true>(const BatchParams &, const Bucket &, bool, cudaStream_t);
template cudaError_t launch_bucket<float, true, false>(const BatchParams &, const Bucket &, bool, cudaStream_t);

TSF_DEBUG_TAKE(debug_take_gen)

}  // namespace tsf
