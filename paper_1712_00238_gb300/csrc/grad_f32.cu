// FP32 instantiation of the type-2 score and gradient gather.
#include "grad_impl.cuh"

namespace sd {
template cudaError_t launch_gather<float>(const GatherArgs<float>&, int, cudaStream_t);
}  // namespace sd
