// FP32 instantiation of the half-spectrum inverse passes.
#include "nufft_half.cuh"
SD_INSTANTIATE_HALF(float)
