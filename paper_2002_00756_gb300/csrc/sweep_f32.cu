// FP32 column sweep with FP32 couplings and elimination (the units compile in parallel).
#include "sweep_launch.cuh"

namespace mg {
template cudaError_t sweep32_run<float, float>(const SweepCall32<float, float>&, cudaStream_t);
}
