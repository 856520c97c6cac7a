#include "sweep_launch.cuh"

namespace mg {
template cudaError_t sweep32_run<float, double>(const SweepCall32<float, double>&, cudaStream_t);
}
