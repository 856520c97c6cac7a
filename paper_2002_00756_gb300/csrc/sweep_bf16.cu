#include "sweep_launch.cuh"

namespace mg {
template cudaError_t sweep32_run<__nv_bfloat16, float>(const SweepCall32<__nv_bfloat16, float>&, cudaStream_t);
}
