// row-march kernels of the three-stage step (orders 2 and 3); state and arithmetic in float.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template cudaError_t Launch<float,float>::step_march3(const StepParams<float> &, const MarchCoefs<float> &, const FastExtra<float> &, int, int, int, int, cudaStream_t);
}  // namespace dugks
