// row-march kernels of the three-stage step (orders 2 and 3); state and arithmetic in double.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template cudaError_t Launch<double,double>::step_march3(const StepParams<double> &, const MarchCoefs<double> &, const FastExtra<double> &, int, int, int, int, cudaStream_t);
}  // namespace dugks
