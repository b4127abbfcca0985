// row-march step kernels of the two-stage scheme (orders 2 and 3), single grid; state and arithmetic double.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template cudaError_t Launch<double,double>::step_march(const StepParams<double> &, const MarchCoefs<double> &, const FastExtra<double> &, int, int, int, cudaStream_t);
}  // namespace dugks
