// row-march step kernels of the two-stage scheme (orders 2 and 3), single grid and batch; state float, arithmetic float.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template cudaError_t Launch<float,float>::step_march(const StepParams<float> &, const MarchCoefs<float> &, const FastExtra<float> &, int, int, int, cudaStream_t);
template cudaError_t Launch<float,float>::batch_step(const BatchUniform<float> &, const MarchCoefs<float> &, const BatchGrid<float> *, const int4 *, int, int, int, int, int, int, cudaStream_t);
template int Launch<float,float>::batch_ctas_per_sm(int, int, int);
template cudaError_t launch_batch_advance<float>(BatchGrid<float> *, int, int, double, cudaStream_t);
}  // namespace dugks
