// row-march step kernels of the two-stage scheme (orders 2 and 3), single grid and batch; state and arithmetic double.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template cudaError_t Launch<double,double>::step_march(const StepParams<double> &, const MarchCoefs<double> &, const FastExtra<double> &, int, int, int, cudaStream_t);
template cudaError_t Launch<double,double>::batch_step(const BatchUniform<double> &, const MarchCoefs<double> &, const BatchGrid<double> *, const int4 *, int, int, int, int, int, int, cudaStream_t);
template int Launch<double,double>::batch_ctas_per_sm(int, int, int);
template cudaError_t launch_batch_advance<double>(BatchGrid<double> *, int, int, double, cudaStream_t);
}  // namespace dugks
