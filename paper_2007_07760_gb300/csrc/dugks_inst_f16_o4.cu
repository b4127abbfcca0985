// TMA-staged kernels for order 4 (radius-2 stencils); state __half, arithmetic float.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template FastGeom Launch<float,__half>::fast_geom(int);
template cudaError_t Launch<float,__half>::step_fast4(const StepParams<float> &, const FaceCoefs<float, 2> &, const FastExtra<float> &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, int, int, cudaStream_t);
}  // namespace dugks
