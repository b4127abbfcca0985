// TMA-staged kernels for order 4 (radius-2 stencils) and the FP64 two-stage step of orders 2 and 3; state double, arithmetic double.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template FastGeom Launch<double,double>::fast_geom(int);
template cudaError_t Launch<double,double>::step_fast4(const StepParams<double> &, const FaceCoefs<double, 2> &, const FastExtra<double> &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, int, int, cudaStream_t);
template FastGeom Launch<double,double>::tile_geom();
template cudaError_t Launch<double,double>::step_tile(const StepParams<double> &, const FaceCoefs<double> &, const FastExtra<double> &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, int, int, cudaStream_t);
}  // namespace dugks
