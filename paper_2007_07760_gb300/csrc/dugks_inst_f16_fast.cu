// tile geometry of the TMA-staged kernels; FP32 arithmetic, distribution stored as half-precision deviations from w_k phi.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template FastGeom Launch<float,__half>::fast_geom(int, int, int);
}  // namespace dugks
