// tile geometry of the TMA-staged kernels; state and arithmetic in double.
// (One translation unit per precision and kernel family, so they compile in parallel.)
#include "dugks_launch.cuh"

namespace dugks {
template FastGeom Launch<double,double>::fast_geom(int, int, int);
}  // namespace dugks
