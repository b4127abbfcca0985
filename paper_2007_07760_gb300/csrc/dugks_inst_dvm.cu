// Streaming-collision DVM / LBM step kernels (dugks_dvm.cuh), FP64 and FP32.
// (One translation unit per kernel family, so they compile in parallel.)
#include <atomic>

#include "dugks_dvm.cuh"
#include "dugks_internal.h"

namespace dugks {

namespace {

template <typename T, bool LBM>
cudaError_t launch_dvm_t(const StepParams<T> &p, const DvmExtra<T> &dv, cudaStream_t s) {
    using DT = DvmTile<T, LBM>;
    auto kern = dvm_step_kernel<T, LBM>;
    // the dynamic shared-memory limit is a per-function, per-device attribute
    static std::atomic<uint64_t> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (uint64_t(1) << dev) : 0;
    if (!bit || !(configured.load(std::memory_order_relaxed) & bit)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DT::smem_bytes);
        if (e != cudaSuccess) return e;
        if (bit) configured.fetch_or(bit, std::memory_order_relaxed);
    }
    const dim3 grid((p.nx + DT::TX - 1) / DT::TX, (p.ny + DT::TY - 1) / DT::TY);
    kern<<<grid, DT::NT, DT::smem_bytes, s>>>(p, dv);
    return cudaGetLastError();
}

template <typename V, int MODE>
cudaError_t launch_dvm_m(const StepParams<typename Lane<V>::T> &p, const DvmExtra<typename Lane<V>::T> &dv,
                         const MarchCoefs<typename Lane<V>::T> &cf, const FastExtra<typename Lane<V>::T> &fe,
                         cudaStream_t s) {
    static_assert(DvmMarch<V>::smem_bytes(64) <= 48 * 1024, "fits without the shared-memory attribute");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.tiles_x, (p.ny + p.tile_h - 1) / p.tile_h);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = DvmMarch<V>::smem_bytes(p.tile_h);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // (the mass partials are written where the caller asks for them; FP64 steps always do)
    if constexpr (sizeof(typename Lane<V>::T) == 4)
        if (p.mass_partial == nullptr) return cudaLaunchKernelEx(&cfg, dvm_march_kernel<V, MODE, false>, p, dv, cf, fe);
    return cudaLaunchKernelEx(&cfg, dvm_march_kernel<V, MODE, true>, p, dv, cf, fe);
}

template <typename V>
cudaError_t launch_dvm_v(const StepParams<typename Lane<V>::T> &p, const DvmExtra<typename Lane<V>::T> &dv,
                         const MarchCoefs<typename Lane<V>::T> &cf, const FastExtra<typename Lane<V>::T> &fe, bool lbm,
                         cudaStream_t s) {
    return lbm ? launch_dvm_m<V, 2>(p, dv, cf, fe, s)
               : dv.s ? launch_dvm_m<V, 1>(p, dv, cf, fe, s) : launch_dvm_m<V, 0>(p, dv, cf, fe, s);
}

}  // namespace

template <typename T>
cudaError_t launch_dvm(const StepParams<T> &p, const DvmExtra<T> &dv, bool lbm, cudaStream_t s) {
    return lbm ? launch_dvm_t<T, true>(p, dv, s) : launch_dvm_t<T, false>(p, dv, s);
}

template <typename T>
cudaError_t launch_dvm_march(const StepParams<T> &p, const DvmExtra<T> &dv, const MarchCoefs<T> &cf,
                             const FastExtra<T> &fe, bool lbm, int cols, cudaStream_t s) {
    if constexpr (sizeof(T) == 4)
        if (cols == 2) return launch_dvm_v<float2>(p, dv, cf, fe, lbm, s);
    return launch_dvm_v<T>(p, dv, cf, fe, lbm, s);
}
int dvm_march_strips(int cols, int nx) { return cols == 2 ? DvmMarch<float2>::strips(nx) : DvmMarch<float>::strips(nx); }

template cudaError_t launch_dvm_march<double>(const StepParams<double> &, const DvmExtra<double> &, const MarchCoefs<double> &, const FastExtra<double> &, bool, int, cudaStream_t);
template cudaError_t launch_dvm_march<float>(const StepParams<float> &, const DvmExtra<float> &, const MarchCoefs<float> &, const FastExtra<float> &, bool, int, cudaStream_t);
template cudaError_t launch_dvm<double>(const StepParams<double> &, const DvmExtra<double> &, bool, cudaStream_t);
template cudaError_t launch_dvm<float>(const StepParams<float> &, const DvmExtra<float> &, bool, cudaStream_t);

}  // namespace dugks
