// dugks_launch.cuh -- launchers of one precision; included once by each
// dugks_inst_*.cu so the three precisions compile in parallel.
#pragma once

#include <atomic>

#include "dugks_internal.h"

namespace dugks {

// Raises a kernel's dynamic shared-memory limit once per device (the attribute is
// per function and device); `done` is the kernel's own bit set of devices.
template <typename K>
static cudaError_t smem_attr_once(K kern, int bytes, std::atomic<uint64_t> &done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (uint64_t(1) << dev) : 0;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

template <typename T, typename ST, int ORDER, int FLUX, int KIND>
static cudaError_t launch_step_t(const StepParams<T> &p, cudaStream_t s) {
    using TL = Tile<T, ST, ORDER, FLUX, KIND, TILE_X, TILE_Y>;
    auto kern = step_kernel<T, ST, ORDER, FLUX, KIND, TILE_X, TILE_Y>;
    static std::atomic<uint64_t> configured{0};
    if (cudaError_t e = smem_attr_once(kern, (int)TL::smem_bytes, configured); e != cudaSuccess) return e;
    dim3 grid((p.nx + TILE_X - 1) / TILE_X, (p.ny + TILE_Y - 1) / TILE_Y);
    kern<<<grid, STEP_THREADS, TL::smem_bytes, s>>>(p);
    return cudaGetLastError();
}

// (each storage compiles only the schemes it serves)
template <typename T, typename ST, int ORDER, int FLUX>
static cudaError_t launch_kind(const StepParams<T> &p, int kind, cudaStream_t s) {
    if constexpr (Store<T, ST>::t2)
        if (kind == KIND_T2) return launch_step_t<T, ST, ORDER, FLUX, KIND_T2>(p, s);
    if constexpr (Store<T, ST>::t3) {
        if (kind == KIND_T3A) return launch_step_t<T, ST, ORDER, FLUX, KIND_T3A>(p, s);
        if (kind == KIND_T3B) return launch_step_t<T, ST, ORDER, FLUX, KIND_T3B>(p, s);
    }
    return cudaErrorInvalidValue;
}

template <typename T, typename ST, int ORDER>
static cudaError_t launch_flux(const StepParams<T> &p, int flux, int kind, cudaStream_t s) {
    return flux == 0 ? launch_kind<T, ST, ORDER, 0>(p, kind, s) : launch_kind<T, ST, ORDER, 1>(p, kind, s);
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::step(const StepParams<T> &p, int order, int flux, int kind, cudaStream_t s) {
    switch (order) {
    case 2: return launch_flux<T, ST, 2>(p, flux, kind, s);
    case 3: return launch_flux<T, ST, 3>(p, flux, kind, s);
    case 4: return launch_flux<T, ST, 4>(p, flux, kind, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::init(const StepParams<T> &p, const T *phi0, T frac_dt, int order, cudaStream_t s) {
    dim3 block(128), grid((p.nx + 127) / 128, p.ny);
    switch (order) {
    case 2: init_kernel<T, ST, 2><<<grid, block, 0, s>>>(p, phi0, frac_dt); break;
    case 3: init_kernel<T, ST, 3><<<grid, block, 0, s>>>(p, phi0, frac_dt); break;
    case 4: init_kernel<T, ST, 4><<<grid, block, 0, s>>>(p, phi0, frac_dt); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::mass_partial(const StepParams<T> &p, cudaStream_t s) {
    dim3 grid(p.tiles_x, (p.ny + p.tile_h - 1) / p.tile_h);
    mass_partial_kernel<T, ST><<<grid, 256, 0, s>>>(p);
    return cudaGetLastError();
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::mass(const MassList<T> &list, int count, int tiles, double *part, unsigned *counters,
                                double *out, int *status, cudaStream_t s) {
    mass_kernel<T, ST><<<dim3(tiles, count), 256, 0, s>>>(list, part, counters, out, status);
    return cudaGetLastError();
}

template <typename T, typename ST, int NW, int MR, int R = 1>
static FastGeom geom_t() {
    using FT = FastTile<T, ST, NW, MR, R>;
    return FastGeom{FT::NT, FT::TX, FT::TY, FT::BW, FT::RH, FT::BWT};
}

// Tile of the radius-2 (orders 4 and 5) two-stage kernel: 10 warps x 3 rows in FP32
// and FP16 storage (measured in FP32 at 4096^2: 893 us against 1159 us for 8 x 2;
// at 1024^2 78 against 84 us), 8 x 2 in FP64. The three-stage kernels keep 8 x 2.
template <typename T>
constexpr int o4_nw() { return sizeof(T) == 8 ? 8 : 10; }
template <typename T>
constexpr int o4_mr() { return sizeof(T) == 8 ? 2 : 3; }

template <typename T, typename ST>
FastGeom Launch<T, ST>::fast_geom(int stages) {
    return stages == 2 ? geom_t<T, ST, o4_nw<T>(), o4_mr<T>(), 2>() : geom_t<T, ST, 8, 2, 2>();
}

// Tiles of radius R: orders 4 and 5 (R = 2, every kind), orders 2 and 3 (R = 1, two-stage)
template <typename T, typename ST, int ORDER, int FLUX, int KIND>
static cudaError_t launch_fast_t(const StepParams<T> &p, const FaceCoefs<T, (ORDER == 4 ? 2 : 1)> &cf,
                                 const FastExtra<T> &fe, const CUtensorMap &tmX, const CUtensorMap &tmPo,
                                 const CUtensorMap &tmPc, cudaStream_t s) {
    constexpr int NW = ORDER == 4 && KIND == KIND_T2 ? o4_nw<T>() : 8, MR = ORDER == 4 && KIND == KIND_T2 ? o4_mr<T>() : 2;
    using FT = FastTile<T, ST, NW, MR, (ORDER == 4 ? 2 : 1)>;
    constexpr size_t smem = KIND == KIND_T3A ? FT::smem_bytes_t3a : FT::smem_bytes;
    auto kern = step_fast_kernel<T, ST, ORDER, FLUX, NW, MR, KIND>;
    static std::atomic<uint64_t> configured{0};
    if (cudaError_t e = smem_attr_once(kern, (int)smem, configured); e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.nx + FT::TX - 1) / FT::TX, (p.ny + FT::TY - 1) / FT::TY);
    cfg.blockDim = dim3(FT::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, cf, fe, tmX, tmPo, tmPc);
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::step_fast4(const StepParams<T> &p, const FaceCoefs<T, 2> &cf, const FastExtra<T> &fe,
                                      const CUtensorMap &tmX, const CUtensorMap &tmPo, const CUtensorMap &tmPc,
                                      int flux, int kind, cudaStream_t s) {
    if constexpr (Store<T, ST>::t2)
        if (kind == KIND_T2)
            return flux == 0 ? launch_fast_t<T, ST, 4, 0, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s)
                             : launch_fast_t<T, ST, 4, 1, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s);
    if constexpr (Store<T, ST>::t3) {
        if (kind == KIND_T3A)
            return flux == 0 ? launch_fast_t<T, ST, 4, 0, KIND_T3A>(p, cf, fe, tmX, tmPo, tmPc, s)
                             : launch_fast_t<T, ST, 4, 1, KIND_T3A>(p, cf, fe, tmX, tmPo, tmPc, s);
        if (kind == KIND_T3B)
            return flux == 0 ? launch_fast_t<T, ST, 4, 0, KIND_T3B>(p, cf, fe, tmX, tmPo, tmPc, s)
                             : launch_fast_t<T, ST, 4, 1, KIND_T3B>(p, cf, fe, tmX, tmPo, tmPc, s);
    }
    return cudaErrorInvalidValue;
}

template <typename T, typename ST>
FastGeom Launch<T, ST>::tile_geom() { return geom_t<T, ST, 8, 2, 1>(); }

template <typename T, typename ST>
cudaError_t Launch<T, ST>::step_tile(const StepParams<T> &p, const FaceCoefs<T> &cf, const FastExtra<T> &fe,
                                     const CUtensorMap &tmX, const CUtensorMap &tmPo, const CUtensorMap &tmPc, int order,
                                     int flux, cudaStream_t s) {
    if (order == 2)
        return flux == 0 ? launch_fast_t<T, ST, 2, 0, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s)
                         : launch_fast_t<T, ST, 2, 1, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s);
    return flux == 0 ? launch_fast_t<T, ST, 3, 0, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s)
                     : launch_fast_t<T, ST, 3, 1, KIND_T2>(p, cf, fe, tmX, tmPo, tmPc, s);
}

// CALL with the lane type of `cols` columns
#define DUGKS_LANES(CALL)                                                                     \
    if (cols == 1) return CALL(T);                                                            \
    if constexpr (sizeof(T) == 4) return CALL(float2);

template <typename V, typename ST, int FLUX, bool FIELD, int KIND, int SUM>
static cudaError_t launch_march_s(const StepParams<typename Lane<V>::T> &p, const MarchCoefs<typename Lane<V>::T> &cf,
                                  const FastExtra<typename Lane<V>::T> &fe, int mode, cudaStream_t s) {
    using MT = MarchTile<V, ST, KIND>;
    const int smem = MT::smem_bytes(p.tile_h);
    static_assert(MT::smem_bytes(64) <= 48 * 1024, "fits without the shared-memory attribute");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.tiles_x, (p.ny + p.tile_h - 1) / p.tile_h);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // pairs, upwind: a body of its own for the rows before the first output costs registers that are
    // spilled. In one wave, where segments are short and a row's latency counts, it gains (450^2, 3 rows:
    // 10.8 -> 10.3 us, FP16 storage 12.4 -> 11.3; 1024^2, 16 rows: 36.0 -> 34.9); over several it
    // loses (2048^2: 105.0 -> 105.1, FP16 storage 117.1 -> 123.1)
    if constexpr (Lane<V>::N == 2 && FLUX == 0)
        if (mode & MARCH_ONE_WAVE)
            return cudaLaunchKernelEx(&cfg, step_march_kernel<V, ST, FLUX, FIELD, KIND, SUM, true>, p, cf, fe, mode);
    return cudaLaunchKernelEx(&cfg, step_march_kernel<V, ST, FLUX, FIELD, KIND, SUM, sizeof(V) == 4>, p, cf, fe, mode);
}

// (the mass partials are written where the caller asks for them; FP64 steps always do: it is one of
// about 350 FP64 instructions a row there)
template <typename V, typename ST, int FLUX, bool FIELD, int KIND>
static cudaError_t launch_march_t(const StepParams<typename Lane<V>::T> &p, const MarchCoefs<typename Lane<V>::T> &cf,
                                  const FastExtra<typename Lane<V>::T> &fe, int mode, cudaStream_t s) {
    if constexpr (KIND != KIND_T3A)
        if (p.mass_partial != nullptr) return launch_march_s<V, ST, FLUX, FIELD, KIND, SUM_MASS>(p, cf, fe, mode, s);
    if constexpr (KIND == KIND_T3A || sizeof(typename Lane<V>::T) == 4)
        return launch_march_s<V, ST, FLUX, FIELD, KIND, SUM_NONE>(p, cf, fe, mode, s);
    return cudaErrorInvalidValue;
}

template <typename V, typename ST, int KIND>
static cudaError_t launch_march_v(const StepParams<typename Lane<V>::T> &p, const MarchCoefs<typename Lane<V>::T> &cf,
                                  const FastExtra<typename Lane<V>::T> &fe, int flux, int mode, cudaStream_t s) {
    if (p.vel_kind == VEL_FIELD)
        return flux == 0 ? launch_march_t<V, ST, 0, true, KIND>(p, cf, fe, mode, s)
                         : launch_march_t<V, ST, 1, true, KIND>(p, cf, fe, mode, s);
    return flux == 0 ? launch_march_t<V, ST, 0, false, KIND>(p, cf, fe, mode, s)
                     : launch_march_t<V, ST, 1, false, KIND>(p, cf, fe, mode, s);
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::step_march(const StepParams<T> &p, const MarchCoefs<T> &cf, const FastExtra<T> &fe, int flux,
                                      int cols, int mode, cudaStream_t s) {
#define CALL(V) launch_march_v<V, ST, KIND_T2>(p, cf, fe, flux, mode, s)
    DUGKS_LANES(CALL)
#undef CALL
    return cudaErrorInvalidValue;
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::step_march3(const StepParams<T> &p, const MarchCoefs<T> &cf, const FastExtra<T> &fe, int flux,
                                       int kind, int cols, int mode, cudaStream_t s) {
#define CALL(V)                                                              \
    (kind == KIND_T3A ? launch_march_v<V, ST, KIND_T3A>(p, cf, fe, flux, mode, s) \
                      : launch_march_v<V, ST, KIND_T3B>(p, cf, fe, flux, mode, s))
    DUGKS_LANES(CALL)
#undef CALL
    return cudaErrorInvalidValue;
}

// a launch that may be scheduled while the kernel ahead of it drains
template <typename K, typename... A>
static cudaError_t launch_dependent(K kern, int blocks, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename V, typename ST>
static cudaError_t launch_batch_v(const BatchUniform<typename Lane<V>::T> &u, const MarchCoefs<typename Lane<V>::T> &cf,
                                  const BatchGrid<typename Lane<V>::T> *grids, const int4 *items, int nitems, int rows,
                                  int ofs, int flux, int ctas, cudaStream_t s) {
    const int smem = MarchTile<V, ST>::smem_bytes(rows), n = ctas < nitems ? ctas : nitems;
    return flux == 0 ? launch_dependent(batch_march_kernel<V, ST, 0>, n, 32, smem, s, u, cf, grids, items, nitems, ofs)
                     : launch_dependent(batch_march_kernel<V, ST, 1>, n, 32, smem, s, u, cf, grids, items, nitems, ofs);
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::batch_step(const BatchUniform<T> &u, const MarchCoefs<T> &cf, const BatchGrid<T> *grids,
                                      const int4 *items, int nitems, int rows, int ofs, int flux, int cols, int ctas,
                                      cudaStream_t s) {
    if (nitems <= 0) return cudaSuccess;
#define CALL(V) launch_batch_v<V, ST>(u, cf, grids, items, nitems, rows, ofs, flux, ctas, s)
    DUGKS_LANES(CALL)
#undef CALL
    return cudaErrorInvalidValue;
}

template <typename V, typename ST>
static int batch_occupancy(int rows, int flux) {
    int n = 0;
    const int smem = MarchTile<V, ST>::smem_bytes(rows);
    const cudaError_t e =
        flux == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_march_kernel<V, ST, 0>, 32, smem)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_march_kernel<V, ST, 1>, 32, smem);
    if (e != cudaSuccess) {
        cudaGetLastError();
        n = 1;
    }
    return n > 0 ? n : 1;
}

template <typename T, typename ST>
int Launch<T, ST>::batch_ctas_per_sm(int flux, int cols, int rows) {
#define CALL(V) batch_occupancy<V, ST>(rows, flux)
    DUGKS_LANES(CALL)
#undef CALL
    return 1;
}

template <typename T>
cudaError_t launch_batch_advance(BatchGrid<T> *grids, int ngrids, int n, double dt, cudaStream_t s) {
    if (ngrids <= 0) return cudaSuccess;
    return launch_dependent(batch_advance_kernel<T>, ngrids, 32, 0, s, grids, n, dt);
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::phi(const StepParams<T> &p, T *out, cudaStream_t s) {
    dim3 block(128), grid((p.nx + 127) / 128, p.ny);
    phi_kernel<T, ST><<<grid, block, 0, s>>>(p, out);
    return cudaGetLastError();
}

template <typename T, typename ST>
cudaError_t Launch<T, ST>::phi64(const StepParams<T> &p, double *out, cudaStream_t s) {
    dim3 block(128), grid((p.nx + 127) / 128, p.ny);
    phi_kernel<T, ST, double><<<grid, block, 0, s>>>(p, out);
    return cudaGetLastError();
}

}  // namespace dugks
