// dugks_internal.h -- host-side launch interface between the C ABI (dugks_api.cu)
// and the per-precision kernel instantiations (dugks_inst_*.cu).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "dugks_fast.cuh"
#include "dugks_kernels.cuh"
#include "dugks_march.cuh"

namespace dugks {

// Tile of one CTA of the generic fused step kernel.
constexpr int TILE_X = 32;
constexpr int TILE_Y = 8;
constexpr int STEP_THREADS = 256;

// Variants of the two-stage kernel of orders 2 and 3: rows of a segment of the row march,
// 0 = 16, 1 = 8, 3 = 32, 5 = 64; 2 and 4 (the defaults) by the rule of march_plan.
constexpr int FAST_VARIANTS = 6;

// Geometry of a TMA-staged kernel (orders 4 and 5).
struct FastGeom {
    int threads, tile_w, tile_h;   // cells written per CTA
    int box_w, box_h;              // state box (elements, rows)
    int box_wt;                    // phi box width (elements)
};

template <typename T, typename ST>
struct Launch {
    static cudaError_t step(const StepParams<T> &p, int order, int flux, int kind, cudaStream_t s);
    static cudaError_t init(const StepParams<T> &p, const T *phi0, T frac_dt, int order, cudaStream_t s);
    static cudaError_t mass_partial(const StepParams<T> &p, cudaStream_t s);
    // masses of `count` grids of at most `tiles` tiles into out[slot]; part: MASS_TILES a grid; counters: 0
    static cudaError_t mass(const MassList<T> &list, int count, int tiles, double *part, unsigned *counters, double *out,
                            int *status, cudaStream_t s);
    static cudaError_t phi(const StepParams<T> &p, T *out, cudaStream_t s);
    // phi widened to double on the device (host read-out: one copy, no host conversion)
    static cudaError_t phi64(const StepParams<T> &p, double *out, cudaStream_t s);
    static FastGeom fast_geom(int stages);
    // the two-stage step of orders 2 and 3 on the TMA-staged path (FP64), tile 8 warps x 2 rows
    static FastGeom tile_geom();
    static cudaError_t step_tile(const StepParams<T> &p, const FaceCoefs<T> &cf, const FastExtra<T> &fe,
                                 const CUtensorMap &tmX, const CUtensorMap &tmPo, const CUtensorMap &tmPc, int order,
                                 int flux, cudaStream_t s);
    // the row march (two-stage, orders 2 and 3): one strip segment of p.tile_h rows per CTA,
    // `cols` columns a lane
    static cudaError_t step_march(const StepParams<T> &p, const MarchCoefs<T> &cf, const FastExtra<T> &fe, int flux,
                                  int cols, int mode, cudaStream_t s);
    // step `ofs` of a group for the grids of a work list; rows: the longest segment
    static cudaError_t batch_step(const BatchUniform<T> &u, const MarchCoefs<T> &cf, const BatchGrid<T> *grids,
                                  const int4 *items, int nitems, int rows, int ofs, int flux, int cols, int ctas,
                                  cudaStream_t s);
    static int batch_ctas_per_sm(int flux, int cols, int rows);
    // order 4 (radius-2 stencils) on the TMA-staged path, tile 8 warps x 2 rows: the
    // two-stage step (KIND_T2) or a kernel of the three-stage step (full storage only)
    static cudaError_t step_fast4(const StepParams<T> &p, const FaceCoefs<T, 2> &cf, const FastExtra<T> &fe,
                                  const CUtensorMap &tmX, const CUtensorMap &tmPo, const CUtensorMap &tmPc, int flux,
                                  int kind, cudaStream_t s);
    // one kernel of the three-stage step (kind KIND_T3A or KIND_T3B; full storage only) as a
    // row march, orders 2 and 3
    static cudaError_t step_march3(const StepParams<T> &p, const MarchCoefs<T> &cf, const FastExtra<T> &fe, int flux,
                                   int kind, int cols, int mode, cudaStream_t s);
};

template <typename T>
cudaError_t launch_batch_advance(BatchGrid<T> *grids, int ngrids, int n, double dt, cudaStream_t s);

// words: as integers, where there are as many partials as gain by it
cudaError_t launch_mass_final(const double *partial, int n, double *out, int *status, int early, bool words, cudaStream_t s);

// One step of the streaming-collision DVM of order 4 (dugks_inst_dvm.cu); lbm: the plain
// streaming of dt = 1 (T = double or float, full storage).
template <typename T>
struct DvmExtra;
template <typename T>
cudaError_t launch_dvm(const StepParams<T> &p, const DvmExtra<T> &dv, bool lbm, cudaStream_t s);
// the same as a row march (orders 2 and 3), `cols` columns a lane, segments of p.tile_h rows
template <typename T>
cudaError_t launch_dvm_march(const StepParams<T> &p, const DvmExtra<T> &dv, const MarchCoefs<T> &cf,
                             const FastExtra<T> &fe, bool lbm, int cols, cudaStream_t s);
int dvm_march_strips(int cols, int nx);
constexpr int dvm_march_width(int cols) { return cols == 2 ? 56 : 26; }

// Every device allocation of the library goes through dev_malloc: cudaMalloc
// behind a host-side test hook (dugks_selftest_fail_allocs) that can make chosen
// allocations report cudaErrorMemoryAllocation without touching the device.
cudaError_t dev_malloc_raw(void **p, size_t bytes);
// The same hook in front of a stream-ordered allocation from `pool` on stream `s`
// (cudaMallocFromPoolAsync): the memory is usable in the order of `s`.
cudaError_t dev_malloc_pool(void **p, size_t bytes, cudaMemPool_t pool, cudaStream_t s);
template <typename P>
inline cudaError_t dev_malloc(P **p, size_t bytes) {
    return dev_malloc_raw(reinterpret_cast<void **>(p), bytes);
}

}  // namespace dugks
