// Host launchers of the TMA-staged step kernel, one translation unit per
// storage type (lbm_step_f64.cu, lbm_step_f32.cu, lbm_step_f16.cu,
// lbm_step_bf16.cu) so the instantiations compile in parallel.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "lbm_device.cuh"

namespace lbm {

// TMA step kernels: the step over column pairs (lbm_pair.cuh; variant 1, FP32 and
// 16-bit storage) with 128 columns per block, the pulled-row kernel
// (lbm_step_pr.cuh; variant 2) with 256; box width (columns) of one TMA copy.
enum { TMA_PR_1 = 1, TMA_PR_2 = 2 };
constexpr int tma_npt(int variant) { return variant == TMA_PR_2 ? 2 : 1; }
constexpr int tma_cols(int variant) { return 128 * tma_npt(variant); }
constexpr int tma_box(int npt) { return npt == 1 ? 144 : 136; }
// Default rows per block of these kernels: small blocks, many waves,
// dynamically balanced across SMs (measured on GB300 at 4096^2).
inline int tma_default_rows(size_t elem_bytes) { return elem_bytes == 4 ? 6 : 12; }

// Launch one step on `stream`; grid.x covers nx in tma_cols(variant)
// columns, grid.y covers ny in `rows` rows.  Returns the launch error.
template <class S>
cudaError_t launch_step_tma(const Grid& g, const CUtensorMap& map, int variant, int rows,
                            dim3 grid, cudaStream_t stream);

// Resident blocks per SM of that kernel (0 if it cannot launch).
template <class S>
int occupancy_step_tma(const Grid& g, int variant);

// Tile step kernel (lbm_tile.cuh): FP64 storage, the automatic choice there.
// Tiles of 2^lw columns x rows; tile_shape picks them from the grid (rows > 0:
// that many rows, as far as they fit).  The launch also covers the open sides
// and the walls of non-equilibrium extrapolation.
enum { STEP_TILE = 3 };
void tile_shape(int nx, int ny, bool corr, int sms, int rows, int* lw_out, int* rows_out);
cudaError_t launch_step_tile(const Grid& g, int lw, int rows, cudaStream_t stream);

struct BatchGrid;
struct WorkItem;
struct BatchCtl;

// One step of the batched kernel (lbm_batch.cuh) for the items of physics
// mode `mode` over `blocks` persistent blocks (pdl: the launch may start while the
// kernel before it in the stream, the step before, still runs), and its
// resident blocks per SM.
template <class S>
cudaError_t launch_batch_step(const BatchGrid* grids, const WorkItem* items, BatchCtl* ctl, int j,
                              int jc, int mode, int blocks, cudaStream_t stream, bool pdl);
template <class S>
int occupancy_batch(int mode);

}  // namespace lbm
