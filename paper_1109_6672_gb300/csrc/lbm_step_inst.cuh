// Definitions of the launchers declared in lbm_launch.h; included by the four
// per-precision translation units.
#pragma once

#include "lbm_launch.h"
#include "lbm_batch.cuh"
#include "lbm_pair.cuh"
#include "lbm_step_pr.cuh"

#include <type_traits>

namespace lbm {

// Launch (or, with occ, resident blocks per SM) of the kernel of physics mode M:
// NPT = 1 the step over column pairs (lbm_pair.cuh), with programmatic
// dependent launch; 2 the pulled-row kernel with two columns per thread.
template <class S, int NPT, int M>
cudaError_t launch_one(const Grid& g, const CUtensorMap& map, int rows, dim3 grid,
                       cudaStream_t stream, int* occ) {
  void (*kernel)(Grid, CUtensorMap, int);
  int threads, smem;
  if constexpr (NPT == 1) {
    kernel = step_pair_kernel<S, M>;
    threads = PAIR_THREADS;
    smem = (int)PairGeom<S>::BYTES;
  } else {
    kernel = step_pr_kernel<S, NPT, M>;
    threads = PR_THREADS;
    smem = (int)PrGeom<S, NPT>::smem_bytes();
  }
  static std::atomic<unsigned long long> allowed{0};
  const cudaError_t e = allow_smem((const void*)kernel, smem, allowed);
  if (e != cudaSuccess) return e;
  if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kernel, threads, smem);
  return launch_ex(kernel, grid, threads, smem, stream, NPT == 1, g, map, rows);
}

// Calls fn(std::integral_constant<int, M>{}) for the kernel of physics mode
// `mode` (one of the BGK modes of mode_of, or with MRT_OK also their MRT
// twins); cudaErrorInvalidValue for a mode without a kernel.
template <int I, int OFF, class Fn>
cudaError_t dispatch_from(int mode, Fn& fn) {
  if constexpr (I == NUM_BGK_MODES) {
    return cudaErrorInvalidValue;
  } else {
    constexpr int M = BGK_MODES[I] | OFF;
    if (mode == M) return fn(std::integral_constant<int, M>{});
    return dispatch_from<I + 1, OFF>(mode, fn);
  }
}

template <bool ALL, class Fn>
cudaError_t dispatch_mode(int mode, Fn&& fn) {
  const int twin = mode & (MODE_MRT | MODE_VARMU);
  if (twin == 0) return dispatch_from<0, 0>(mode, fn);
  if constexpr (ALL) {
    if (twin == MODE_MRT) return dispatch_from<0, MODE_MRT>(mode, fn);
    if (twin == MODE_VARMU) return dispatch_from<0, MODE_VARMU>(mode, fn);
    return dispatch_from<0, MODE_MRT | MODE_VARMU>(mode, fn);
  }
  return cudaErrorInvalidValue;
}

// The two-node-per-thread variant is built for BGK with constant tau only.
template <class S, int NPT>
cudaError_t launch_mode(const Grid& g, const CUtensorMap& map, int rows, dim3 grid,
                        cudaStream_t stream, int* occ) {
  return dispatch_mode<NPT == 1>(mode_of(g), [&](auto m) {
    return launch_one<S, NPT, decltype(m)::value>(g, map, rows, grid, stream, occ);
  });
}

template <class S>
cudaError_t dispatch_variant(const Grid& g, const CUtensorMap& map, int variant, int rows,
                             dim3 grid, cudaStream_t stream, int* occ) {
  if (variant == TMA_PR_2) return launch_mode<S, 2>(g, map, rows, grid, stream, occ);
  if constexpr (sizeof(S) < 8) return launch_mode<S, 1>(g, map, rows, grid, stream, occ);
  return cudaErrorInvalidValue;  // FP64 storage takes the tile kernel instead
}

template <class S>
cudaError_t launch_step_tma(const Grid& g, const CUtensorMap& map, int variant, int rows,
                            dim3 grid, cudaStream_t stream) {
  return dispatch_variant<S>(g, map, variant, rows, grid, stream, nullptr);
}

template <class S, int M>
cudaError_t batch_one(const BatchGrid* grids, const WorkItem* items, BatchCtl* ctl, int j, int jc,
                      int blocks, cudaStream_t stream, bool pdl, int* occ) {
  static std::atomic<unsigned long long> allowed{0};
  const size_t smem = BatchGeom<S>::smem_bytes();
  const cudaError_t e = allow_smem((const void*)batch_step_kernel<S, M>, (int)smem, allowed);
  if (e != cudaSuccess) return e;
  if (occ)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, batch_step_kernel<S, M>,
                                                         BatchGeom<S>::threads,
                                                         smem);
  return launch_ex(batch_step_kernel<S, M>, dim3(blocks), BatchGeom<S>::threads, smem, stream, pdl,
                   grids, items, ctl, j, jc);
}

template <class S>
cudaError_t batch_mode(const BatchGrid* grids, const WorkItem* items, BatchCtl* ctl, int j, int jc,
                       int mode, int blocks, cudaStream_t stream, bool pdl, int* occ) {
  return dispatch_mode<true>(mode, [&](auto m) {
    return batch_one<S, decltype(m)::value>(grids, items, ctl, j, jc, blocks, stream, pdl, occ);
  });
}

template <class S>
cudaError_t launch_batch_step(const BatchGrid* grids, const WorkItem* items, BatchCtl* ctl, int j,
                              int jc, int mode, int blocks, cudaStream_t stream, bool pdl) {
  return batch_mode<S>(grids, items, ctl, j, jc, mode, blocks, stream, pdl, nullptr);
}

template <class S>
int occupancy_batch(int mode) {
  int occ = 0;
  batch_mode<S>(nullptr, nullptr, nullptr, 0, 0, mode, 1, nullptr, false, &occ);
  return occ;
}

template <class S>
int occupancy_step_tma(const Grid& g, int variant) {
  int occ = 0;
  dispatch_variant<S>(g, CUtensorMap{}, variant, 1, dim3(1), nullptr, &occ);
  return occ;
}

}  // namespace lbm
