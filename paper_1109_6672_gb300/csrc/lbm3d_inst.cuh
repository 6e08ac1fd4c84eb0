// Instantiation of the D3Q19 kernels for one storage precision S (included
// by lbm3d_f64.cu and lbm3d_f32.cu with LBM3_S and LBM3_NAME defined).
#pragma once

#include "lbm3d_launch.h"

namespace lbm3 {

template <class S, int M, int TY, bool SPLIT>
constexpr auto step3d() {
  if constexpr (SPLIT)
    return step3d_async_kernel<S, M, TY>;
  else
    return step3d_kernel<S, M, TY>;
}

// The step, then the ghost slots of the walls, if there are any.
template <class S, int M, int TY, bool SPLIT>
cudaError_t launch_tile3(const Grid3& g, dim3 grid, int zrows, int lx, cudaStream_t st) {
  constexpr size_t SM = step3d_smem<S, TY, SPLIT>();
  static std::atomic<unsigned long long> allowed{0};
  cudaError_t e = lbm::allow_smem((const void*)step3d<S, M, TY, SPLIT>(), (int)SM, allowed);
  if (e != cudaSuccess) return e;
  if constexpr (SPLIT)
    step3d_async_kernel<S, M, TY><<<grid, threads3<TY, true>(), SM, st>>>(g, zrows);
  else
    step3d_kernel<S, M, TY><<<grid, threads3<TY, false>(), SM, st>>>(g, zrows, lx);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  WallSides w{};
  int sides = 0;
  long long nodes = 0;
  const long long n[3] = {(long long)g.ny * g.nz, (long long)g.nx * g.nz, (long long)g.nx * g.ny};
  for (int s = 0; s < 6; ++s)
    if (g.bc[s] != BC3_PERIODIC) {
      w.side[sides++] = s;
      nodes = n[s / 2] > nodes ? n[s / 2] : nodes;
    }
  if (!sides) return cudaSuccess;
  return lbm::launch_ex(walls3d_kernel<S, M>,
                        dim3((unsigned)((nodes + WALL3_NODES - 1) / WALL3_NODES), sides),
                        WALL3_NODES, 0, st, true, g, w);
}

// Launch shapes (tile rows, separate halo warps): (8, no) for both precisions
// (step3d_kernel); for FP32 storage also (16, no) and, with asynchronous copies
// (step3d_async_kernel), (4, yes) and (8, yes).
template <class S, int M>
cudaError_t launch_mode3(const Grid3& g, dim3 grid, int zrows, int ty, int split, int lx,
                         cudaStream_t st) {
  if constexpr (sizeof(S) == 4) {
    if (ty == 16) return launch_tile3<S, M, 16, false>(g, grid, zrows, lx, st);
    if (ty == 4 && split) return launch_tile3<S, M, 4, true>(g, grid, zrows, lx, st);
    if (ty == 8 && split) return launch_tile3<S, M, 8, true>(g, grid, zrows, lx, st);
  }
  return launch_tile3<S, M, 8, false>(g, grid, zrows, lx, st);
}

template <class S>
cudaError_t launch_step3d(const Grid3& g, dim3 grid, int zrows, int ty, int split, int lx,
                          cudaStream_t st) {
  switch (mode3_of(g)) {
    case M3_TOTAL | M3_ZFULL | M3_CORR:
      return launch_mode3<S, M3_TOTAL | M3_ZFULL | M3_CORR>(g, grid, zrows, ty, split, lx, st);
    case M3_TOTAL | M3_ZFULL:
      return launch_mode3<S, M3_TOTAL | M3_ZFULL>(g, grid, zrows, ty, split, lx, st);
    case M3_TOTAL | M3_CORR:
      return launch_mode3<S, M3_TOTAL | M3_CORR>(g, grid, zrows, ty, split, lx, st);
    case M3_TOTAL:
      return launch_mode3<S, M3_TOTAL>(g, grid, zrows, ty, split, lx, st);
    case M3_CORR:
      return launch_mode3<S, M3_CORR>(g, grid, zrows, ty, split, lx, st);
    case M3_FORCE | M3_CORR:
      return launch_mode3<S, M3_FORCE | M3_CORR>(g, grid, zrows, ty, split, lx, st);
    case M3_FORCE:
      return launch_mode3<S, M3_FORCE>(g, grid, zrows, ty, split, lx, st);
    default:
      return launch_mode3<S, 0>(g, grid, zrows, ty, split, lx, st);
  }
}

template <class S, int TY, bool SPLIT>
cudaError_t attributes3d_tile(int mode, cudaFuncAttributes* a) {
  switch (mode) {
    case M3_TOTAL | M3_ZFULL | M3_CORR:
      return cudaFuncGetAttributes(a, step3d<S, M3_TOTAL | M3_ZFULL | M3_CORR, TY, SPLIT>());
    case M3_TOTAL | M3_ZFULL:
      return cudaFuncGetAttributes(a, step3d<S, M3_TOTAL | M3_ZFULL, TY, SPLIT>());
    case M3_TOTAL | M3_CORR:
      return cudaFuncGetAttributes(a, step3d<S, M3_TOTAL | M3_CORR, TY, SPLIT>());
    case M3_TOTAL:
      return cudaFuncGetAttributes(a, step3d<S, M3_TOTAL, TY, SPLIT>());
    case M3_CORR:
      return cudaFuncGetAttributes(a, step3d<S, M3_CORR, TY, SPLIT>());
    case M3_FORCE | M3_CORR:
      return cudaFuncGetAttributes(a, step3d<S, M3_FORCE | M3_CORR, TY, SPLIT>());
    case M3_FORCE:
      return cudaFuncGetAttributes(a, step3d<S, M3_FORCE, TY, SPLIT>());
    default:
      return cudaFuncGetAttributes(a, step3d<S, 0, TY, SPLIT>());
  }
}

template <class S>
cudaError_t launch_aux3d(int what, const Grid3& g, void* buf, const double* const* in,
                         double* const* out, double T0, double* pops, int* flag, double* partial,
                         int blocks, cudaStream_t st) {
  if (what == AUX3_INIT) {
    if (g.energy_model == 0)
      init3d_kernel<S, true><<<blocks, 256, 0, st>>>(g, static_cast<S*>(buf), in[0], in[1],
                                                      in[2], in[3], in[4], 1.0 / T0);
    else
      init3d_kernel<S, false><<<blocks, 256, 0, st>>>(g, static_cast<S*>(buf), in[0], in[1],
                                                       in[2], in[3], in[4], 1.0 / T0);
  } else if (what == AUX3_EXPORT) {
    export3d_kernel<S><<<blocks, 256, 0, st>>>(
        g, static_cast<const S*>(buf), out ? out[0] : nullptr, out ? out[1] : nullptr,
        out ? out[2] : nullptr, out ? out[3] : nullptr, out ? out[4] : nullptr, T0, pops, flag);
  } else {
    conserved3d_kernel<S><<<blocks, RED3, 0, st>>>(g, static_cast<const S*>(buf), partial);
    conserved3d_final_kernel<><<<1, 32, 0, st>>>(partial, blocks, partial + 5 * blocks);
  }
  return cudaGetLastError();
}

}  // namespace lbm3
