// D3Q19 kernels with FP64 storage and arithmetic.
#include "lbm3d_inst.cuh"

namespace lbm3 {
cudaError_t launch_step3d_f64(const Grid3& g, dim3 grid, int zrows, int ty, int split, int lx,
                              cudaStream_t st) {
  return launch_step3d<double>(g, grid, zrows, ty, split, lx, st);
}
cudaError_t launch_aux3d_f64(int what, const Grid3& g, void* buf, const double* const* in,
                             double* const* out, double T0, double* pops, int* flag,
                             double* partial, int blocks, cudaStream_t st) {
  return launch_aux3d<double>(what, g, buf, in, out, T0, pops, flag, partial, blocks, st);
}
}  // namespace lbm3
