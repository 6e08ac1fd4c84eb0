// Building blocks of the TMA-staged step kernels: the compile-time physics mode
// and the mbarrier / bulk-tensor-copy primitives.
//
// The physics mode (total or internal energy, form of Z, correction, force)
// is a template parameter, so the per-direction code is straight-line.
#pragma once

#include <cuda.h>

#include "lbm_device.cuh"

namespace lbm {

// ---- compile-time physics mode ---------------------------------------------

enum { MODE_TOTAL = 1, MODE_ZFULL = 2, MODE_CORR = 4, MODE_FORCE = 8, MODE_MRT = 16,
       MODE_VARMU = 32 };

// The BGK modes mode_of() produces (total energy with the full or simple Z,
// internal energy with or without gravity; each with or without the
// correction); each has an MRT twin (| MODE_MRT), and each of those a twin
// with a temperature-dependent viscosity (| MODE_VARMU).
constexpr int NUM_BGK_MODES = 8;
constexpr int BGK_MODES[NUM_BGK_MODES] = {MODE_TOTAL | MODE_ZFULL | MODE_CORR,
                                          MODE_TOTAL | MODE_ZFULL,
                                          MODE_TOTAL | MODE_CORR,
                                          MODE_TOTAL,
                                          MODE_FORCE | MODE_CORR,
                                          MODE_FORCE,
                                          MODE_CORR,
                                          0};

template <int M>
struct Mode {
  static constexpr bool total = (M & MODE_TOTAL) != 0;
  static constexpr bool zfull = (M & MODE_ZFULL) != 0;
  static constexpr bool corr = (M & MODE_CORR) != 0;
  static constexpr bool force = (M & MODE_FORCE) != 0;
  static constexpr bool mrt = (M & MODE_MRT) != 0;
  static constexpr bool varmu = (M & MODE_VARMU) != 0;
};

// The eight modes the validated parameters can produce (Z only matters for
// total energy; gravity needs internal energy).
inline int mode_of(const Grid& g) {
  int m = 0;
  if (g.energy_model == E_TOTAL) {
    m |= MODE_TOTAL;
    if (g.z_full) m |= MODE_ZFULL;
  } else if (g.has_force) {
    m |= MODE_FORCE;
  }
  if (g.correction) m |= MODE_CORR;
  if (g.collision == COLL_MRT) m |= MODE_MRT;
  if (g.mu_law != MU_TAU) m |= MODE_VARMU;
  return m;
}

// ---- TMA pipeline primitives ----------------------------------------------

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_test(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for phase `parity` of the barrier, giving up after `limit_ns`.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity,
                                          unsigned long long limit_ns) {
  if (mbar_test(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_test(bar, parity)) {
    if (global_ns() - t0 > limit_ns) return false;
  }
  return true;
}

__device__ __forceinline__ void tma_load_box(unsigned dst, const CUtensorMap* map, unsigned bar,
                                             int cx, int ca, int cy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(cx), "r"(ca), "r"(cy), "r"(bar)
      : "memory");
}

}  // namespace lbm
