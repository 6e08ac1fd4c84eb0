// Tile step kernel, FP64 storage: the launch (lbm_tile.cuh has the kernel).
#include <algorithm>
#include <cmath>

#include "lbm_launch.h"
#include "lbm_step_inst.cuh"
#include "lbm_tile.cuh"

namespace lbm {

namespace {

// FP64 instructions of a warp: a node's update, and a halo node's moments.
constexpr int COST_NODE = 170, COST_HALO = 40;

}  // namespace

// Tile of a grid: the shape whose fullest SM has the fewest FP64 instructions.
// Tiles stay at 96 nodes, so that three blocks and more share an SM: with up to
// 256 nodes a tile, a 256^2 cavity in 16 x 14 tiles (two blocks an SM, one at a
// time; 2540 instructions on the fullest SM) took 38 us a step, in 8 x 12 tiles
// (five an SM; 2950) 33.7, in 32 x 4 tiles (four; 3200) 37.9; the 198^2 cavity
// 24.6 in 16 x 6 (1770), 33.6 in 16 x 8 (2280).
// rows > 0: that many rows per tile (as many as fit the nodes and, with the
// correction, the halo's two warps).  W = 1 always gives a tile.
void tile_shape(int nx, int ny, bool corr, int sms, int rows, int* lw_out, int* rows_out) {
  long long best = -1;
  for (int lw = 5; lw >= 0; --lw) {
    const int W = 1 << lw;
    if (lw > 0 && W / 2 >= nx) continue;  // a narrower tile holds the row
    const int most =
        std::min({TILE_MAX_NODES / W, 32, ny, rows > 0 ? rows : 32,
                  corr ? (TILE_MAX_THREADS - TILE_MAX_NODES) / 2 - W : 32});  // 2 W + 2 R
    for (int R = rows > 0 ? std::max(most, 1) : 1; R <= most; ++R) {
      const int warps = (W * R + 31) / 32, halo = corr ? (2 * W + 2 * R + 31) / 32 : 0;
      const long long blocks = (long long)((nx + W - 1) / W) * ((ny + R - 1) / R);
      const long long cost = (blocks + sms - 1) / sms * (warps * COST_NODE + halo * COST_HALO);
      if (best < 0 || cost < best) {
        best = cost;
        *lw_out = lw;
        *rows_out = R;
      }
    }
  }
}

cudaError_t launch_step_tile(const Grid& g, int lw, int rows, cudaStream_t stream) {
  TileArgs ta{};
  ta.lw = lw;
  ta.rows = rows;
  const int W = 1 << lw;
  ta.tx = (g.nx + W - 1) / W;
  ta.ghost_blocks = g.nee ? (nee_ghosts(g) + GHOST_THREADS - 1) / GHOST_THREADS : 0;
  if (g.bc[0] == BC_INLET) {
    // Eq. 53's state at step t and its equilibria (Eq. 18a, 18b or Eq. 38)
    const double sn = std::sin(g.in_omega * (double)g.t);
    const double rho = g.in_rho + g.in_drho * sn, th = g.pd.thw[0] + g.in_dth * sn;
    const double ux = g.pd.uw[0][0] + g.in_du * sn, uy = g.pd.uw[0][1];
    const double usq = ux * ux + uy * uy;
    const bool total = g.energy_model == E_TOTAL;
    const double es = g.pd.b6 * th + (total ? 0.5 * usq : 0.0), p = rho * th / 3.0;
    const int A[3] = {1, 5, 8};
    for (int i = 0; i < 3; ++i) {
      const int a = A[i];
      const double e2 = i == 0 ? 1.0 : 2.0, w = i == 0 ? 1.0 / 9.0 : 1.0 / 36.0;
      const double eu = ex(a) * ux + ey(a) * uy;
      ta.fin[i] = rho * w * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * usq +
                             (th - 1.0) * (1.5 * e2 - 1.0) +
                             1.5 * eu * (th - 1.0) * (3.0 * e2 - 4.0));
      ta.hin[i] = es * ta.fin[i];
      if (total)
        ta.hin[i] += w * p * (3.0 * eu + 9.0 * eu * eu - 3.0 * usq + th * (1.5 * e2 - 1.0));
    }
  }
  const int warps = (W * rows + 31) / 32;
  const int halo = g.correction ? (2 * W + 2 * rows + 31) / 32 : 0;
  const dim3 grid(ta.ghost_blocks + ta.tx * ((g.ny + rows - 1) / rows));
  return dispatch_mode<true>(mode_of(g), [&](auto m) {
    return launch_ex(step_tile_kernel<double, decltype(m)::value>, grid, 32 * (warps + halo), 0,
                     stream, true, g, ta);
  });
}

}  // namespace lbm
