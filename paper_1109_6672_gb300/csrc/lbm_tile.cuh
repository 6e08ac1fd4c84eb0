// Tile step kernel (FP64 storage, single grids).
//
// What bounds it: FP64 arithmetic.  GB300's SM starts one FP64 warp instruction
// every 16 clocks (19 unless it is an FMA of three registers) and one warp can
// start one every 64 (measured, independent chains, however many lanes are
// active), and a node's update is about 170 of them.  Memory is idle by
// comparison (288 B a node), so the populations are pulled straight from global
// memory into registers; what matters is that no FP64 work is done twice, that
// every SM gets the same share of it, that at least four warps of an SM are at
// it at any time, and that the chain of one node is short.
//
// A block owns a tile of W x R nodes, one thread per node, plus threads of
// their own for the tile's halo (the row below and above, the columns left and
// right), which only form q = rho u (theta - 1) for the correction's
// differences.  All q go through shared memory over one barrier; the pulled
// populations stay in registers.  W (a power of two up to 32) and R are chosen
// per grid by tile_shape.  The pulled-row kernel's blocks of 128 columns by
// two or more rows left most SMs without work on small grids (a 4 x 33 channel
// used 4 of 128 lanes of 17 blocks, each row's 290 instructions behind the last
// row's): the channel's step took 33 us there and 13 here, a 256^2 cavity's 56
// and 34, a 600 x 4 open channel's 41 (with its second pass) and 8, the 198^2
// large-temperature-difference cavity's 89 and 25.
//
// Sides: walls and periodic copies are written by the edge nodes of the tile
// (wall_side, per side in closed form).  Walls of non-equilibrium
// extrapolation need only the state at time t, so blocks of their own (the
// first of the grid) write their ghost slots in the same launch; open sides are
// written by the edge nodes too (the inlet's six values come with the launch).
//
// Launched with programmatic dependent launch: a block waits for the previous
// step before its first load and lets the next step's blocks start behind it,
// so the next launch's latency overlaps this step.  (The release comes after
// the wait, so no two steps but neighbours are ever in flight; loads bypass L1.)
#pragma once

#include "lbm_node.cuh"
#include "lbm_open.cuh"

namespace lbm {

constexpr int TILE_MAX_NODES = 96;                    // W R
constexpr int TILE_MAX_THREADS = TILE_MAX_NODES + 64;  // plus the halo's 2 W + 2 R nodes
constexpr int GHOST_THREADS = 32;                      // ghosts of one extrapolation block

struct TileArgs {
  int lw, rows;       // log2 W, R
  int tx;             // tiles per row of tiles
  int ghost_blocks;   // blocks of extrapolated wall nodes (first in the grid)
  double fin[3], hin[3];  // the inlet's populations 1, 5, 8 of this step
};

// h^eq of direction A at (rho, u, theta) with the specific energy es, and f^eq.
template <class C, int A>
__device__ __forceinline__ void eq_at(bool total, C rho, C ux, C uy, C th, C es, C& f, C& h) {
  constexpr int e2 = ex(A) * ex(A) + ey(A) * ey(A);
  const C usq = ux * ux + uy * uy;
  const C eu = C(ex(A)) * ux + C(ey(A)) * uy;
  const C w = wgt<C>(e2 == 1 ? 1 : 5);
  const C even = C(4.5) * eu * eu - C(1.5) * usq +
                 (e2 == 1 ? C(0.5) + C(0.5) * th : C(2) * th - C(1));
  const C odd = (e2 == 1 ? C(4.5) - C(1.5) * th : C(3) * th) * eu;
  f = rho * w * (even + odd);
  h = es * f;
  if (total)
    h += w * C(1.0 / 3.0) * (rho * th) *
         (C(9) * eu * eu - C(3) * usq + C(3) * eu + (e2 == 1 ? C(0.5) : C(2)) * th);
}

// State of a boundary node: absolute f*, h* (v), moments, specific energy.
template <class C>
struct EdgeNode {
  const C* v;
  C rho, ux, uy, th, es;
};

// Population A of node (x, y) leaving through wall SIDE comes back as its
// opposite B: f by halfway bounce-back with the moving-wall term, h by the
// ghost equilibrium (isothermal; (rg, ugx, ugy, thg, esg) the ghost's state) or
// bounce-back with the wall's work (adiabatic).  The rules of boundary_writes.
template <class S, bool TOTAL, int SIDE, int A>
__device__ __forceinline__ void wall_one(const Grid& g, S* __restrict__ dst, int x, int y,
                                         const EdgeNode<typename Io<S>::C>& n, bool iso,
                                         typename Io<S>::C rg, typename Io<S>::C ugx,
                                         typename Io<S>::C ugy, typename Io<S>::C thg,
                                         typename Io<S>::C esg) {
  using C = typename Io<S>::C;
  constexpr int B = opp(A);
  constexpr bool diag = ex(A) != 0 && ey(A) != 0;
  const Phys<C>& k = phys<C>(g);
  const C uwx = k.uw[SIDE][0], uwy = k.uw[SIDE][1];
  const C euw = C(ex(A)) * uwx + C(ey(A)) * uwy;
  const C w = wgt<C>(diag ? 5 : 1);
  // odd part of f^eq_A at (rho, u_w, theta)
  const C fodd = n.rho * w * (diag ? C(3) * n.th : C(4.5) - C(1.5) * n.th) * euw;
  const C fb = n.v[A] - C(2) * fodd;
  dst[slot(g, B, x + ex(A), y + ey(A))] = Io<S>::from(fb);
  C hin;
  if (iso) {
    C f, hg, hq;
    eq_at<C, B>(TOTAL, rg, ugx, ugy, thg, esg, f, hg);
    eq_at<C, B>(TOTAL, n.rho, n.ux, n.uy, n.th, n.es, f, hq);
    hin = hg + (n.v[9 + B] - hq);
  } else {
    C hodd;  // odd part of h^eq_A at (rho, u_w, theta)
    if constexpr (TOTAL)
      hodd = (k.b6 * n.th + C(0.5) * (uwx * uwx + uwy * uwy)) * fodd +
             w * (n.rho * n.th) * euw;
    else
      hodd = k.b6 * n.th * fodd;
    hin = n.v[9 + A] - C(2) * hodd;
    if constexpr (TOTAL) hin -= euw * (fb + n.v[A]);  // the wall's work
  }
  dst[slot(g, 9 + B, x + ex(A), y + ey(A))] = Io<S>::from(hin);
}

// The populations leaving node (x, y), which lies on side SIDE, through it.
// xl / xr: a population that also leaves through the x- / x+ side belongs to
// that side's wall (y sides only).
template <class S, bool TOTAL, int SIDE>
__device__ __forceinline__ void wall_side(const Grid& g, S* __restrict__ dst, int x, int y,
                                          const EdgeNode<typename Io<S>::C>& n, bool xl,
                                          bool xr) {
  using C = typename Io<S>::C;
  const Phys<C>& k = phys<C>(g);
  const bool iso = g.bc[SIDE] == BC_ISO;
  C rg = 1, ugx = 0, ugy = 0, thg = 1, esg = 0;
  if (iso) {
    constexpr int ny = SIDE == 2 ? -1 : (SIDE == 3 ? 1 : 0);
    thg = fmax(C(2) * k.thw[SIDE] - n.th, C(0.5) * k.thw[SIDE]);
    rg = n.rho * (n.th - C(3 * ny) * k.g) * rcp_(thg);
    ugx = C(2) * k.uw[SIDE][0] - n.ux;
    ugy = C(2) * k.uw[SIDE][1] - n.uy;
    esg = k.b6 * thg;
    if constexpr (TOTAL) esg += C(0.5) * (ugx * ugx + ugy * ugy);
  }
  // leaving: the axis direction and the diagonals A1 (towards x- or y-) and A2
  constexpr int A0 = SIDE == 0 ? 3 : (SIDE == 1 ? 1 : (SIDE == 2 ? 4 : 2));
  constexpr int A1 = SIDE == 0 ? 7 : (SIDE == 1 ? 8 : (SIDE == 2 ? 7 : 6));
  constexpr int A2 = SIDE == 0 ? 6 : (SIDE == 1 ? 5 : (SIDE == 2 ? 8 : 5));
  wall_one<S, TOTAL, SIDE, A0>(g, dst, x, y, n, iso, rg, ugx, ugy, thg, esg);
  if (!xl) wall_one<S, TOTAL, SIDE, A1>(g, dst, x, y, n, iso, rg, ugx, ugy, thg, esg);
  if (!xr) wall_one<S, TOTAL, SIDE, A2>(g, dst, x, y, n, iso, rg, ugx, ugy, thg, esg);
}

// Every ghost slot that boundary node (x, y) owns.
template <class S, bool TOTAL>
__device__ __forceinline__ void edge_writes(const Grid& g, S* __restrict__ dst, int x, int y,
                                            const EdgeNode<typename Io<S>::C>& n,
                                            const TileArgs& ta) {
  const bool x0 = x == 0, x1 = x == g.nx - 1, y0 = y == 0, y1 = y == g.ny - 1;
  const bool wx0 = x0 && g.bc[0] != BC_PERIODIC, wx1 = x1 && g.bc[1] != BC_PERIODIC;
  const bool wy0 = y0 && g.bc[2] != BC_PERIODIC, wy1 = y1 && g.bc[3] != BC_PERIODIC;
  if (wx0) {
    if (g.bc[0] == BC_INLET) {
      constexpr int A[3] = {1, 5, 8};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        dst[slot(g, A[i], -1, y - ey(A[i]))] = Io<S>::from(ta.fin[i]);
        dst[slot(g, 9 + A[i], -1, y - ey(A[i]))] = Io<S>::from(ta.hin[i]);
      }
    } else if (!(g.nee & 1)) {
      wall_side<S, TOTAL, 0>(g, dst, x, y, n, false, false);
    }
  }
  if (wx1) {
    if (g.bc[1] == BC_OUTLET) {
      // the ghost column copies the last one (y periodic): to where the nodes
      // that the copies reach pull them
      constexpr int A[3] = {3, 6, 7};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int to = y + ey(A[i]);
        const int yy = (to < 0 ? to + g.ny : (to >= g.ny ? to - g.ny : to)) - ey(A[i]);
        dst[slot(g, A[i], x + 1, yy)] = Io<S>::from(n.v[A[i]]);
        dst[slot(g, 9 + A[i], x + 1, yy)] = Io<S>::from(n.v[9 + A[i]]);
      }
    } else if (!(g.nee >> 1 & 1)) {
      wall_side<S, TOTAL, 1>(g, dst, x, y, n, false, false);
    }
  }
  if (wy0 && !(g.nee >> 2 & 1)) wall_side<S, TOTAL, 2>(g, dst, x, y, n, wx0, wx1);
  if (wy1 && !(g.nee >> 3 & 1)) wall_side<S, TOTAL, 3>(g, dst, x, y, n, wx0, wx1);
  // periodic copies: the node at wrap(x + e) pulls population a from there - e
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const bool ox = ex(a) < 0 ? x0 : (ex(a) > 0 ? x1 : false);
    const bool oy = ey(a) < 0 ? y0 : (ey(a) > 0 ? y1 : false);
    const bool wall = (ex(a) < 0 ? wx0 : (ex(a) > 0 ? wx1 : false)) ||
                      (ey(a) < 0 ? wy0 : (ey(a) > 0 ? wy1 : false));
    if (!(ox || oy) || wall) continue;
    const int sx = ox ? (ex(a) < 0 ? g.nx : -1) : x;
    const int sy = oy ? (ey(a) < 0 ? g.ny : -1) : y;
    dst[slot(g, a, sx, sy)] = Io<S>::from(n.v[a]);
    dst[slot(g, 9 + a, sx, sy)] = Io<S>::from(n.v[9 + a]);
  }
}

// One node k of a wall of non-equilibrium extrapolation (the rules of
// nee_ghost in lbm_open.cuh, over pairs): the wall node's pre-collision pairs
// are its equilibria plus the non-equilibrium part of the node F next to it.
template <class S, int M>
__device__ __forceinline__ void tile_ghost(const Grid& g, const S* src, S* __restrict__ dst,
                                           int k) {
  using C = typename Io<S>::C;
  using MD = Mode<M>;
  constexpr int A[4] = {1, 2, 5, 6};
  int side, gx, gy;
  if (k < 2 * (g.ny + 2)) {
    side = k < g.ny + 2 ? 0 : 1;
    gx = side == 0 ? -1 : g.nx;
    gy = k - (side == 0 ? 0 : g.ny + 2) - 1;
  } else {
    k -= 2 * (g.ny + 2);
    side = k < g.nx ? 2 : 3;
    gx = k - (side == 2 ? 0 : g.nx);
    gy = side == 2 ? -1 : g.ny;
  }
  if (!(g.nee >> side & 1)) return;
  const bool xs = side < 2;
  const bool yper = g.bc[2] == BC_PERIODIC, xper = g.bc[0] == BC_PERIODIC;
  const int nxo = side == 0 ? -1 : (side == 1 ? 1 : 0), nyo = side == 2 ? -1 : (side == 3 ? 1 : 0);
  int fx = gx - nxo, fy = gy - nyo;
  bool corner = false;
  if (xs && (gy < 0 || gy >= g.ny)) {
    if (yper) return;
    corner = true;
    fy = gy < 0 ? 0 : g.ny - 1;
  }
  const Phys<C>& kp = phys<C>(g);
  C d[NPOP], qx, qy;
  Pairs<C> q;
  Mom<C> m;
  pull_raw<S>(g, src, fx, fy, d);
  to_pairs(d, q);
  pair_moments<C, M, false>(kp, q, m, qx, qy);
  Mom<C> w;  // the wall node's state
  w.ux = kp.uw[side][0];
  w.uy = kp.uw[side][1];
  const bool adia = g.bc[side] != BC_ISO;
  if (!adia) {
    w.th = kp.thw[side];
  } else {
    C d2[NPOP];
    Pairs<C> q2;
    Mom<C> m2;
    pull_raw<S>(g, src, fx - nxo, fy - nyo, d2);
    to_pairs(d2, q2);
    pair_moments<C, M, false>(kp, q2, m2, qx, qy);
    w.th = fmax((C(4) * m.th - m2.th) * C(1.0 / 3.0), C(0.5) * m.th);
  }
  w.r0 = m.r0 * (m.th - C(3) * kp.g * C(nyo)) * rcp_(w.th);
  const C uw2 = w.ux * w.ux + w.uy * w.uy;
  w.es = kp.b6 * w.th + (MD::total ? C(0.5) * uw2 : C(0));
  w.sh = C(0);
  Shells<C> ef, ew;
  pair_shells<C, MD::total, false>(kp, m.r0, m, ef);
  pair_shells<C, MD::total, false>(kp, w.r0, w, ew);
  // F's pairs less twice its equilibria; the normal heat flux of that part of h
  // (less the wall's viscous work) is taken out on an adiabatic wall
  C en[4], qn = C(0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = i >> 1;
    const C e2 = ef.eu[i] * ef.eu[i];
    q.S[i] -= C(2) * (ef.A[s] + ef.B[s] * e2);
    q.D[i] -= C(2) * (ef.L[s] * ef.eu[i]);
    q.Sh[i] -= C(2) * (ef.HA[s] + ef.HB[s] * e2);
    q.Dh[i] -= C(2) * (ef.HL[s] * ef.eu[i]);
    en[i] = C(ex(A[i]) * nxo + ey(A[i]) * nyo);
    C hn = q.Dh[i];
    if constexpr (MD::total) {
      const C zw2 = MD::zfull ? C(0.5) * uw2 : C(0);
      hn -= ew.eu[i] * q.S[i] - zw2 * q.D[i];
    }
    qn += en[i] * hn;
  }
  if (!adia) qn = C(0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = i >> 1;
    const C e2 = ew.eu[i] * ew.eu[i];
    q.S[i] += C(2) * (ew.A[s] + ew.B[s] * e2);
    q.D[i] += C(2) * (ew.L[s] * ew.eu[i]);
    q.Sh[i] += C(2) * (ew.HA[s] + ew.HB[s] * e2);
    q.Dh[i] += C(2) * (ew.HL[s] * ew.eu[i]) - C(i < 2 ? 6.0 / 9.0 : 6.0 / 36.0) * en[i] * qn;
  }
  C v[NPOP];
  pair_collide<C, M & ~MODE_CORR, false>(kp, g.mu_law, q, w, C(0), C(0), v);
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    if (ex(a) * nxo + ey(a) * nyo >= 0) continue;  // not into the domain
    int dx = gx + ex(a), dy = gy + ey(a);
    if (corner) {
      if (dx != fx || dy != fy) continue;  // a corner ghost feeds the corner node only
    } else {
      if (dx < 0 || dx >= g.nx) {
        if (!xper) continue;  // the x side's rule has it
        dx = dx < 0 ? dx + g.nx : dx - g.nx;
      }
      if (dy < 0 || dy >= g.ny) {
        if (!yper) continue;
        dy = dy < 0 ? dy + g.ny : dy - g.ny;
      }
    }
    dst[slot(g, a, dx - ex(a), dy - ey(a))] = Io<S>::from(v[a]);
    dst[slot(g, 9 + a, dx - ex(a), dy - ey(a))] = Io<S>::from(v[9 + a]);
  }
}

template <class S, int M>
__global__ void __launch_bounds__(TILE_MAX_THREADS, 3)
    step_tile_kernel(const __grid_constant__ Grid g, const __grid_constant__ TileArgs ta) {
  using C = typename Io<S>::C;
  using MD = Mode<M>;
  static_assert(sizeof(S) == 8, "the tile kernel reads and writes FP64 storage");
  __shared__ C qxs[TILE_MAX_NODES + 2 * 32];  // [R][W + 2], R <= 32
  __shared__ C qys[TILE_MAX_NODES + 2 * 32];  // [R + 2][W]
  const S* src = static_cast<const S*>(g.src);
  S* __restrict__ dst = static_cast<S*>(g.dst);
  const int t = threadIdx.x;
  pdl_wait();
  pdl_release();
  int b = blockIdx.x;
  if (b < ta.ghost_blocks) {
    const int k = b * GHOST_THREADS + t;
    if (t < GHOST_THREADS && k < nee_ghosts(g)) tile_ghost<S, M>(g, src, dst, k);
    return;
  }
  b -= ta.ghost_blocks;
  const int W = 1 << ta.lw, R = ta.rows;
  const int by = b / ta.tx;
  const int x0 = (b - by * ta.tx) * W, y0 = by * R;
  const int nx = g.nx, ny = g.ny;
  const int w = min(W, nx - x0), rr = min(R, ny - y0);  // the tile's nodes
  const int nodes = W * R;
  const int first_halo = (nodes + 31) & ~31;

  int x = 0, y = 0, lx = 0, ly = 0, what = 0;  // 0 idle, 1 node, 2..5 halo of side what - 2
  if (t < first_halo) {
    lx = t & (W - 1);
    ly = t >> ta.lw;
    x = x0 + lx;
    y = y0 + ly;
    what = (t < nodes && lx < w && ly < rr) ? 1 : 0;
  } else if (MD::corr) {
    const int hh = t - first_halo;
    if (hh < 2 * W) {  // below, above
      lx = hh & (W - 1);
      what = lx < w ? (hh < W ? 4 : 5) : 0;
      ly = what == 4 ? -1 : rr;
    } else if (hh < 2 * W + 2 * R) {  // left, right
      ly = (hh - 2 * W) >> 1;
      what = ly < rr ? 2 + (hh & 1) : 0;
      lx = what == 2 ? -1 : w;
    }
    x = x0 + lx;
    y = y0 + ly;
    if (x < 0) {
      if (g.bc[0] != BC_PERIODIC) what = 0;
      x += nx;
    } else if (x >= nx) {
      if (g.bc[1] != BC_PERIODIC) what = 0;
      x -= nx;
    }
    if (y < 0) {
      if (g.bc[2] != BC_PERIODIC) what = 0;
      y += ny;
    } else if (y >= ny) {
      if (g.bc[3] != BC_PERIODIC) what = 0;
      y -= ny;
    }
  }
  const Phys<C>& k = phys<C>(g);
  Pairs<C> q;
  Mom<C> m;
  C qx = 0, qy = 0;
  if (what) {
    C d[NPOP];
    pull_raw<S>(g, src, x, y, d);
    to_pairs(d, q);
    pair_moments<C, M, false>(k, q, m, qx, qy);
  }
  C dx = 0, dy = 0;
  if constexpr (MD::corr) {
    if (what == 1 || what == 2 || what == 3) qxs[ly * (W + 2) + lx + 1] = qx;
    if (what == 1 || what >= 4) qys[(ly + 1) * W + lx] = qy;
    __syncthreads();
    if (what == 1) {
      const bool ml = x == 0 && g.bc[0] != BC_PERIODIC, mr = x == nx - 1 && g.bc[1] != BC_PERIODIC;
      const bool mb = y == 0 && g.bc[2] != BC_PERIODIC, mt = y == ny - 1 && g.bc[3] != BC_PERIODIC;
      const C l = ml ? mirror_q<C>(g, 0, 0, m.r0, m.th, qx) : qxs[ly * (W + 2) + lx];
      const C r = mr ? mirror_q<C>(g, 1, 0, m.r0, m.th, qx) : qxs[ly * (W + 2) + lx + 2];
      const C dn = mb ? mirror_q<C>(g, 2, 1, m.r0, m.th, qy) : qys[ly * W + lx];
      const C up = mt ? mirror_q<C>(g, 3, 1, m.r0, m.th, qy) : qys[(ly + 2) * W + lx];
      dx = r - l;
      dy = up - dn;
    }
  }
  if (what != 1) return;
  C v[NPOP];
  pair_collide<C, M, false>(k, g.mu_law, q, m, dx, dy, v);
  S* p = dst + slot(g, 0, x, y);
#pragma unroll
  for (int a = 0; a < NPOP; ++a) p[(plane(a) - plane(0)) * g.pitch] = Io<S>::from(v[a]);
  if (x == 0 || y == 0 || x == nx - 1 || y == ny - 1) {
    const EdgeNode<C> n{v, m.r0, m.ux, m.uy, m.th, m.es};
    edge_writes<S, MD::total>(g, dst, x, y, n, ta);
  }
}

}  // namespace lbm
