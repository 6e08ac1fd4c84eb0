// Pulled-row step over pairs of columns (FP32 and 16-bit storage).
//
// What bounds it: HBM for FP32 storage on grids beyond L2 (144 B a node), issued
// instructions and their latency for everything else.  The earlier kernel
// (lbm_step_pr.cuh: one column a thread, the update per direction) issued 663
// thread instructions a node with FP32 and 739 with 16-bit storage (ncu, 2048^2
// box).  Here a thread owns two adjacent columns, so that
//  - the update (lbm_node.cuh, over opposite pairs) runs in packed FP32, two
//    nodes an instruction;
//  - stores are one 8-byte (FP32) or 4-byte (16-bit) word per population, and a
//    16-bit conversion rounds both nodes' values of a population at once,
// and a node takes 331 (in blocks of 5 rows) and 390.  us a step (without reads of the fields), before ->
// after: 1024^2 cavity BF16 37.0 -> 26.7, 3001 x 2003 box FP16 169.6 -> 134.0, 512^2
// cavity FP32 13.2 -> 8.9, 1733 x 1021 MRT channel with a power-law viscosity FP32
// 71.5 -> 54.8, 4096^2 box FP32 373.2 -> 350.8 (at the measured copy rate).
// FP16 storage holds 256 x the deviation; the update runs on the scaled values
// (every term is linear in them), which saves the scalings of loads and stores.
//
// Staging is that of the earlier kernel: the 18 values that row r pulls are three
// contiguous plane groups (e_y = +1 of row r - 1, 0 of row r, -1 of row r + 1),
// each one TMA box; a ring of D pulled rows, guarded by mbarriers.  A block is two
// warps of nodes (128 columns) and a helper warp that issues the copies and
// forms q_x of the two columns beside the strip; one barrier a row publishes q_x
// and frees the slot of row r - 1.
//
// Registers decide: the L1 left beside the rings is small, so most of what is
// spilled goes to L2 (a version that kept the populations of the held row in registers
// spilled about 100 bytes a row and took 1.3 to 2 times as long).  So a row is
// read from its slot twice, for q and for the collision, its moments are formed
// again, the two roles have loops of their own, and nothing but the update itself
// is in the row loop.  At 128 registers FP32 storage spills nothing; 16-bit storage,
// whose 18 packed results and random words are live together, 8 to 44 bytes (28 in the
// cavity's mode).  (Without a helper, each warp on its own with 64 columns and
// 12 to 16 warps an SM, the halo columns cost every warp a pass of its own: 376
// and 488 instructions a node, 1024^2 BF16 31.1 us, 3001 x 2003 FP16 206.)
//
// Ghost slots are written after the last row: periodic copies from the stored
// values, a walled x side's from records that its nodes left in shared memory (one
// thread per population), a y side's by the threads of its row.  Open sides and
// walls of non-equilibrium extrapolation are rewritten by side_fixup_kernel.
//
// Waits are bounded (2 s); see pr_block.
#pragma once

#include "lbm_node.cuh"
#include "lbm_step_pr.cuh"

namespace lbm {

constexpr int PAIR_COLS = 128;                   // columns per block
constexpr int PAIR_COMPUTE = PAIR_COLS / 2;      // threads that own columns
constexpr int PAIR_THREADS = PAIR_COMPUTE + 32;  // plus the helper warp

// ---- 32-bit words of two columns -------------------------------------------

template <class S>
struct PairIo;
template <>
struct PairIo<float> {
  static constexpr int scale = 1;
  using W = float2;
  __device__ __forceinline__ static F2 ld(const float* p) {
    return mk2(*reinterpret_cast<const float2*>(p));
  }
  __device__ __forceinline__ static F2 ld_two(const float* p) { return F2(p[0], p[1]); }
  __device__ __forceinline__ static float one(float v) { return v; }
  __device__ __forceinline__ static W pack(F2 v, unsigned) { return v.v; }
  __device__ __forceinline__ static float lo(W w) { return w.x; }
  __device__ __forceinline__ static float hi(W w) { return w.y; }
};
template <>
struct PairIo<__nv_bfloat16> {
  static constexpr int scale = 1;
  using W = unsigned;
  using S = __nv_bfloat16;
  __device__ __forceinline__ static F2 ld(const S* p) {
    const unsigned w = *reinterpret_cast<const unsigned*>(p);
    return F2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  }
  __device__ __forceinline__ static float one(S v) {
    return __uint_as_float((unsigned)__bfloat16_as_ushort(v) << 16);
  }
  __device__ __forceinline__ static F2 ld_two(const S* p) { return F2(one(p[0]), one(p[1])); }
  // bits 31-16 of r round the second column's value, bits 15-0 the first's
  __device__ __forceinline__ static W pack(F2 v, unsigned r) {
    unsigned d;
    asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(r));
    return d;
  }
  __device__ __forceinline__ static S lo(W w) {
    return __ushort_as_bfloat16((unsigned short)(w & 0xFFFFu));
  }
  __device__ __forceinline__ static S hi(W w) {
    return __ushort_as_bfloat16((unsigned short)(w >> 16));
  }
};
template <>
struct PairIo<__half> {
  static constexpr int scale = 256;
  using W = unsigned;
  using S = __half;
  __device__ __forceinline__ static F2 ld(const S* p) {
    return mk2(__half22float2(*reinterpret_cast<const __half2*>(p)));
  }
  __device__ __forceinline__ static float one(S v) { return __half2float(v); }
  __device__ __forceinline__ static F2 ld_two(const S* p) { return F2(one(p[0]), one(p[1])); }
  __device__ __forceinline__ static W pack(F2 v, unsigned r) {
    unsigned d;
    asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(r));
    return d;
  }
  __device__ __forceinline__ static S lo(W w) {
    return __ushort_as_half((unsigned short)(w & 0xFFFFu));
  }
  __device__ __forceinline__ static S hi(W w) { return __ushort_as_half((unsigned short)(w >> 16)); }
};

// ---- geometry of a block's shared memory -----------------------------------

// Four staged rows of 10.4 KB (FP32) or 5.2 KB (16-bit): two are being read, two
// in flight.  Five blocks an SM (128 registers a thread; six would leave 96,
// which spill).
template <class S>
struct PairGeom {
  static constexpr int LEFT = 8;
  static constexpr int BOX = PAIR_COLS + 2 * LEFT;  // columns x0 - 8 .. x0 + 135
  static constexpr int GB =  // elements per box, 128-byte multiple
      (int)(((size_t)6 * BOX * sizeof(S) + 127) / 128 * 128 / sizeof(S));
  static constexpr int SLOT = 3 * GB;
  static constexpr int D = 4;
  static constexpr int BLOCKS = 5;
  static constexpr unsigned BOX_BYTES = 6 * BOX * sizeof(S);
  static constexpr int QROW = PAIR_COLS + 4;  // column c at c + 2, halos at 1 and c_end + 2
  static constexpr int XROWS = 8;             // rows of x-edge records
  static constexpr int XVALS = 15;            // 14 used
  static constexpr size_t OFF_Q = (size_t)D * SLOT * sizeof(S);
  static constexpr size_t OFF_REC = OFF_Q + 2 * QROW * sizeof(float);
  static constexpr size_t OFF_BAR = OFF_REC + 2 * XROWS * XVALS * sizeof(float);
  static constexpr size_t BYTES = OFF_BAR + 8 * D;
  static_assert((GB * sizeof(S)) % 128 == 0 && OFF_BAR % 8 == 0, "alignment");
};

// Pulled populations of two adjacent columns from a slot; sc: staged column of
// the first (even).  one: of a single column, in both halves.
template <class S>
__device__ __forceinline__ void pair_pull(const S* slot, int sc, F2 d[NPOP]) {
  using G = PairGeom<S>;
#pragma unroll
  for (int a = 0; a < NPOP; ++a) {
    const int grp = pgroup(a), lp = plane(a) - 6 * grp;
    const S* p = slot + grp * G::GB + lp * G::BOX + sc - ex(a % 9);
    d[a] = ex(a % 9) == 0 ? PairIo<S>::ld(p) : PairIo<S>::ld_two(p);
  }
}

// ---- x-edge records ---------------------------------------------------------

// Population B (the opposite of the leaving A) of a recorded node: index and
// plane from its velocity.
__device__ __forceinline__ int pop_of(int vx, int vy) {
  return vy == 0 ? (vx > 0 ? 1 : 3) : (vy > 0 ? (vx > 0 ? 5 : 6) : (vx > 0 ? 8 : 7));
}

// f^eq and h^eq of direction (vx, vy) != 0 at (rho, u, theta) with the specific
// energy es.
template <class C>
__device__ __forceinline__ void eq_dir_rt(bool total, C vx, C vy, bool diag, C rho, C ux, C uy,
                                          C th, C es, C& f, C& h) {
  const C usq = ux * ux + uy * uy;
  const C eu = vx * ux + vy * uy;
  const C w = diag ? C(1.0f / 36.0f) : C(1.0f / 9.0f);
  const C even = C(4.5f) * eu * eu + C(-1.5f) * usq +
                 (diag ? C(2.0f) * th + C(-1.0f) : C(0.5f) * th + C(0.5f));
  const C odd = (diag ? C(3.0f) * th : C(-1.5f) * th + C(4.5f)) * eu;
  f = rho * w * (even + odd);
  h = es * f;
  if (total)
    h = h + w * (rho * th) * C(1.0f / 3.0f) *
                (C(9.0f) * eu * eu + C(-3.0f) * usq + C(3.0f) * eu +
                 (diag ? C(2.0f) : C(0.5f)) * th);
}

// What comes back for a population A = (vx, vy) leaving a boundary node through
// wall `side` (the rules of boundary_writes): fb, hin, absolute values.
template <class C>
__device__ __forceinline__ void wall_back(const Grid& g, int side, bool total, C vx, C vy,
                                          bool diag, C fA, C hA, C hB, C rho, C ux, C uy, C th,
                                          C es, C thg, C inv_thg, C& fb, C& hin) {
  const Phys<float>& k = g.pf;
  const C uwx = C(k.uw[side][0]), uwy = C(k.uw[side][1]);
  const C euw = vx * uwx + vy * uwy;
  const C w = diag ? C(1.0f / 36.0f) : C(1.0f / 9.0f);
  const C fodd = rho * w * (diag ? C(3.0f) * th : C(-1.5f) * th + C(4.5f)) * euw;
  fb = fA + C(-2.0f) * fodd;
  if (g.bc[side] == BC_ISO) {
    // the ghost: theta linear through the wall (thg, floored), u mirrored, the
    // node's pressure carried by hydrostatic balance
    const float ny = side == 2 ? -1.0f : (side == 3 ? 1.0f : 0.0f);
    const C rg = rho * (th + C(-3.0f * k.g * ny)) * inv_thg;
    const C ugx = uwx + uwx + C(-1.0f) * ux, ugy = uwy + uwy + C(-1.0f) * uy;
    const C esg = C(k.b6) * thg + (total ? C(0.5f) * (ugx * ugx + ugy * ugy) : C(0.0f));
    C f, hg, hq;
    eq_dir_rt<C>(total, C(-1.0f) * vx, C(-1.0f) * vy, diag, rg, ugx, ugy, thg, esg, f, hg);
    eq_dir_rt<C>(total, C(-1.0f) * vx, C(-1.0f) * vy, diag, rho, ux, uy, th, es, f, hq);
    hin = hg + (hB + C(-1.0f) * hq);
  } else {
    C hodd = C(k.b6) * th * fodd;
    if (total)
      hodd = hodd + C(0.5f) * (uwx * uwx + uwy * uwy) * fodd + w * (rho * th) * euw;
    hin = hA + C(-2.0f) * hodd;
    if (total) hin = hin + C(-1.0f) * euw * (fb + fA);  // the wall's work
  }
}

// Ghost slots of the x sides for rows [row0, row0 + n), one thread per (row,
// side, population): walls from the records, periodic copies (of the stored
// values) where the block holds the side's column.
template <class S, int M>
__device__ __forceinline__ void pair_xsides(const Grid& g, S* __restrict__ dst, const float* rec,
                                            int row0, int n, bool xl, bool xr) {
  using G = PairGeom<S>;
  using MD = Mode<M>;
  for (int i = threadIdx.x; i < 6 * n; i += PAIR_COMPUTE) {
    const int row = i / 6, side = (i / 3) & 1, dir = i % 3;
    if (side ? !xr : !xl) continue;
    const int vx = side ? 1 : -1, vy = dir == 0 ? 0 : (dir == 1 ? 1 : -1);
    const int x = side ? g.nx - 1 : 0, y = row0 + row;
    if (g.bc[side] == BC_PERIODIC) {
      // population A leaves through the side: to the opposite ghost column, and
      // across a periodic y side's corner; a y wall's corner is that wall's
      const bool oy = vy < 0 ? y == 0 : (vy > 0 ? y == g.ny - 1 : false);
      if (oy && g.bc[vy < 0 ? 2 : 3] != BC_PERIODIC) continue;
      const int A = pop_of(vx, vy);
      const int gx = side ? -1 : g.nx, gy = oy ? (vy < 0 ? g.ny : -1) : y;
      dst[slot(g, A, gx, gy)] = dst[slot(g, A, x, y)];
      dst[slot(g, 9 + A, gx, gy)] = dst[slot(g, 9 + A, x, y)];
      continue;
    }
    const float* r = rec + (row * 2 + side) * G::XVALS;
    const float rho = r[9], ux = r[10], uy = r[11], th = r[12], es = r[13];
    const float thw = g.pf.thw[side];
    const float thg = fmaxf(2.0f * thw - th, 0.5f * thw);
    float fb, hin;
    wall_back<float>(g, side, MD::total, (float)vx, (float)vy, vy != 0, r[dir], r[3 + dir],
                     r[6 + dir], rho, ux, uy, th, es, thg, 1.0f / thg, fb, hin);
    const int B = pop_of(-vx, -vy);
    const unsigned h = Io<S>::sr ? sr_hash(g, x, y) : 0u;
    put<S>(g, dst, B, x + vx, y + vy, fb, h, 18 + B);
    put<S>(g, dst, 9 + B, x + vx, y + vy, hin, h, 27 + B);
  }
}

// ---- first and last rows ----------------------------------------------------

// What a thread keeps of its two nodes in the first (up = 0) or last row: f*,
// h* of the three populations leaving through the y side, h* of their
// opposites, and the moments (absolute, unscaled).
struct YEdge {
  F2 f[3], h[3], hb[3], rho, ux, uy, th, es;
};

// Ghost slots of y side `up` that columns c and c + 1 of row y own: walls, or
// copies of the stored values.  A population that also leaves through an x side
// is left to that side if it is a wall or periodic along with y.
template <class S, int M>
__device__ __forceinline__ void pair_yside(const Grid& g, S* __restrict__ dst, int c, int y,
                                           bool has2, int up, const YEdge& e) {
  using MD = Mode<M>;
  const int nx = g.nx, ny = g.ny;
  const int side = 2 + up, vy = up ? 1 : -1;
  const bool wall = g.bc[side] != BC_PERIODIC;
  const float thw = g.pf.thw[side];
  const F2 thg(fmaxf(2.0f * thw - e.th.v.x, 0.5f * thw), fmaxf(2.0f * thw - e.th.v.y, 0.5f * thw));
  const F2 inv_thg(1.0f / thg.v.x, 1.0f / thg.v.y);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int vx = d == 0 ? 0 : (d == 1 ? 1 : -1);
    const int A = d == 0 ? (up ? 2 : 4) : pop_of(vx, vy);
    const int B = d == 0 ? (up ? 4 : 2) : pop_of(-vx, -vy);
    F2 fb = F2(0.0f), hin = F2(0.0f);
    if (wall)
      wall_back<F2>(g, side, MD::total, F2((float)vx), F2((float)vy), vx != 0, e.f[d], e.h[d],
                    e.hb[d], e.rho, e.ux, e.uy, e.th, e.es, thg, inv_thg, fb, hin);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int x = c + i;
      if (i == 1 && !has2) continue;
      const bool ol = vx < 0 && x == 0, orr = vx > 0 && x == nx - 1;
      if (wall) {
        if ((ol && g.bc[0] != BC_PERIODIC) || (orr && g.bc[1] != BC_PERIODIC)) continue;
        const unsigned h = Io<S>::sr ? sr_hash(g, x, y) : 0u;
        put<S>(g, dst, B, x + vx, y + vy, i ? fb.v.y : fb.v.x, h, 18 + B);
        put<S>(g, dst, 9 + B, x + vx, y + vy, i ? hin.v.y : hin.v.x, h, 27 + B);
      } else {
        if (ol || orr) continue;  // the x side's wall, or its periodic copy
        const int gy = up ? -1 : ny;
        dst[slot(g, A, x, gy)] = dst[slot(g, A, x, y)];
        dst[slot(g, 9 + A, x, gy)] = dst[slot(g, 9 + A, x, y)];
      }
    }
  }
}

// ---- a block's share ----------------------------------------------------------

// Initialise the ring's mbarriers (once per kernel, all threads call).
template <class S>
__device__ __forceinline__ void pair_init(unsigned char* smem) {
  using G = PairGeom<S>;
  if (threadIdx.x == 0) {
    const unsigned bar = smem_u32(smem + G::OFF_BAR);
    for (int i = 0; i < G::D; ++i) mbar_init(bar + 8 * i, 1);
    mbar_fence_init();
  }
  __syncthreads();
}

// Row barrier of the block's 96 threads; any thread's `bad` reaches all.
__device__ __forceinline__ bool pair_barrier(bool bad) {
  unsigned r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, 96, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((unsigned)bad)
      : "memory");
  return r != 0;
}
static_assert(PAIR_THREADS == 96, "barrier 1 counts the block's threads");
// Barrier of the threads that own columns.
__device__ __forceinline__ void pair_compute_barrier() {
  asm volatile("barrier.cta.sync 2, 64;" ::: "memory");
}
static_assert(PAIR_COMPUTE == 64, "barrier 2 counts the threads that own columns");

constexpr unsigned long long PAIR_WAIT_NS = 2000000000ull;  // 2 s

// The helper warp's part of a block's share (pair_block): lane 0 issues the
// copies, lanes 0 and 1 form q_x of the columns left and right of the strip.
template <class S, int M>
__device__ __forceinline__ int pair_helper(const Grid& g, const CUtensorMap* map, const S* src,
                                           int x0, int y0, int y1, int rs, int nq,
                                           unsigned char* smem, int kbase, int pre,
                                           const PrNext& next, int* pre_out) {
  using G = PairGeom<S>;
  using MD = Mode<M>;
  using IO = PairIo<S>;
  constexpr int D = G::D;
  const S* ring = reinterpret_cast<const S*>(smem);
  float* qxs = reinterpret_cast<float*>(smem + G::OFF_Q);
  const unsigned ring_s = smem_u32(ring), bar_s = smem_u32(smem + G::OFF_BAR);
  const int hl = threadIdx.x - PAIR_COMPUTE, nx = g.nx, ny = g.ny;
  int issued = pre;
  auto issue_upto = [&](int kmax) {
    kmax = min(kmax, nq + next.nq - 1);
    for (; issued <= kmax; ++issued) {
      const int s = (kbase + issued) % D;
      const unsigned bar = bar_s + 8 * s;
      const bool own = issued < nq;
      const CUtensorMap* mp = own ? map : next.map;
      const int xs = own ? x0 : next.x0, yn = own ? ny : next.ny;
      int nr = own ? rs + issued : next.rs + (issued - nq);
      nr = nr < 0 ? nr + yn : (nr >= yn ? nr - yn : nr);
      mbar_expect_tx(bar, 3 * G::BOX_BYTES);
#pragma unroll
      for (int grp = 0; grp < 3; ++grp)
        tma_load_box(ring_s + (unsigned)((s * G::SLOT + grp * G::GB) * sizeof(S)), mp, bar,
                     xs - G::LEFT + XOFF, 6 * grp, nr + grp);
    }
  };
  if (hl == 0) issue_upto(D - 2);
  const int right = min(PAIR_COLS, nx - x0);  // local column right of the nodes
  int hsrc = 0, hcol = 0;                     // 0 none, 1 ring, 2 global (wrapped)
  if (MD::corr && hl < 2) {
    const int hc = hl == 0 ? x0 - 1 : x0 + right;
    if (hc >= 0 && hc < nx) {
      hsrc = 1;
      hcol = hc - x0 + G::LEFT;  // staged column
    } else if (g.bc[hl] == BC_PERIODIC) {
      hsrc = 2;
      hcol = hl == 0 ? nx - 1 : 0;
    }
  }
  // a wrapped column is not staged: its row's values are loaded a row ahead
  float hd[NPOP];
  auto load_row = [&](int r) {
    r = r < 0 ? r + ny : (r >= ny ? r - ny : r);
    const S* p = src + slot(g, 0, hcol, r);
#pragma unroll
    for (int a = 0; a < NPOP; ++a)
      hd[a] = IO::one(__ldcg(p + (plane(a) - plane(0)) * g.pitch - ey(a % 9) * g.rp - ex(a % 9)));
  };
  if (hsrc == 2) load_row(rs);
  int qs = 0;
#pragma unroll 1
  for (int r = y0 - 1; r <= y1; ++r) {
    bool ok = true;
    const int k = r - rs;
    if (k >= 0 && k < nq) {
      const int s = (kbase + k) % D;
      ok = mbar_wait(bar_s + 8 * s, ((kbase + k) / D) & 1, PAIR_WAIT_NS);
      if (hsrc) {
        if (hsrc == 1) {
          const S* p = ring + s * G::SLOT + hcol;
#pragma unroll
          for (int a = 0; a < NPOP; ++a) {
            const int grp = pgroup(a), lp = plane(a) - 6 * grp;
            hd[a] = IO::one(p[grp * G::GB + lp * G::BOX - ex(a % 9)]);
          }
        }
        // (both halves of a packed pair: the arithmetic of the nodes' own q)
        F2 d[NPOP], qx, qy;
#pragma unroll
        for (int a = 0; a < NPOP; ++a) d[a] = F2(hd[a]);
        Pairs<F2> q;
        Mom<F2> m;
        to_pairs(d, q);
        pair_moments<F2, M, Io<S>::dev, IO::scale>(g.pf, q, m, qx, qy);
        qxs[qs * G::QROW + (hl == 0 ? 1 : right + 2)] = qx.v.x;
        if (hsrc == 2 && k + 1 < nq) load_row(r + 1);
      }
    }
    if (pair_barrier(!ok)) {
      // a staged row never arrived: record, drain what is in flight, leave
      // (bit 2: the drain itself ran out, see pr_block)
      if (hl == 0) {
        bool drained = true;
        for (int j = max(k, 0); j < issued; ++j)
          drained = mbar_wait(bar_s + 8 * ((kbase + j) % D), ((kbase + j) / D) & 1,
                              PAIR_WAIT_NS / 4) && drained;
        if (g.status) atomicOr(g.status, drained ? 1 : 3);
      }
      return 1;
    }
    // everyone is done with pulled row r - 1: refill its slot
    if (hl == 0) issue_upto(k + D - 1);
    qs ^= 1;
  }
  if (pre_out) *pre_out = max(issued - nq, 0);
  return 0;
}

// The part of the 64 threads that own columns.
template <class S, int M>
__device__ __forceinline__ int pair_columns(const Grid& g, S* __restrict__ dst, int x0, int y0,
                                            int y1, int rs, int nq, unsigned char* smem,
                                            int kbase) {
  using G = PairGeom<S>;
  using MD = Mode<M>;
  using IO = PairIo<S>;
  constexpr bool DEV = Io<S>::dev;
  constexpr int KI = IO::scale;
  constexpr float K = KI;
  constexpr int D = G::D;
  const S* ring = reinterpret_cast<const S*>(smem);
  float* rec = reinterpret_cast<float*>(smem + G::OFF_REC);
  const Phys<float>& ph = g.pf;
  const int lc = 2 * threadIdx.x;  // first local column
  const int c = x0 + lc;           // and column
  float* qmine = reinterpret_cast<float*>(smem + G::OFF_Q) + 2 + lc;
  const unsigned bar_s = smem_u32(smem + G::OFF_BAR);
  const int nx = g.nx, ny = g.ny;
  const bool wall_l = g.bc[0] != BC_PERIODIC, wall_r = g.bc[1] != BC_PERIODIC;
  const bool wall_b = g.bc[2] != BC_PERIODIC, wall_t = g.bc[3] != BC_PERIODIC;
  const bool has1 = c < nx, has2 = c + 1 < nx;
  // walled x sides of this thread's columns: bit 0 left, 1 right at the first
  // column, 2 right at the second
  const int xwall = (has1 && c == 0 && wall_l ? 1 : 0) | (c == nx - 1 && wall_r ? 2 : 0) |
                    (c + 1 == nx - 1 && wall_r ? 4 : 0);
  const bool xl = x0 == 0, xr = nx - 1 < x0 + PAIR_COLS;  // the block holds the side's column
  const unsigned ht = sr_step(g.t);
  // The y-edge rows' values wait in local memory (a thread's own) for the end of
  // the loop.
  constexpr int NKEEP = 28;
  volatile float keep[2 * NKEEP];

  F2 pqx = F2(0.0f), pqy = F2(0.0f), qy_below = F2(0.0f);
  int qs = 0;
  int sl = kbase % D, ph_bit = (kbase / D) & 1;  // slot and phase of the next staged row
  const S* prev = ring;                          // slot of the last row
#pragma unroll 1
  for (int r = y0 - 1; r <= y1; ++r) {
    bool ok = true;
    F2 cqx = F2(0.0f), cqy = F2(0.0f);
    const S* cur = prev;
    if (r >= rs && r < rs + nq) {
      ok = mbar_wait(bar_s + 8 * sl, ph_bit, PAIR_WAIT_NS);
      cur = ring + sl * G::SLOT;
      if (++sl == D) {
        sl = 0;
        ph_bit ^= 1;
      }
      if constexpr (MD::corr) {
        F2 d[NPOP];
        Pairs<F2> q;
        Mom<F2> m;
        pair_pull<S>(cur, lc + G::LEFT, d);
        to_pairs(d, q);
        pair_moments<F2, M, DEV, KI>(ph, q, m, cqx, cqy);
        float* qp = qmine + qs * G::QROW;
        if (has2)
          *reinterpret_cast<float2*>(qp) = cqx.v;
        else if (has1)
          *qp = cqx.v.x;
      }
    }
    const int ro = r - 1;
    if (has1 && ro >= y0) {
      Pairs<F2> q;
      Mom<F2> m;
      {
        F2 d[NPOP], qx, qy;
        pair_pull<S>(prev, lc + G::LEFT, d);
        to_pairs(d, q);
        pair_moments<F2, M, DEV, KI>(ph, q, m, qx, qy);
      }
      F2 dx = F2(0.0f), dy = F2(0.0f);
      if constexpr (MD::corr) {
        const float* qp = qmine + (qs ^ 1) * G::QROW;
        float l = qp[-1], rr = qp[has2 ? 2 : 1];
        if (xwall) {  // mirror ghosts
          const F2 rho = DEV ? m.r0 + F2(1.0f) : m.r0, th = DEV ? m.th + F2(1.0f) : m.th;
          if (xwall & 1) l = mirror_q<float, KI>(g, 0, 0, rho.v.x, th.v.x, pqx.v.x);
          if (xwall & 2) rr = mirror_q<float, KI>(g, 1, 0, rho.v.x, th.v.x, pqx.v.x);
          if (xwall & 4) rr = mirror_q<float, KI>(g, 1, 0, rho.v.y, th.v.y, pqx.v.y);
        }
        dx = F2(has2 ? pqx.v.y : rr, rr) - F2(l, pqx.v.x);
        F2 up = cqy, dn = qy_below;
        if ((wall_t && ro == ny - 1) || (wall_b && ro == 0)) {
          const F2 rho = DEV ? m.r0 + F2(1.0f) : m.r0;
          const F2 om = DEV ? m.th : m.th + F2(-1.0f);  // theta - 1
          if (wall_t && ro == ny - 1)
            up = F2(2.0f * K * ph.uw[3][1]) * rho *
                     (g.bc[3] == BC_ISO ? F2(ph.thw[3] - 1.0f) : om) - pqy;
          if (wall_b && ro == 0)
            dn = F2(2.0f * K * ph.uw[2][1]) * rho *
                     (g.bc[2] == BC_ISO ? F2(ph.thw[2] - 1.0f) : om) - pqy;
        }
        dy = up - dn;
      }
      F2 v[NPOP];
      pair_collide<F2, M, DEV, KI>(ph, g.mu_law, q, m, dx, dy, v);
      // stores: one word per population
      S* p = dst + (long long)(ro + 1) * g.rp + XOFF + c;
      typename IO::W w[NPOP];
      if constexpr (Io<S>::sr) {
        unsigned ra = sr_node(c, ro, ht), rb = sr_node(c + 1, ro, ht);
#pragma unroll
        for (int a = 0; a < NPOP; a += 2) {
          // a node's word j rounds populations 2j (high half) and 2j + 1
          ra = lcg_next(ra);
          rb = lcg_next(rb);
          w[a] = IO::pack(v[a], __byte_perm(ra, rb, 0x7632));
          w[a + 1] = IO::pack(v[a + 1], __byte_perm(ra, rb, 0x5410));
        }
      } else {
#pragma unroll
        for (int a = 0; a < NPOP; ++a) w[a] = IO::pack(v[a], 0u);
      }
      if (has2) {
#pragma unroll
        for (int a = 0; a < NPOP; ++a)
          *reinterpret_cast<typename IO::W*>(p + plane(a) * g.pitch) = w[a];
      } else {
#pragma unroll
        for (int a = 0; a < NPOP; ++a) p[plane(a) * g.pitch] = IO::lo(w[a]);
      }
      if (xwall) {
        // record (absolute values): f*_A, h*_A, h*_B of the three leaving
        // populations, the moments
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          if (!(xwall & (side == 0 ? 1 : 6))) continue;
          const bool hi = side == 1 && (xwall & 4);
          float* e = rec + (((ro - y0) % G::XROWS) * 2 + side) * G::XVALS;
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const int A = side == 0 ? (i == 0 ? 3 : (i == 1 ? 6 : 7))
                                    : (i == 0 ? 1 : (i == 1 ? 5 : 8));
            const int B = opp(A);
            e[i] = (hi ? v[A].v.y : v[A].v.x) * (1.0f / K) + pref<S>(g, A);
            e[3 + i] = (hi ? v[9 + A].v.y : v[9 + A].v.x) * (1.0f / K) + pref<S>(g, 9 + A);
            e[6 + i] = (hi ? v[9 + B].v.y : v[9 + B].v.x) * (1.0f / K) + pref<S>(g, 9 + B);
          }
          e[9] = (hi ? m.r0.v.y : m.r0.v.x) + (DEV ? 1.0f : 0.0f);
          e[10] = hi ? m.ux.v.y : m.ux.v.x;
          e[11] = hi ? m.uy.v.y : m.uy.v.x;
          e[12] = (hi ? m.th.v.y : m.th.v.x) + (DEV ? 1.0f : 0.0f);
          e[13] = (hi ? m.es.v.y : m.es.v.x) + (DEV ? ph.b6 : 0.0f);
        }
      }
      if (ro == 0 || ro == ny - 1) {
#pragma unroll
        for (int up = 0; up < 2; ++up) {
          if (ro != (up ? ny - 1 : 0)) continue;
          volatile float* e = keep + up * NKEEP;
          int n = 0;
          auto put2 = [&](F2 x, float add, float mul) {
            e[n++] = x.v.x * mul + add;
            e[n++] = x.v.y * mul + add;
          };
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const int A = up ? (d == 0 ? 2 : (d == 1 ? 5 : 6)) : (d == 0 ? 4 : (d == 1 ? 8 : 7));
            const int B = opp(A);
            put2(v[A], pref<S>(g, A), 1.0f / K);
            put2(v[9 + A], pref<S>(g, 9 + A), 1.0f / K);
            put2(v[9 + B], pref<S>(g, 9 + B), 1.0f / K);
          }
          put2(m.r0, DEV ? 1.0f : 0.0f, 1.0f);
          put2(m.ux, 0.0f, 1.0f);
          put2(m.uy, 0.0f, 1.0f);
          put2(m.th, DEV ? 1.0f : 0.0f, 1.0f);
          put2(m.es, DEV ? ph.b6 : 0.0f, 1.0f);
        }
      }
    }
    if (pair_barrier(!ok)) return 1;
    if ((xl || xr) && ro >= y0 && ((ro - y0 + 1) % G::XROWS == 0 || ro == y1 - 1)) {
      const int c0 = (ro - y0) / G::XROWS * G::XROWS;
      pair_xsides<S, M>(g, dst, rec, y0 + c0, ro - y0 - c0 + 1, xl, xr);
      if (ro != y1 - 1) pair_compute_barrier();  // the records are free
    }
    qy_below = pqy;
    pqx = cqx;
    pqy = cqy;
    qs ^= 1;
    prev = cur;
  }
#pragma unroll 1
  for (int up = 0; up < 2; ++up) {
    if (!has1 || (up ? y1 != ny : y0 != 0)) continue;
    YEdge e;
    volatile float* f = keep + up * NKEEP;
    int n = 0;
    auto get2 = [&]() {
      const float x = f[n], y = f[n + 1];
      n += 2;
      return F2(x, y);
    };
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      e.f[d] = get2();
      e.h[d] = get2();
      e.hb[d] = get2();
    }
    e.rho = get2();
    e.ux = get2();
    e.uy = get2();
    e.th = get2();
    e.es = get2();
    pair_yside<S, M>(g, dst, c, up ? ny - 1 : 0, has2, up, e);
  }
  return 0;
}

// One block's share of a step: columns [x0, x0 + 128), rows [y0, y0 + rows) of
// grid g (the contract of pr_block: kbase counts the rows this block staged
// before, `pre` rows of this share are in flight already, and the copies run on
// into `next`; pre and *pre_out matter in the helper's lane 0 alone).  Returns 0,
// or 1 if a staged row never arrived.
template <class S, int M>
__device__ __forceinline__ int pair_block(const Grid& g, const CUtensorMap* map, const void* src,
                                          void* dst, int x0, int y0, int rows,
                                          unsigned char* smem, int kbase, int pre = 0,
                                          PrNext next = PrNext{nullptr, 0, 0, 0, 0},
                                          int* pre_out = nullptr) {
  const int y1 = min(y0 + rows, g.ny);
  int rs;
  const int nq = pr_span(g.ny, g.bc[2] == BC_PERIODIC, g.bc[3] == BC_PERIODIC, y0, rows, rs);
  if (threadIdx.x >= PAIR_COMPUTE)
    return pair_helper<S, M>(g, map, static_cast<const S*>(src), x0, y0, y1, rs, nq, smem, kbase,
                             pre, next, pre_out);
  return pair_columns<S, M>(g, static_cast<S*>(dst), x0, y0, y1, rs, nq, smem, kbase);
}

template <class S, int M>
__global__ void __launch_bounds__(PAIR_THREADS, PairGeom<S>::BLOCKS)
    step_pair_kernel(const __grid_constant__ Grid g, const __grid_constant__ CUtensorMap map,
                     int rows) {
  extern __shared__ __align__(1024) unsigned char smem[];
  pair_init<S>(smem);
  pdl_wait();
  pdl_release();
  const int y0 = blockIdx.y * rows;
  if (y0 >= g.ny) return;  // whole block
  pair_block<S, M>(g, &map, g.src, g.dst, blockIdx.x * PAIR_COLS, y0, rows, smem, 0);
}

}  // namespace lbm
