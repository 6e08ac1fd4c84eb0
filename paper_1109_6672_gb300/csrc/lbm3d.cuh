// Device side of the three-dimensional extension of the coupled DDF thermal
// lattice Boltzmann step (arXiv:1109.6672, BGK scheme of Sec. III.C.1
// carried to D3Q19; the paper states that its formulation extends to 3-D).
//
// Equilibria: Eq. 18a / 18b with D = 3 (R T0 = 1/3, c = 1).  Correction
// term: on D3Q19 the third-order moment of f^eq deviates from Eq. 10d by
//   D_iii = Q_i   and   D_iik = D_iki = D_kii = Q_k / 6   (i != k),
// Q = rho u (1 - theta) (the diagonal is Eq. 20; the cross entries come from
// the missing (1,1,1) velocities), so the argument that gives Eq. 28 from
// Eq. 27 asks for second moments
//   G_ii = dQ_i/dx_i + (1/6) sum_{k != i} dQ_k/dx_k,
//   G_ij = (dQ_j/dx_i + dQ_i/dx_j) / 6   (i != j),
// with the central differences of Eq. 50 along every axis.  C_a is the
// even quadratic polynomial of e_a orthogonal to the constants (the D3Q19
// counterpart of Eq. 49: only second-order moments):
//   C_a = sum_ij A_ij (e_ai e_aj - kappa d_ij), kappa = 10/19,
//   A_kk = (G_kk + (4/7) tr G) / 6,  A_ij = G_ij / 8,
// i.e. C_0 = -(5/21) tr G, C_(+-x) = A_xx - (5/21) tr G,
// C_(+-1,+-1,0) = A_xx + A_yy - (5/21) tr G +- G_xy / 4 (sign of e_x e_y).
//
// State layout (one buffer; two buffers ping-pong): element (a, x, y, z),
// a = 0..37 (f_0..f_18, h_0..h_18), x in [-1, nx], y in [-1, ny], z in
// [-1, nz] (a one-node ghost ring) at
//     ((z + 1) * (ny + 2) + (y + 1)) * 38 * pitch + plane(a) * pitch + x + 32,
// f_q and h_q in neighbouring planes (plane = 2 q, 2 q + 1),
// pitch a multiple of 32 and >= nx + 33.  As in 2-D, a buffer holds the
// post-collision value f*_a(s) at the slot s from which node s + e_a pulls
// it: the canonical pre-collision state of node x is buf_a(x - e_a).  Across
// periodic sides the pull wraps; the ghost slots hold what walls return
// (walls3d_kernel).
//
// Kernel: a block owns a tile of (x, y) and marches along z over its z range.
// For each plane it first computes the moments (and q = -Q) of the tile plus a
// one-node halo ring (wrapped periodically) into a 3-plane ring of q in shared
// memory, then collides the plane below, whose own moments the thread kept in
// registers and whose pulled populations it parked in shared memory (a
// per-thread column, two planes deep (three with asynchronous copies), so no
// barrier guards it).  Each side of the
// box is periodic or a halfway wall.
#pragma once

#include "lbm_node.cuh"

namespace lbm3 {

using lbm::Io;

constexpr int Q19 = 19;
constexpr int NP3 = 38;
constexpr int XOFF3 = 32;

// D3Q19: rest, +-x, +-y, +-z, then the face diagonals (+-1,+-1,0),
// (+-1,0,+-1), (0,+-1,+-1), each velocity followed by its opposite.
__host__ __device__ constexpr int e3x(int a) {
  return (a == 1 || a == 7 || a == 9 || a == 11 || a == 13) ? 1
         : (a == 2 || a == 8 || a == 10 || a == 12 || a == 14) ? -1 : 0;
}
__host__ __device__ constexpr int e3y(int a) {
  return (a == 3 || a == 7 || a == 10 || a == 15 || a == 17) ? 1
         : (a == 4 || a == 8 || a == 9 || a == 16 || a == 18) ? -1 : 0;
}
__host__ __device__ constexpr int e3z(int a) {
  return (a == 5 || a == 11 || a == 14 || a == 15 || a == 18) ? 1
         : (a == 6 || a == 12 || a == 13 || a == 16 || a == 17) ? -1 : 0;
}
__host__ __device__ constexpr int e3sq(int a) {
  return e3x(a) * e3x(a) + e3y(a) * e3y(a) + e3z(a) * e3z(a);
}
template <class C>
__host__ __device__ constexpr C w3(int a) {
  return a == 0 ? C(1) / C(3) : (a <= 6 ? C(1) / C(18) : C(1) / C(36));
}

// Storage plane of population a: f_q and h_q side by side, so that the two pull
// from the same places as one box.
__host__ __device__ constexpr int plane3(int a) { return 2 * (a % Q19) + a / Q19; }

enum { M3_TOTAL = 1, M3_ZFULL = 2, M3_CORR = 4, M3_FORCE = 8 };

template <class C>
struct Phys3 {
  C omega_f, omega_h;  // 2 / (2 tau + 1)
  C kz;                // omega_h - omega_f (Eq. 36)
  C b6, six_b;         // b / 6, 6 / b
  C uw[6][3];          // wall velocities of the sides x-, x+, y-, y+, z-, z+
  C thw[6];            // wall theta = T_w / T0 (isothermal walls)
  C g;                 // gravity along -z: a = (0, 0, -rho g)
};

enum { BC3_PERIODIC = 0, BC3_ISO = 1, BC3_ADIA = 2 };

struct Grid3 {
  void* src;
  void* dst;
  int nx, ny, nz, pitch;
  long long lp, zs;  // line stride (38 pitch) and plane stride ((ny + 2) lp)
  int energy_model, correction, z_full;
  int bc[6];  // sides x-, x+, y-, y+, z-, z+ (2 axis + high end): BC3_PERIODIC
              // or a halfway wall
  void* wm;   // moments of the wall nodes (wall_record3), for walls3d_kernel
  Phys3<double> pd;
  Phys3<float> pf;
};

template <class C>
__host__ __device__ __forceinline__ const Phys3<C>& phys3(const Grid3& g) {
  if constexpr (sizeof(C) == 8)
    return g.pd;
  else
    return g.pf;
}

__host__ __device__ __forceinline__ long long slot3(const Grid3& g, int a, int x, int y, int z) {
  return (long long)(z + 1) * g.zs + (long long)(y + 1) * g.lp +
         (long long)plane3(a) * g.pitch +
         (x + XOFF3);
}

__device__ __forceinline__ int wrap3(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// A population's way along axis `ax` to coordinate c, one beyond a side at most:
// across periodic sides it wraps, across walls it ends in the ghost slot.
__host__ __device__ __forceinline__ int wrap_axis3(const Grid3& g, int ax, int c, int n) {
  return g.bc[2 * ax] != BC3_PERIODIC ? c : (c < 0 ? c + n : (c >= n ? c - n : c));
}
__host__ __device__ __forceinline__ long long wrap_slot3(const Grid3& g, int a, int x, int y,
                                                         int z) {
  return slot3(g, a, wrap_axis3(g, 0, x, g.nx), wrap_axis3(g, 1, y, g.ny),
               wrap_axis3(g, 2, z, g.nz));
}

// Where a node column (x, y) pulls from: the offsets of rows y - e_y at x, and the
// columns x - e_x, relative to x.
struct Pull3 {
  long long row[3];
  int xe, xw;  // e_x = 1, e_x = -1
  __device__ __forceinline__ Pull3(const Grid3& g, int x, int y) {
#pragma unroll
    for (int e = -1; e <= 1; ++e)
      row[e + 1] = (long long)(wrap_axis3(g, 1, y - e, g.ny) + 1) * g.lp + (x + XOFF3);
    xe = wrap_axis3(g, 0, x - 1, g.nx) - x;
    xw = wrap_axis3(g, 0, x + 1, g.nx) - x;
  }
  // each(a, address) for the 38 values of the node at plane z: buf_a(x - e_a)
  template <class S, class F>
  __device__ __forceinline__ void addresses(const Grid3& g, const S* src, int z, F&& each) const {
    const S* pz[3];
#pragma unroll
    for (int e = -1; e <= 1; ++e)
      pz[e + 1] = src + (long long)(wrap_axis3(g, 2, z - e, g.nz) + 1) * g.zs;
#pragma unroll
    for (int q = 0; q < Q19; ++q) {
      const S* p = pz[e3z(q) + 1] + (long long)plane3(q) * g.pitch + row[e3y(q) + 1] +
                   (e3x(q) == 0 ? 0 : (e3x(q) > 0 ? xe : xw));
      each(q, p);
      each(Q19 + q, p + g.pitch);
    }
  }
};

// The node update over the nine pairs of opposite velocities k = 0 .. 8,
// (a, o) = (2 k + 1, 2 k + 2): with S = f_a + f_o and D = f_a - f_o everything
// splits into even and odd parts per pair (as in lbm_node.cuh for D2Q9), so the
// moments are sums over pairs, and a pair is loaded, relaxed and stored by
// itself: few values are live at a time.

// Eq. 35 and Eq. 37 (or the internal-energy form under Eq. 38): rho, u, theta,
// the specific energy es = sum h / rho and sum h; q = -Q = rho u (theta - 1).
// ld(a) gives stored population a = 0 .. 37.
template <class C>
struct Mom3 {
  C rho, ux, uy, uz, th, es, sh;
};
template <class C, int M, class Ld>
__device__ __forceinline__ void moments3(const Phys3<typename lbm::Scalar<C>::T>& k, Ld&& ld,
                                         Mom3<C>& m, C q[3]) {
  using lbm::fma_;
  C sf = ld(0), sh = ld(Q19);
  C j[3] = {C(0.0), C(0.0), C(0.0)};
#pragma unroll
  for (int a = 1; a < Q19; a += 2) {
    const C fa = ld(a), fo = ld(a + 1);
    sf = sf + (fa + fo);
    sh = sh + (ld(Q19 + a) + ld(Q19 + a + 1));
    const C d = fa - fo;
    const int e[3] = {e3x(a), e3y(a), e3z(a)};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (e[i] > 0) j[i] = a == 2 * i + 1 ? d : j[i] + d;
      if (e[i] < 0) j[i] = j[i] - d;
    }
  }
  m.rho = sf;
  m.sh = sh;
  if constexpr ((M & M3_FORCE) != 0)  // rho u = sum e f + a / 2
    j[2] = fma_(C(-0.5 * k.g), sf, j[2]);
  const C inv = lbm::rcp_(sf);
  m.ux = j[0] * inv;
  m.uy = j[1] * inv;
  m.uz = j[2] * inv;
  m.es = sh * inv;
  if constexpr ((M & M3_TOTAL) != 0)
    m.th = C(k.six_b) * fma_(C(-0.5), fma_(m.uz, m.uz, fma_(m.uy, m.uy, m.ux * m.ux)), m.es);
  else
    m.th = C(k.six_b) * m.es;
  const C om = m.th + C(-1.0);
#pragma unroll
  for (int i = 0; i < 3; ++i) q[i] = j[i] * om;
}

// Equilibria per shell (0: axis, w = 1/18; 1: diagonal, w = 1/36),
//   f^eq = A + B (e.u)^2 +- L e.u,  h^eq = HA + HB (e.u)^2 +- HL e.u:
//   f^eq: rho w [1 - 3/2 u^2 + 9/2 eu^2 +- (6 - 3 theta) eu] (axis),
//         rho w [1 - 3/2 u^2 + 9/2 eu^2 + 3/2 (theta - 1) +- (3/2 + 3/2 theta) eu],
//   h^eq: Es f^eq + w p [9 eu^2 - 3 u^2 + (0 axis | 3/2 theta diagonal) +- 3 eu].
template <class C>
struct Shells3 {
  C usq, A[2], B[2], L[2], HA[2], HB[2], HL[2];
};
template <class C, bool TOTAL>
__device__ __forceinline__ void shells3(C rho, C ux, C uy, C uz, C th, C es, Shells3<C>& e) {
  using lbm::fma_;
  using T = typename lbm::Scalar<C>::T;
  const C usq = fma_(uz, uz, fma_(uy, uy, ux * ux));
  e.usq = usq;
  const C r1 = rho * C(T(1) / T(18)), r2 = r1 * C(0.5);
  const C a0 = fma_(C(-1.5), usq, C(1.0));
  e.A[0] = r1 * a0;
  e.A[1] = r2 * fma_(C(1.5), th, a0 + C(-1.5));
  e.B[0] = C(4.5) * r1;
  e.B[1] = C(4.5) * r2;
  e.L[0] = r1 * fma_(C(-3.0), th, C(6.0));
  e.L[1] = r2 * fma_(C(1.5), th, C(1.5));
  if constexpr (TOTAL) {
    const C p1 = (rho * th) * C(T(1) / T(54)), p2 = p1 * C(0.5);  // w p
    const C hu = C(-3.0) * usq;
    e.HA[0] = fma_(es, e.A[0], p1 * hu);
    e.HA[1] = fma_(es, e.A[1], p2 * fma_(C(1.5), th, hu));
    e.HB[0] = fma_(es, e.B[0], C(9.0) * p1);
    e.HB[1] = fma_(es, e.B[1], C(9.0) * p2);
    e.HL[0] = fma_(es, e.L[0], C(3.0) * p1);
    e.HL[1] = fma_(es, e.L[1], C(3.0) * p2);
  } else {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      e.HA[s] = es * e.A[s];
      e.HB[s] = es * e.B[s];
      e.HL[s] = es * e.L[s];
    }
  }
}

// Collision (Eq. 34 with +(1 - w_f/2) C', Eq. 36 or Eq. 38; C' = C_a plus Guo's
// force along -z) of a node, pair by pair: ld(a) gives the stored populations,
// st(a, v) takes the post-collision ones.  dq[k][j]: the undivided central
// differences q_j(x + e_k) - q_j(x - e_k) of q = -Q.
// C_a / 2 in the differences D_kj = -dq[k][j] with s = D_xx + D_yy + D_zz (the
// closed form at the top): (5/144) D_kk - (41/1008) s on axis k, and
// (33/1008) s - (5/144) D_nn +- (D_ij + D_ji)/96 on the diagonals of the plane
// (i, j) with normal n.  The rest populations follow from the conserved sums.
template <class C, int M, class Ld, class St>
__device__ __forceinline__ void collide3(const Phys3<typename lbm::Scalar<C>::T>& k,
                                         const Mom3<C>& m, const C dq[3][3], Ld&& ld, St&& st) {
  using lbm::fma_;
  using T = typename lbm::Scalar<C>::T;
  constexpr bool total = (M & M3_TOTAL) != 0, corr = (M & M3_CORR) != 0,
                 force = (M & M3_FORCE) != 0;
  Shells3<C> e;
  shells3<C, total>(m.rho, m.ux, m.uy, m.uz, m.th, m.es, e);
  C s = C(0.0), dk[3], ox[3];  // ox: off-diagonal sums of the planes yz, xz, xy
  if constexpr (corr) {
    s = dq[0][0] + (dq[1][1] + dq[2][2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) dk[i] = dq[i][i] * C(T(-5) / T(144));
    ox[0] = (dq[1][2] + dq[2][1]) * C(T(-1) / T(96));
    ox[1] = (dq[0][2] + dq[2][0]) * C(T(-1) / T(96));
    ox[2] = (dq[0][1] + dq[1][0]) * C(T(-1) / T(96));
  }
  C gx = C(0.0), gy = C(0.0), gz = C(0.0), ah = C(0.0);
  if constexpr (force) {
    ah = m.rho * C(-0.5 * k.g);  // half of a_z
    gx = ah * m.ux * C(0.25);
    gy = ah * m.uy * C(0.25);
    gz = ah * m.uz;
  }
  // FP64, where operations are what counts, takes the rates into the shells,
  // w X^eq + (1 - w) X with w = 1 - (1 - w) exactly, so that what the collision
  // conserves stays; FP32 relaxes the small difference, X^eq + (1 - w)(X - X^eq), which
  // rounds less.
  constexpr bool FOLD = sizeof(C) == 8;
  const C wf1 = C(T(0.5) * (T(1) - k.omega_f)), wh1 = C(T(0.5) * (T(1) - k.omega_h));
  const C kzh = C(T(0.5) * k.kz);
  const C zc = (M & M3_ZFULL) ? C(-0.5) * e.usq : C(0.0);  // Z = e.u + zc
  const C kzz = kzh * zc;
  C cs = C(0.0);
  if constexpr (FOLD) {
    const C v = fma_(C(-2.0), wh1, C(1.0)), w = fma_(C(-2.0), wf1, C(1.0));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      e.HA[q] = v * e.HA[q];
      e.HB[q] = v * e.HB[q];
      e.HL[q] = v * e.HL[q];
      if constexpr (!total) {
        e.A[q] = w * e.A[q];
        e.B[q] = w * e.B[q];
        e.L[q] = w * e.L[q];
      }
    }
    cs = fma_(C(2.0), wf1, C(1.0));  // 2 - w, for C'/2
  }
  const C u[3] = {m.ux, m.uy, m.uz};
  C sE = C(0.0), shE = C(0.0);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int a = 2 * i + 1, o = a + 1, sh = i < 3 ? 0 : 1;
    C eu;
    if (i < 3)
      eu = u[i];
    else if (i < 5)
      eu = i == 3 ? m.ux + m.uy : m.ux - m.uy;
    else if (i < 7)
      eu = i == 5 ? m.ux + m.uz : m.ux - m.uz;
    else
      eu = i == 7 ? m.uy + m.uz : m.uy - m.uz;
    const C e2 = eu * eu;
    const C fe = fma_(e.B[sh], e2, e.A[sh]), fo = e.L[sh] * eu;
    C c = C(0.0), g = C(0.0);  // half of C', even and odd
    if constexpr (corr) {
      if (i < 3) {
        c = fma_(C(T(41) / T(1008)), s, dk[i]);
      } else {
        const int n = i < 5 ? 2 : (i < 7 ? 1 : 0);
        const C base = fma_(C(T(-33) / T(1008)), s, C(-1.0) * dk[n]);
        c = ((i - 3) & 1) ? base - ox[n] : base + ox[n];
      }
    }
    if constexpr (force) {
      const bool odd = (i - 3) & 1;
      if (i < 2)
        c = fma_(C(T(-1) / T(6)), gz, c);
      else if (i == 2)
        c = fma_(C(T(1) / T(3)), gz, c);
      else if (i < 5)
        c = fma_(C(T(-1) / T(12)), gz, c);
      else {
        c = fma_(C(T(1) / T(6)), gz, c);
        const C t = i < 7 ? gx : gy;
        c = odd ? c - t : c + t;
      }
      if (i == 2) g = ah * C(T(1) / T(6));
      if (i >= 5) g = ah * C(odd ? T(-1) / T(12) : T(1) / T(12));
    }
    const bool cf = corr || force, gf = force && (i == 2 || i >= 5);
    const C fa = ld(a), fb = ld(o), ha = ld(Q19 + a), hb = ld(Q19 + o);
    const C S = fa + fb, D = fa - fb;
    C nE, nO, fE, fO;
    if constexpr (FOLD && !total) {
      fE = fma_(wf1, S, cf ? fma_(cs, c, fe) : fe);
      fO = fma_(wf1, D, gf ? fma_(cs, g, fo) : fo);
    } else {
      nE = fma_(C(-2.0), cf ? fe - c : fe, S);  // twice n = f - f^eq + C'/2
      nO = fma_(C(-2.0), gf ? fo - g : fo, D);
      fE = fma_(wf1, nE, cf ? fe + c : fe);
      fO = fma_(wf1, nO, gf ? fo + g : fo);
    }
    st(a, fE + fO);
    st(o, fE - fO);
    const C he = fma_(e.HB[sh], e2, e.HA[sh]), ho = e.HL[sh] * eu;
    const C Sh = ha + hb, Dh = ha - hb;
    C hE = fma_(wh1, FOLD ? Sh : fma_(C(-2.0), he, Sh), he);
    C hO = fma_(wh1, FOLD ? Dh : fma_(C(-2.0), ho, Dh), ho);
    if constexpr (total) {  // Eq. 36
      const C ke = kzh * eu;
      hE = fma_(ke, nO, (M & M3_ZFULL) ? fma_(kzz, nE, hE) : hE);
      hO = fma_(ke, nE, (M & M3_ZFULL) ? fma_(kzz, nO, hO) : hO);
    }
    st(Q19 + a, hE + hO);
    st(Q19 + o, hE - hO);
    sE = i == 0 ? fE : sE + fE;
    shE = i == 0 ? hE : shE + hE;
  }
  st(0, fma_(C(-2.0), sE, m.rho));
  st(Q19, fma_(C(-2.0), shE, m.sh));
}

// f^eq (Eq. 18a, D = 3) and h^eq (Eq. 18b, D = 3, or Es f^eq) per pair of
// opposite velocities:
//   axis (e^2 = 1):     f = rho w [1 - 3/2 u^2 + 9/2 eu^2 +- (6 - 3 theta) eu]
//   diagonal (e^2 = 2): f = rho w [1 - 3/2 u^2 + 9/2 eu^2 + 3/2 (theta - 1)
//                                  +- (3/2 + 3/2 theta) eu]
//   h = Es f + w p [+-3 eu + 9 eu^2 - 3 u^2 + (0 axis | 3/2 theta diagonal)]
// The rest populations are the remainders of sum f^eq = rho and
// sum h^eq = rho Es (Eqs. 19a/19b make this an identity), Es being the
// node's own specific energy.
template <class C, bool TOTAL>
__device__ __forceinline__ void equilibria3(C rho, C ux, C uy, C uz, C th, C es, C feq[Q19],
                                            C heq[Q19]) {
  const C usq = ux * ux + uy * uy + uz * uz;
  const C A0 = C(1) - C(1.5) * usq;
  const C lin1 = C(6) - C(3) * th, lin2 = C(1.5) + C(1.5) * th;
  const C base2 = A0 + C(1.5) * (th - C(1));
  const C p = rho * th * (C(1) / C(3));
  const C hu = C(-3) * usq;
  C sf = 0, sh = 0;
#pragma unroll
  for (int a = 1; a < Q19; a += 2) {
    const C eu = C(e3x(a)) * ux + C(e3y(a)) * uy + C(e3z(a)) * uz;
    const bool axis = a <= 6;
    const C w = w3<C>(a);
    const C even = (axis ? A0 : base2) + C(4.5) * eu * eu;
    const C odd = (axis ? lin1 : lin2) * eu;
    feq[a] = rho * w * (even + odd);
    feq[a + 1] = rho * w * (even - odd);
    if constexpr (TOTAL) {
      const C he = hu + C(9) * eu * eu + (axis ? C(0) : C(1.5) * th);
      const C ho = C(3) * eu;
      heq[a] = es * feq[a] + w * p * (he + ho);
      heq[a + 1] = es * feq[a + 1] + w * p * (he - ho);
    } else {
      heq[a] = es * feq[a];
      heq[a + 1] = es * feq[a + 1];
    }
    sf += feq[a] + feq[a + 1];
    sh += heq[a] + heq[a + 1];
  }
  feq[0] = rho - sf;
  heq[0] = rho * es - sh;
}

// The populations of node (x, y, z) that leave through a wall come back
// into the node as their opposites (halfway walls at x = -1/2 and nx - 1/2,
// likewise in y and z; a population leaving through an edge of two walled
// sides takes the first of x, y, z): with b the opposite of a,
// f_b = f*_a - 2 (odd part of f^eq_a at the node's rho and theta and the
// wall velocity); h on an isothermal wall h_b = h^eq_b(ghost) +
// (h*_b - h^eq_b), the ghost one spacing outside at u_g = 2 u_w - u,
// theta_g = max(2 theta_w - theta, theta_w / 2), rho_g theta_g =
// rho (theta - 3 g n_z) (the node's pressure carried across by hydrostatic
// balance, n_z the z component of the outward normal); h on an adiabatic
// wall h_b = h*_a - 2 (odd part of h^eq_a at (rho, u_w, theta)), for total
// energy plus the wall's work on the pair u_w . (f_b e_b - f*_a e_a) =
// -(e_a . u_w)(f_b + f*_a) (no heat crosses a moving adiabatic wall; its
// work does).  Each goes to the slot from which the node pulls b:
// x - e_b = x + e_a, a ghost slot.
__host__ __device__ constexpr int e3ax(int a, int ax) {
  return ax == 0 ? e3x(a) : (ax == 1 ? e3y(a) : e3z(a));
}
// The five populations that leave through side (2 axis + high end), 5 bits each, and
// the components of all 19 velocities plus one, 2 bits each.
__host__ __device__ constexpr unsigned leaving3(int side) {
  unsigned l = 0;
  int n = 0;
  for (int a = 1; a < Q19; ++a)
    if (e3ax(a, side >> 1) == ((side & 1) ? 1 : -1)) l |= (unsigned)a << (5 * n++);
  return l;
}
__host__ __device__ constexpr unsigned long long components3(int ax) {
  unsigned long long c = 0;
  for (int a = 0; a < Q19; ++a) c |= (unsigned long long)(e3ax(a, ax) + 1) << (2 * a);
  return c;
}

// Where the step leaves the moments of wall node (x, y, z) for walls3d_kernel: a
// record per node of each side, six values `n` apart; a node on several walls has one,
// at the first axis.
__host__ __device__ __forceinline__ long long wall_record3(const Grid3& g, int x, int y, int z,
                                                           long long& n) {
  const long long nyz = (long long)g.ny * g.nz, nxz = (long long)g.nx * g.nz;
  if (g.bc[0] != BC3_PERIODIC && (x == 0 || x == g.nx - 1)) {
    n = nyz;
    return (x == 0 ? 0 : 6 * nyz) + (long long)z * g.ny + y;
  }
  if (g.bc[2] != BC3_PERIODIC && (y == 0 || y == g.ny - 1)) {
    n = nxz;
    return 12 * nyz + (y == 0 ? 0 : 6 * nxz) + (long long)z * g.nx + x;
  }
  n = (long long)g.nx * g.ny;
  return 12 * (nyz + nxz) + (z == 0 ? 0 : 6 * n) + (long long)y * g.nx + x;
}
// Values of all records.
__host__ __device__ __forceinline__ long long wall_values3(const Grid3& g) {
  return 12 * ((long long)g.ny * g.nz + (long long)g.nx * g.nz + (long long)g.nx * g.ny);
}
template <class C>
__device__ __forceinline__ void record_wall3(const Grid3& g, int x, int y, int z,
                                             const Mom3<C>& m) {
  const bool wall = (g.bc[0] != BC3_PERIODIC && (x == 0 || x == g.nx - 1)) ||
                    (g.bc[2] != BC3_PERIODIC && (y == 0 || y == g.ny - 1)) ||
                    (g.bc[4] != BC3_PERIODIC && (z == 0 || z == g.nz - 1));
  if (!wall) return;
  long long n;
  C* o = static_cast<C*>(g.wm) + wall_record3(g, x, y, z, n);
  const C v[6] = {m.rho, m.ux, m.uy, m.uz, m.th, m.es};
#pragma unroll
  for (int c = 0; c < 6; ++c) o[c * n] = v[c];
}

// The ghost slots of the walls, after the step: WALL3_NODES nodes of a side a block
// (blockIdx.y: which of the walled sides).  The nodes' moments come from the step's
// records (pulling their populations once more read 80 MB for a 101 x 87 x 65 duct,
// 18 us), the post-collision values from its stores.  Apart from the step because a
// wall node's rules are as long as its collision: in the step, every warp with one such
// node (at x walls one lane of 32) waits for them, and their code costs the other warps
// registers (256^3 periodic FP32 nodes 1.40 ms a step with it, 1.22 without).  It is
// bound by latency: 8.5 us in FP32 and 12 us in FP64 for the four walls of a
// 101 x 87 x 65 and a 75 x 61 x 53 duct.
struct WallSides {
  int side[6];
};
constexpr int WALL3_NODES = 64;
template <class S, int M>
__global__ void __launch_bounds__(WALL3_NODES)
    walls3d_kernel(const __grid_constant__ Grid3 g, const WallSides w) {
  using C = typename Io<S>::C;
  constexpr bool TOTAL = (M & M3_TOTAL) != 0;
  const Phys3<C>& k = phys3<C>(g);
  int side = w.side[0];
#pragma unroll
  for (int i = 1; i < 6; ++i)
    if (blockIdx.y == i) side = w.side[i];
  const int ax = side >> 1;
  const unsigned n0 = ax == 0 ? g.ny : g.nx, n1 = ax == 2 ? g.ny : g.nz;
  const long long i = (long long)blockIdx.x * WALL3_NODES + threadIdx.x;
  if (i >= (long long)n0 * n1) return;
  const int u = (int)(i % n0), v = (int)(i / n0);
  const int e = (side & 1) ? (ax == 0 ? g.nx : (ax == 1 ? g.ny : g.nz)) - 1 : 0;
  const int x = ax == 0 ? e : u, y = ax == 0 ? u : (ax == 1 ? e : v), z = ax == 2 ? e : v;
  unsigned list = leaving3(0);
#pragma unroll
  for (int i = 1; i < 6; ++i)
    if (side == i) list = leaving3(i);

  lbm::pdl_wait();  // the step's stores
  S* dst = static_cast<S*>(g.dst);
  const S* p = dst + slot3(g, 0, x, y, z);
  // every load before the first store: f*_a, h*_a of what leaves, h* of its opposite
  C fa[5], ha[5], hb[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const int a = (list >> (5 * j)) & 31, b = (a & 1) ? a + 1 : a - 1;
    fa[j] = Io<S>::to(__ldcg(p + (long long)(2 * a) * g.pitch));
    ha[j] = Io<S>::to(__ldcg(p + (long long)(2 * a + 1) * g.pitch));
    hb[j] = Io<S>::to(__ldcg(p + (long long)(2 * b + 1) * g.pitch));
  }
  long long n;
  const C* rec = static_cast<const C*>(g.wm) + wall_record3(g, x, y, z, n);
  const C rho = __ldcg(rec), ux = __ldcg(rec + n), uy = __ldcg(rec + 2 * n),
          uz = __ldcg(rec + 3 * n), th = __ldcg(rec + 4 * n), es = __ldcg(rec + 5 * n);
  const bool iso = g.bc[side] == BC3_ISO;
  const C uwx = k.uw[side][0], uwy = k.uw[side][1], uwz = k.uw[side][2];
  Shells3<C> eq, gh;
  shells3<C, TOTAL>(rho, ux, uy, uz, th, es, eq);
  C ugx = 0, ugy = 0, ugz = 0, E = 0;
  if (iso) {
    const C thg = fmax(C(2) * k.thw[side] - th, C(0.5) * k.thw[side]);
    ugx = C(2) * uwx - ux;
    ugy = C(2) * uwy - uy;
    ugz = C(2) * uwz - uz;
    C esg = k.b6 * thg;
    if constexpr (TOTAL) esg += C(0.5) * (ugx * ugx + ugy * ugy + ugz * ugz);
    // the node's pressure carried to the ghost by hydrostatic balance:
    // rho_g theta_g = rho (theta - 3 g n_z), n_z the outward normal's z
    // component (gravity acts along -z)
    const C rg = rho * lbm::rcp_(thg) * (ax == 2 ? th - ((side & 1) ? C(3) : C(-3)) * k.g : th);
    shells3<C, TOTAL>(rg, ugx, ugy, ugz, thg, esg, gh);
  } else {
    E = k.b6 * th;
    if constexpr (TOTAL) E += C(0.5) * (uwx * uwx + uwy * uwy + uwz * uwz);
  }
  // velocities of a shell share a coefficient; the first of a list is the one along the
  // normal, the others are diagonals
  static_assert((leaving3(0) & 31) == 2 && (leaving3(3) & 31) == 3 && (leaving3(5) & 31) == 5,
                "the normal comes first");
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const int s = j == 0 ? 0 : 1;
    const int a = (list >> (5 * j)) & 31, b = (a & 1) ? a + 1 : a - 1;
    const int ex = (int)((components3(0) >> (2 * a)) & 3) - 1;
    const int ey = (int)((components3(1) >> (2 * a)) & 3) - 1;
    const int ez = (int)((components3(2) >> (2 * a)) & 3) - 1;
    // an earlier axis's wall takes the populations leaving through an edge
    if (ax > 0 && g.bc[0] != BC3_PERIODIC && (unsigned)(x + ex) >= (unsigned)g.nx) continue;
    if (ax > 1 && g.bc[2] != BC3_PERIODIC && (unsigned)(y + ey) >= (unsigned)g.ny) continue;
    const C cx = (C)ex, cy = (C)ey, cz = (C)ez;  // e_a = -e_b
    const C euw = cx * uwx + cy * uwy + cz * uwz;
    const C fodd = eq.L[s] * euw;  // odd part of f^eq_a at (rho, u_w, theta)
    const long long o = wrap_slot3(g, 0, x + ex, y + ey, z + ez);
    const C fb = fa[j] - C(2) * fodd;
    dst[o + (long long)(2 * b) * g.pitch] = Io<S>::from(fb);
    C hin;
    if (iso) {
      const C eg = -(cx * ugx + cy * ugy + cz * ugz), en = -(cx * ux + cy * uy + cz * uz);
      const C hg = gh.HA[s] + eg * (gh.HB[s] * eg + gh.HL[s]);
      const C hq = eq.HA[s] + en * (eq.HB[s] * en + eq.HL[s]);
      hin = hg + (hb[j] - hq);
    } else {
      C hodd = E * fodd;
      if constexpr (TOTAL) hodd += (s == 0 ? w3<C>(1) : w3<C>(7)) * (rho * th) * euw;
      hin = ha[j] - C(2) * hodd;
      // total energy: the wall's work on the pair, u_w . (f_b e_b - f*_a e_a)
      if constexpr (TOTAL) hin -= euw * (fb + fa[j]);
    }
    dst[o + (long long)(2 * b + 1) * g.pitch] = Io<S>::from(hin);
  }
}

// The mirror ghost of Eq. 50 across wall side SIDE of a node with rho and
// theta: component j of 2 q_w - q0, q_w = -Q_w = rho u_w (theta_w - 1), theta_w
// the wall's on an isothermal wall and the node's own on an adiabatic one.
template <class C, int SIDE>
__device__ __forceinline__ C mirror_q3(const Grid3& g, C rho, C th, int j, C q0) {
  const Phys3<C>& k = phys3<C>(g);
  const C thw = g.bc[SIDE] == BC3_ISO ? k.thw[SIDE] : th;
  return C(2) * rho * k.uw[SIDE][j] * (thw - C(1)) - q0;
}

constexpr int TX3 = 32;

// Cells of the one-node halo ring around a TX x TY tile, and the threads of a
// block: one per tile cell, plus (SPLIT) whole warps of their own for the
// halo cells; otherwise the tile's first threads take a halo cell each too.
__host__ __device__ constexpr int nhalo3(int tx, int ty) { return 2 * (tx + 2) + 2 * ty; }
template <int TY, bool SPLIT>
__host__ __device__ constexpr int threads3() {
  return TX3 * TY + (SPLIT ? (nhalo3(TX3, TY) + 31) / 32 * 32 : 0);
}

// Dynamic shared memory of the step kernels with tiles of TX3 x TY cells: the
// parked populations of two planes (three with halo warps), [2][38][tile cells], then
// the q ring [3][3][halo tile] (a 16 x 16 tile, which FP64 storage may take instead of
// 32 x 8, has the smaller ring).
template <class S, int TY, bool SPLIT>
__host__ __device__ constexpr size_t step3d_smem() {
  using C = typename Io<S>::C;
  return sizeof(C) * ((size_t)(SPLIT ? 3 : 2) * NP3 * TX3 * TY + 9 * (TX3 + 2) * (TY + 2));
}

// Resident blocks per SM the register budget is sized for: two 256-thread
// blocks (8-row tiles), two 224-thread blocks (4-row tiles with halo warps)
// or one block otherwise; FP64 one.
template <class S, int TY, bool SPLIT>
__host__ __device__ constexpr int step3d_min_blocks() {
  return sizeof(S) == 8 ? 1 : (SPLIT ? (TY == 4 ? 2 : 1) : (TY == 8 ? 2 : 1));
}

// First node of a block's tile (2^lx x TY cells): blockIdx.x counts the tiles of
// (x, y), x first (along y alone a launch would end at 65535).
__device__ __forceinline__ void tile_origin3(int nx, int lx, int TY, int& x0, int& y0) {
  const int n = (nx + (1 << lx) - 1) >> lx, row = (int)blockIdx.x / n;
  x0 = ((int)blockIdx.x - row * n) << lx;
  y0 = row * TY;
}

// q at plane r - 1 around cell `cell` and at planes r - 2 and r, as differences
// dq[k][j] = q_j(x + e_k) - q_j(x - e_k); across a wall Eq. 50 takes the mirror
// ghost (mirror_q3).  qc: the ring's plane r - 1; q2, q1, q0: q at planes r - 2 .. r.
template <class C>
__device__ __forceinline__ void differences3(const Grid3& g, const Mom3<C>& pm, int x, int y,
                                             int z, const C* qc, int HX, int HN, const C* q2,
                                             const C* q1, const C* q0, C dq[3][3]) {
  const bool wxl = x == 0 && g.bc[0] != BC3_PERIODIC;
  const bool wxh = x == g.nx - 1 && g.bc[1] != BC3_PERIODIC;
  const bool wyl = y == 0 && g.bc[2] != BC3_PERIODIC;
  const bool wyh = y == g.ny - 1 && g.bc[3] != BC3_PERIODIC;
  const bool wb = z == 0 && g.bc[4] != BC3_PERIODIC;
  const bool wt = z == g.nz - 1 && g.bc[5] != BC3_PERIODIC;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const C* qj = qc + j * HN;
    C xp = qj[1], xm = qj[-1], yp = qj[HX], ym = qj[-HX], up = q0[j], dn = q2[j];
    if (wxl || wxh || wyl || wyh || wb || wt) {
      if (wxl) xm = mirror_q3<C, 0>(g, pm.rho, pm.th, j, q1[j]);
      if (wxh) xp = mirror_q3<C, 1>(g, pm.rho, pm.th, j, q1[j]);
      if (wyl) ym = mirror_q3<C, 2>(g, pm.rho, pm.th, j, q1[j]);
      if (wyh) yp = mirror_q3<C, 3>(g, pm.rho, pm.th, j, q1[j]);
      if (wb) dn = mirror_q3<C, 4>(g, pm.rho, pm.th, j, q1[j]);
      if (wt) up = mirror_q3<C, 5>(g, pm.rho, pm.th, j, q1[j]);
    }
    dq[0][j] = xp - xm;
    dq[1][j] = yp - ym;
    dq[2][j] = up - dn;
  }
}

// Halo cell k of the ring around a tile of TX x TY cells at (x0, y0): its place in
// the ring plane (-1: none) and its node (wrapped).
__device__ __forceinline__ int halo_cell3(const Grid3& g, int k, int TX, int TY, int x0, int y0,
                                          int& hx, int& hy) {
  const int HX = TX + 2, HY = TY + 2;
  hx = hy = 0;
  if (k < 0 || k >= nhalo3(TX, TY)) return -1;
  int cx, cy;
  if (k < HX) {
    cx = k;
    cy = 0;
  } else if (k < 2 * HX) {
    cx = k - HX;
    cy = HY - 1;
  } else {
    const int i = k - 2 * HX;  // the side columns, rows 1 .. HY - 2
    cx = (i & 1) ? HX - 1 : 0;
    cy = 1 + (i >> 1);
  }
  hx = x0 + cx - 1;
  hy = y0 + cy - 1;
  const int cell = (hx <= g.nx && hy <= g.ny) ? cy * HX + cx : -1;
  hx = wrap3(hx, g.nx);
  hy = wrap3(hy, g.ny);
  return cell;
}

// One time step of every node of the block's tile over z in [z0, z0 + zrows).
// Per plane r: pull the populations of plane r (each tile cell: parked in shared
// memory for the collision a plane later) and form q = -Q = rho u (theta - 1) of
// the tile and its halo ring into a 3-plane ring; one barrier; collide plane
// r - 1, pair by pair from the parked values, with its neighbours' q from the ring
// (along z from registers).  The slot written at plane r + 1 was last read by the
// collision of plane r - 2, which every thread finished before the barrier of
// plane r, so one barrier per plane suffices (and threads that are done with the
// collision go on pulling the next plane while the others collide).
//
// The FP64 unit bounds it (16 to 19 clocks an SM and warp
// instruction, lbm_tile.cuh): the update over pairs takes half the operations of
// one written per direction, cells beyond a ragged edge do no arithmetic, and
// the tile is 32 x 8 or 16 x 16 (lx: log2 of its columns), whichever leaves fewer
// cells idle.  75 x 61 x 53 duct: 490 us a step with a wrapped 32 x 8 tile, an update
// per direction and the walls in the step, 313 us now (297 the step, 12 the walls).
template <class S, int M, int TY>
__global__ void __launch_bounds__(threads3<TY, false>(), (step3d_min_blocks<S, TY, false>()))
    step3d_kernel(const __grid_constant__ Grid3 g, int zrows, int lx) {
  using C = typename Io<S>::C;
  constexpr int NT = TX3 * TY;
  if constexpr (sizeof(S) == 4) lx = 5;
  const int TXr = 1 << lx, TYr = NT >> lx;
  const int HX = TXr + 2, HN = HX * (TYr + 2);
  extern __shared__ __align__(16) unsigned char smem3[];
  C* park = reinterpret_cast<C*>(smem3);  // [2][NP3][NT]
  C* qs = park + 2 * NP3 * NT;            // [3][3][HN]

  const int t = threadIdx.x;
  const int tx = t & (TXr - 1), ty = t >> lx;
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  int x0, y0;
  tile_origin3(nx, lx, TYr, x0, y0);
  const int z0 = blockIdx.z * zrows;
  if (z0 >= nz) return;
  const int z1 = min(z0 + zrows, nz);
  const S* src = static_cast<const S*>(g.src);
  S* dst = static_cast<S*>(g.dst);
  const Phys3<C>& ph = phys3<C>(g);

  // this thread's interior cell and node; a cell one beyond a ragged edge is the
  // wrapped neighbour of the last node
  const int cell = (ty + 1) * HX + tx + 1;
  const int x = x0 + tx, y = y0 + ty;
  const bool interior = x <= nx && y <= ny;
  const bool mine = interior && x < nx && y < ny;
  const Pull3 pull(g, x < nx ? x : 0, y < ny ? y : 0);
  int hx, hy;
  const int hcell = halo_cell3(g, t, TXr, TYr, x0, y0, hx, hy);
  const Pull3 hpull(g, hx, hy);

  Mom3<C> pm;
  pm.rho = pm.th = C(1);
  pm.ux = pm.uy = pm.uz = pm.es = pm.sh = C(0);
  // q of this thread's node at planes r - 2, r - 1 and r
  C q2[3] = {0, 0, 0}, q1[3] = {0, 0, 0}, q[3] = {0, 0, 0};
  int s = 0;  // plane r's slot in the ring of q
  for (int r = z0 - 1; r <= z1; ++r) {
    const int zr = wrap3(r, nz);
    if (r == z1) lbm::pdl_release();
    // moments of plane r: this thread's cell (wrapped), and its halo cell
    Mom3<C> cm = pm;
    if (interior) {
      C d[NP3];
      pull.addresses(g, src, zr, [&](int a, const S* p) { d[a] = Io<S>::to(Io<S>::ld(p)); });
      C* pk = park + (r & 1) * NP3 * NT + t;
#pragma unroll
      for (int a = 0; a < NP3; ++a) pk[a * NT] = d[a];
      moments3<C, M>(ph, [&](int a) { return d[a]; }, cm, q);
#pragma unroll
      for (int j = 0; j < 3; ++j) qs[(s * 3 + j) * HN + cell] = q[j];
    }
    if (hcell >= 0) {
      C d[NP3], hq[3];
      Mom3<C> hm;
      hpull.addresses(g, src, zr, [&](int a, const S* p) { d[a] = Io<S>::to(Io<S>::ld(p)); });
      moments3<C, M>(ph, [&](int a) { return d[a]; }, hm, hq);
#pragma unroll
      for (int j = 0; j < 3; ++j) qs[(s * 3 + j) * HN + hcell] = hq[j];
    }
    __syncthreads();
    const int zc = r - 1;  // plane to collide
    if (zc >= z0 && mine) {
      C dq[3][3];
      if constexpr ((M & M3_CORR) != 0)
        differences3<C>(g, pm, x, y, zc, qs + (s == 0 ? 2 : s - 1) * 3 * HN + cell, HX, HN, q2, q1,
                        q, dq);
      C* pk = park + (zc & 1) * NP3 * NT + t;  // parked by this thread at plane zc
      S* p = dst + slot3(g, 0, x, y, zc);
      const auto st = [&](int a, C v) { p[(long long)plane3(a) * g.pitch] = Io<S>::from(v); };
      if constexpr (sizeof(S) == 8) {  // pair by pair: two registers a value
        collide3<C, M>(ph, pm, dq, [&](int a) { return pk[a * NT]; }, st);
      } else {  // all reads before the first store
        C d[NP3];
#pragma unroll
        for (int a = 0; a < NP3; ++a) d[a] = pk[a * NT];
        collide3<C, M>(ph, pm, dq, [&](int a) { return d[a]; }, st);
      }
      record_wall3<C>(g, x, y, zc, pm);
    }
    pm = cm;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      q2[j] = q1[j];
      q1[j] = q[j];
    }
    s = s == 2 ? 0 : s + 1;
  }
}

// The same step with the populations of plane r + 1 on their way from memory to
// shared memory (4-byte asynchronous copies, a thread its own) while planes r and
// r - 1 are worked on, and warps of their own for the halo cells, which hold the next
// plane's values in registers: FP32 storage.  Two blocks are resident; what bounds it
// is the latency of the eight colliding warps' arithmetic (at 128^3 44 % of the issue slots
// used, 52 % of the memory's rate), not the loads, which the copies hide.  256^3 nodes:
// 1.44 ms a step with synchronous loads and the faces in the step, 1.15 now (5.1 GB, 0.77
// at the measured copy rate); 64^3 nodes 45.5 -> 23.0 us, a walled 101 x 87 x 65 duct
// 90.8 -> 68.5.
__device__ __forceinline__ void copy_async4(void* s, const void* p) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(s)),
               "l"(p)
               : "memory");
}
template <class S, int M, int TY>
__global__ void __launch_bounds__(threads3<TY, true>(), (step3d_min_blocks<S, TY, true>()))
    step3d_async_kernel(const __grid_constant__ Grid3 g, int zrows) {
  using C = typename Io<S>::C;
  static_assert(sizeof(S) == 4 && sizeof(C) == 4, "copies of 4 bytes");
  constexpr int NT = TX3 * TY, HX = TX3 + 2, HN = HX * (TY + 2);
  extern __shared__ __align__(16) unsigned char smem3[];
  C* park = reinterpret_cast<C*>(smem3);  // [3][NP3][NT]
  C* qs = park + 3 * NP3 * NT;            // [3][3][HN]

  const int t = threadIdx.x;
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  int x0, y0;
  tile_origin3(nx, 5, TY, x0, y0);
  const int z0 = blockIdx.z * zrows;
  if (z0 >= nz) return;
  // The walls' blocks may start (they wait for the whole step): with short z ranges, whose
  // launch is what the step lasts, at once (us a step of walled ducts, released here, with
  // the last plane, and before the walls had a launch of their own: 16^3 8.5, 10.3, 10.3;
  // 32^3 10.3, 11.6, 10.3), else with the last plane, where they do not hold up the
  // loads (128^3 released at once 190, with the last plane 180).
  if (zrows <= 2) lbm::pdl_release();
  const int z1 = min(z0 + zrows, nz);
  const S* src = static_cast<const S*>(g.src);
  const Phys3<C>& ph = phys3<C>(g);

  if (t >= NT) {  // halo warps
    int hx, hy;
    const int cell = halo_cell3(g, t - NT, TX3, TY, x0, y0, hx, hy);
    const Pull3 pull(g, hx, hy);
    C d[NP3];
    const auto load = [&](int r) {
      if (cell >= 0)
        pull.addresses(g, src, wrap3(r, nz),
                       [&](int a, const S* p) { d[a] = Io<S>::to(Io<S>::ld(p)); });
    };
    load(z0 - 1);
    C* qc = qs + cell;
    int s = 0;
    for (int r = z0 - 1; r <= z1; ++r) {
      if (cell >= 0) {
        C hq[3];
        Mom3<C> hm;
        moments3<C, M>(ph, [&](int a) { return d[a]; }, hm, hq);
#pragma unroll
        for (int j = 0; j < 3; ++j) qc[(s * 3 + j) * HN] = hq[j];
      }
      if (r < z1) load(r + 1);
      __syncthreads();
      s = s == 2 ? 0 : s + 1;
    }
    return;
  }

  const int tx = t & (TX3 - 1), ty = t / TX3;
  const int cell = (ty + 1) * HX + tx + 1;
  const int x = x0 + tx, y = y0 + ty;
  // a cell one beyond a ragged edge is the wrapped neighbour of the last node
  const bool interior = x <= nx && y <= ny;
  const bool mine = interior && x < nx && y < ny;
  const Pull3 pull(g, x < nx ? x : 0, y < ny ? y : 0);
  const auto fetch = [&](int r, int s) {  // plane r into park slot s
    C* pk = park + s * NP3 * NT + t;
    if (interior)
      pull.addresses(g, src, wrap3(r, nz),
                     [&](int a, const S* p) { copy_async4(pk + a * NT, p); });
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(z0 - 1, 0);
  Mom3<C> pm;
  pm.rho = pm.th = C(1);
  pm.ux = pm.uy = pm.uz = pm.es = pm.sh = C(0);
  C q2[3] = {0, 0, 0}, q1[3] = {0, 0, 0}, q[3] = {0, 0, 0};
  int s = 0;  // plane r's slot in both rings
  for (int r = z0 - 1; r <= z1; ++r) {
    const int sn = s == 2 ? 0 : s + 1, sp = s == 0 ? 2 : s - 1;  // of planes r + 1, r - 1
    if (r < z1) {
      fetch(r + 1, sn);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (zrows > 2) lbm::pdl_release();
    }
    Mom3<C> cm = pm;
    if (interior) {
      const C* pk = park + s * NP3 * NT + t;
      moments3<C, M>(ph, [&](int a) { return pk[a * NT]; }, cm, q);
#pragma unroll
      for (int j = 0; j < 3; ++j) qs[(s * 3 + j) * HN + cell] = q[j];
    }
    __syncthreads();
    const int zc = r - 1;  // plane to collide
    if (zc >= z0 && mine) {
      C dq[3][3];
      if constexpr ((M & M3_CORR) != 0)
        differences3<C>(g, pm, x, y, zc, qs + sp * 3 * HN + cell, HX, HN, q2, q1, q, dq);
      const C* pk = park + sp * NP3 * NT + t;
      S* p = static_cast<S*>(g.dst) + slot3(g, 0, x, y, zc);
      collide3<C, M>(ph, pm, dq, [&](int a) { return pk[a * NT]; },
                     [&](int a, C v) { p[(long long)plane3(a) * g.pitch] = Io<S>::from(v); });
      record_wall3<C>(g, x, y, zc, pm);
    }
    pm = cm;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      q2[j] = q1[j];
      q1[j] = q[j];
    }
    s = sn;
  }
}

// ---- initialisation, export, reductions -----------------------------------

// Equilibrium state (FP64) of node i at the given fields, scattered into the
// slots the next pull reads: buf_a(x - e_a).
template <class S, bool TOTAL>
__global__ void init3d_kernel(const Grid3 g, S* buf, const double* __restrict__ rho,
                              const double* __restrict__ ux, const double* __restrict__ uy,
                              const double* __restrict__ uz, const double* __restrict__ T,
                              double invT0) {
  const long long n = (long long)g.nx * g.ny * g.nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % g.nx), y = (int)((i / g.nx) % g.ny), z = (int)(i / g.nx / g.ny);
    const double th = T[i] * invT0;
    const double es = TOTAL ? g.pd.b6 * th + 0.5 * (ux[i] * ux[i] + uy[i] * uy[i] + uz[i] * uz[i])
                            : g.pd.b6 * th;
    double feq[Q19], heq[Q19];
    equilibria3<double, TOTAL>(rho[i], ux[i], uy[i], uz[i], th, es, feq, heq);
    for (int a = 0; a < Q19; ++a) {
      const long long o = wrap_slot3(g, a, x - e3x(a), y - e3y(a), z - e3z(a));
      buf[o] = Io<S>::from((typename Io<S>::C)feq[a]);
      buf[o + g.pitch] = Io<S>::from((typename Io<S>::C)heq[a]);  // the next plane
    }
  }
}

// Canonical populations (FP64) of node (x, y, z).
template <class S>
__device__ __forceinline__ void pull3_fp64(const Grid3& g, const S* __restrict__ buf, int x,
                                           int y, int z, double p[NP3]) {
  for (int a = 0; a < NP3; ++a) {
    const int q = a % Q19;
    p[a] = (double)Io<S>::to(buf[wrap_slot3(g, a, x - e3x(q), y - e3y(q), z - e3z(q))]);
  }
}

// rho, u, T (FP64) and optionally the canonical populations [38][nz][ny][nx];
// *nonfinite set to 1 if a moment is NaN or infinite.
template <class S>
__global__ void export3d_kernel(const Grid3 g, const S* __restrict__ buf, double* rho, double* ux,
                                double* uy, double* uz, double* T, double T0, double* pops,
                                int* nonfinite) {
  const long long n = (long long)g.nx * g.ny * g.nz;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % g.nx), y = (int)((i / g.nx) % g.ny), z = (int)(i / g.nx / g.ny);
    double p[NP3];
    pull3_fp64<S>(g, buf, x, y, z, p);
    if (pops)
      for (int a = 0; a < NP3; ++a) pops[(long long)a * n + i] = p[a];
    if (rho) {
      double r = 0, jx = 0, jy = 0, jz = 0, sh = 0;
      for (int a = 0; a < Q19; ++a) {
        r += p[a];
        jx += e3x(a) * p[a];
        jy += e3y(a) * p[a];
        jz += e3z(a) * p[a];
        sh += p[Q19 + a];
      }
      const double vx = jx / r, vy = jy / r, vz = (jz - 0.5 * r * g.pd.g) / r;
      const double th = g.energy_model == 0
                            ? g.pd.six_b * (sh / r - 0.5 * (vx * vx + vy * vy + vz * vz))
                            : g.pd.six_b * sh / r;
      rho[i] = r;
      ux[i] = vx;
      uy[i] = vy;
      uz[i] = vz;
      T[i] = th * T0;
      if (nonfinite && !(isfinite(r) && isfinite(vx) && isfinite(vy) && isfinite(vz) &&
                         isfinite(th)))
        *nonfinite = 1;
    }
  }
}

// Per-block FP64 partial sums of rho, rho u (3) and hbar, fixed order.
constexpr int RED3 = 256;
template <class S>
__global__ void __launch_bounds__(RED3) conserved3d_kernel(const Grid3 g, const S* __restrict__ buf,
                                                           double* partial) {
  __shared__ double sm[5][RED3];
  const long long n = (long long)g.nx * g.ny * g.nz;
  double acc[5] = {0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % g.nx), y = (int)((i / g.nx) % g.ny), z = (int)(i / g.nx / g.ny);
    double p[NP3];
    pull3_fp64<S>(g, buf, x, y, z, p);
    for (int a = 0; a < Q19; ++a) {
      acc[0] += p[a];
      acc[1] += e3x(a) * p[a];
      acc[2] += e3y(a) * p[a];
      acc[3] += e3z(a) * p[a];
      acc[4] += p[Q19 + a];
    }
  }
  for (int k = 0; k < 5; ++k) sm[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int s = RED3 / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int k = 0; k < 5; ++k) sm[k][threadIdx.x] += sm[k][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) partial[5 * blockIdx.x + k] = sm[k][0];
}

template <int UNUSED = 0>
__global__ void conserved3d_final_kernel(const double* __restrict__ partial, int nb, double* out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int k = 0; k < 5; ++k) {
    double s = 0;
    for (int i = 0; i < nb; ++i) s += partial[5 * i + k];
    out[k] = s;
  }
}

}  // namespace lbm3
