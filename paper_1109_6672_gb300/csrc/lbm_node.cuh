// The node update written over pairs of opposite velocities.
//
// With S_k = f_a + f_o and D_k = f_a - f_o for the four pairs (a, o) =
// (1, 3), (2, 4), (5, 7), (6, 8), the equilibria (Eq. 18a, 18b, the Eq. 38
// form), the correction (Eq. 49), the Guo force and both relaxations split
// into an even part E and an odd part O that never mix until the end,
// f*_a = E + O, f*_o = E - O; only quantities of a pair are evaluated, and the
// rest populations follow from the conserved sums (sum f* = rho,
// sum h* = sum h).  Written per direction the same update took about 290 FP64
// operations a node (counted from the FP64 pipe, halo columns included); here
// it is about 145 for the internal-energy model with gravity and correction
// and 175 for total energy.
//
// C is double, float, or F2 (two nodes at once in packed FP32 instructions).
#pragma once

#include <atomic>

#include "lbm_step_tma.cuh"

namespace lbm {

// Programmatic dependent launch: wait for the previous launch of the stream
// (all of it, its writes visible), let the next one's blocks start.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch, with pdl as a programmatic dependent of the launch before it in the
// stream.  A refused launch leaves no pending error behind for the next call.
template <class... P, class... A>
cudaError_t launch_ex(void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                      cudaStream_t stream, bool pdl, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// Allows a kernel `bytes` of dynamic shared memory.  The attribute belongs to a
// device: `done` (one per kernel) has a bit for each that has it.
inline cudaError_t allow_smem(const void* kernel, int bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0;  // (beyond: every time)
  if (e == cudaSuccess && (done.load(std::memory_order_acquire) & bit)) return e;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    done.fetch_or(bit, std::memory_order_release);
  else
    cudaGetLastError();
  return e;
}

// Two FP32 values, one per node: add, mul and fma are single packed
// instructions (add/mul/fma.rn.f32x2), which issue at half the instructions
// per node of scalar FP32 (the packed fma reached the same 128 fma per SM and
// clock as the scalar one in half the issue slots).
struct F2 {
  float2 v;
  __device__ __forceinline__ F2() {}
  __device__ __forceinline__ F2(float x) : v(make_float2(x, x)) {}
  __device__ __forceinline__ F2(double x) : F2((float)x) {}
  __device__ __forceinline__ F2(float x, float y) : v(make_float2(x, y)) {}
};
__device__ __forceinline__ F2 mk2(float2 v) {
  F2 r;
  r.v = v;
  return r;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return mk2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return mk2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 fma_(F2 a, F2 b, F2 c) { return mk2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  return mk2(__ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v));  // exact product: a - b rounded once
}
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

template <class C>
struct Scalar {
  using T = C;
};
template <>
struct Scalar<F2> {
  using T = float;
};

// Reciprocal: the hardware approximation x0 and one step of a Householder
// iteration on 1/v (residual e = 1 - v x0): x0 (1 + e) squares the relative
// error, x0 (1 + e + e^2) cubes it.  FP32: 2^-23 -> correctly rounded but for
// rare ties; FP64: 2^-20 or better -> below 2^-53, four FP64 operations where
// the compiler's division takes about ten.
__device__ __forceinline__ double rcp_(double v) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(v));
  const double e = fma(-v, x, 1.0);
  return fma(x, fma(e, e, e), x);
}
__device__ __forceinline__ float rcp_approx(float v) {
  float x;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(v));
  return x;
}
__device__ __forceinline__ float rcp_(float v) {
  const float x = rcp_approx(v);
  return fmaf(x, fmaf(v, -x, 1.0f), x);
}
__device__ __forceinline__ F2 rcp_(F2 v) {
  const F2 x(rcp_approx(v.v.x), rcp_approx(v.v.y));
  const F2 e = fma_(v, x * F2(-1.0f), F2(1.0f));
  return fma_(x, e, x);
}
// Square root of theta: the hardware reciprocal square root y0 corrected by
// the cubic Householder step on 1/sqrt(v) (e = 1 - v y0^2: y0 (1 + e/2 +
// 3 e^2/8)), times v.
__device__ __forceinline__ double sqrt_(double v) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  const double s = v * y;
  const double e = fma(-s, y, 1.0);
  return fma(s, e * fma(e, 0.375, 0.5), s);
}
__device__ __forceinline__ float sqrt_(float v) { return sqrtf(v); }
__device__ __forceinline__ F2 sqrt_(F2 v) { return F2(sqrtf(v.v.x), sqrtf(v.v.y)); }
__device__ __forceinline__ double pow_(double v, double n) { return pow(v, n); }
__device__ __forceinline__ float pow_(float v, float n) { return powf(v, n); }
__device__ __forceinline__ F2 pow_(F2 v, F2 n) {
  return F2(powf(v.v.x, n.v.x), powf(v.v.y, n.v.y));
}
// min(v, a number whose square is far from overflow); NaN stays NaN.  FP64 compares the
// exponents (the FP64 unit's time is what its steps lack: with v > 1e100 a 198^2
// Sutherland cavity took 25.30 us a step instead of 25.21): 2^332 up to infinity.
__device__ __forceinline__ double cap_(double v) {
  const unsigned top = (1023u + 332u) << 20;
  const unsigned hi = (unsigned)__double2hiint(v);
  return hi - top <= 0x7FF00000u - top ? __hiloint2double((int)top, 0) : v;
}
__device__ __forceinline__ float cap_(float v) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "f"(1e15f));
  return r;
}
__device__ __forceinline__ F2 cap_(F2 v) { return F2(cap_(v.v.x), cap_(v.v.y)); }

// A node's populations as pairs: rest, sums, differences, of f and of h.
template <class C>
struct Pairs {
  C f0, h0, S[4], D[4], Sh[4], Dh[4];
};
template <class C>
__device__ __forceinline__ void to_pairs(const C d[NPOP], Pairs<C>& q) {
  constexpr int A[4] = {1, 2, 5, 6};
  q.f0 = d[0];
  q.h0 = d[9];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int a = A[k], o = opp(A[k]);
    q.S[k] = d[a] + d[o];
    q.D[k] = d[a] - d[o];
    q.Sh[k] = d[9 + a] + d[9 + o];
    q.Dh[k] = d[9 + a] - d[9 + o];
  }
}

// Moments (Eq. 35 with the force shift, Eq. 37 or the Eq. 38 form) and
// q = -Q = rho u (theta - 1).  (r0, th, es) are rho, theta, Es for absolute
// storage and rho - 1, theta - 1, Es - b/6 for deviation storage, there formed
// from the sums of the stored deviations so that nothing is rounded at the scale
// of the populations (the references' own sums are taken in FP64 on the host:
// dref).  The balance of internal energy, rho (Es - b/6) - rho u^2 / 2, is then
// one subtraction of two FP32 numbers, and FP32's correctly rounded subtraction
// gives the value an FP64 subtraction rounded back to FP32 would: the exact
// difference is an FP64 number when the exponents differ by at most 28, and
// otherwise lies within 2^-28 of the larger operand, far from any FP32 rounding
// tie.  The populations may be held K times too large (K a power of two;
// deviation storage): sh, the sum of h, and q are then K times too large as
// well, the rest is not.
template <class C>
struct Mom {
  C r0, ux, uy, th, es, sh;
};
template <class C, int M, bool DEV, int K = 1>
__device__ __forceinline__ void pair_moments(const Phys<typename Scalar<C>::T>& k,
                                             const Pairs<C>& q, Mom<C>& m, C& qx, C& qy) {
  using MD = Mode<M>;
  const C sf = q.f0 + ((q.S[0] + q.S[1]) + (q.S[2] + q.S[3]));
  m.sh = q.h0 + ((q.Sh[0] + q.Sh[1]) + (q.Sh[2] + q.Sh[3]));
  const C jx = q.D[0] + (q.D[2] - q.D[3]);
  C jy = q.D[1] + (q.D[2] + q.D[3]);
  m.r0 = K == 1 ? sf : sf * C(1.0 / K);
  const C rho = DEV ? m.r0 + C(1.0) : m.r0;
  if constexpr (MD::force) jy = fma_(C(-0.5 * K * k.g), rho, jy);
  const C inv = rcp_(rho);
  const C ivk = K == 1 ? inv : inv * C(1.0 / K);
  m.ux = jx * ivk;
  m.uy = jy * ivk;
  if constexpr (DEV) {
    // rho (Es - b/6)
    const C e = fma_(C(-k.b6), m.r0,
                     K == 1 ? m.sh + C(k.dref) : fma_(m.sh, C(1.0 / K), C(k.dref)));
    m.es = e * inv;
    if constexpr (MD::total) {
      const C kin = fma_(jy, m.uy, jx * m.ux);
      m.th = C(k.six_b) * (fma_(C(-0.5 / K), kin, e) * inv);
    } else {
      m.th = C(k.six_b) * m.es;
    }
    qx = jx * m.th;
    qy = jy * m.th;
  } else {
    m.es = m.sh * inv;
    if constexpr (MD::total)
      m.th = C(k.six_b) * fma_(C(-0.5), fma_(m.uy, m.uy, m.ux * m.ux), m.es);
    else
      m.th = C(k.six_b) * m.es;
    const C om = m.th + C(-1.0);
    qx = jx * om;
    qy = jy * om;
  }
}

// q = -Q of the mirror ghost across a wall side: 2 rho u_w (theta_w - 1) - q (K
// times too large, as q).
template <class C, int K = 1>
__device__ __forceinline__ C mirror_q(const Grid& g, int side, int comp, C rho, C th, C q) {
  const Phys<C>& k = phys<C>(g);
  const C thw = g.bc[side] == BC_ISO ? k.thw[side] : th;
  return C(2 * K) * rho * k.uw[side][comp] * (thw - C(1)) - q;
}

// Relaxation rates of a node (node_rates): the constants, or with a viscosity
// law mu(theta)/mu0 = L the rates w = 2 / (2 tau + 1), tau_f = tau_f0 L /
// (rho theta), tau_h = tau_f r, over one common reciprocal.  Sutherland:
// L = theta^(3/2) (1 + s) / (theta + s), so with X = rho (theta + s) and
// Y = 2 tau_f0 (1 + s) sqrt(theta), w_f = 2 X / (X + Y), w_h = 2 X / (X + r Y);
// power law: X = rho theta, Y = 2 tau_f0 theta^n.  Y is capped where w is zero to
// rounding, so that neither an overflowing theta^n nor the product of the two
// denominators turns it into NaN.  kz: w_h - w_f, or for MRT
// (1 - w_h/2)(1/r - 1) w_f (Eq. 47 with tau_f + 1/2 = 1/w_f).
template <class C, int M>
__device__ __forceinline__ void pair_rates(const Phys<typename Scalar<C>::T>& k, int mu_law, C rho,
                                           C th, C& wf, C& wh, C& kz) {
  using MD = Mode<M>;
  if constexpr (!MD::varmu) {
    wf = C(k.omega_f);
    wh = C(k.omega_h);
    kz = C(k.kz);
  } else {
    C X, Y;
    if (mu_law == MU_POWER) {
      X = rho * th;
      Y = C(2 * k.tau_f0) * pow_(th, C(k.mu_n));
    } else {
      X = rho * (th + C(k.mu_s));
      Y = C(2 * k.tau_f0 * (1 + k.mu_s)) * sqrt_(th);
    }
    Y = cap_(Y);
    const C a = X + Y, b = fma_(C(k.tau_ratio), Y, X);
    const C t = (X + X) * rcp_(a * b);
    wf = t * b;
    wh = t * a;
    if constexpr (MD::mrt)
      kz = fma_(C(-0.5), wh, C(1.0)) * wf * C(1 / k.tau_ratio - 1);
    else
      kz = wh - wf;
  }
}

// Equilibria per pair, f^eq_a = fe + fo, f^eq_o = fe - fo (Eq. 18a), likewise
// h^eq (Eq. 18b or the Eq. 38 form), as deviations from the rest equilibria for
// deviation storage.  Per shell s (0: the axis
// pairs, 1: the diagonals) they are linear in e.u and its square,
//   fe = A + B (e.u)^2, fo = L e.u, he = HA + HB (e.u)^2, ho = HL e.u:
//   f^eq = w rho [base + 9/2 eu^2 +- lin eu],
//   h^eq = Es f^eq + w p [9 eu^2 - 3 u^2 + theta (3 e^2 - 2)/2 +- 3 eu],
// all K times too large.
template <class C>
struct Shells {
  C eu[4], usq;
  C A[2], B[2], L[2], HA[2], HB[2], HL[2];
};
template <class C, bool TOTAL, bool DEV, int K = 1>
__device__ __forceinline__ void pair_shells(const Phys<typename Scalar<C>::T>& k, C rho,
                                            const Mom<C>& m, Shells<C>& q) {
  using T = typename Scalar<C>::T;
  q.eu[0] = m.ux;
  q.eu[1] = m.uy;
  q.eu[2] = m.ux + m.uy;
  q.eu[3] = m.uy - m.ux;
  const C usq = fma_(m.uy, m.uy, m.ux * m.ux);
  q.usq = usq;
  const C r1 = rho * C(T(K) / T(9)), r2 = rho * C(T(K) / T(36));
  C lin1, lin2;
  if constexpr (DEV) {
    const C hu = C(-1.5) * usq;
    q.A[0] = fma_(r1, fma_(C(0.5), m.th, hu), m.r0 * C(T(K) / T(9)));
    q.A[1] = fma_(r2, fma_(C(2.0), m.th, hu), m.r0 * C(T(K) / T(36)));
    lin1 = fma_(C(-1.5), m.th, C(3.0));
    lin2 = fma_(C(3.0), m.th, C(3.0));
  } else {
    const C a0 = fma_(C(-1.5), usq, C(0.5));  // 1 - 3/2 u^2 + (theta - 1)/2 = a0 + theta/2
    q.A[0] = r1 * fma_(C(0.5), m.th, a0);
    q.A[1] = r2 * fma_(C(2.0), m.th, a0 + C(-1.5));
    lin1 = fma_(C(-1.5), m.th, C(4.5));
    lin2 = C(3.0) * m.th;
  }
  q.B[0] = C(4.5) * r1;
  q.B[1] = C(4.5) * r2;
  q.L[0] = r1 * lin1;
  q.L[1] = r2 * lin2;
  const C Es = DEV ? m.es + C(k.b6) : m.es;
  if constexpr (TOTAL) {
    const C th = DEV ? m.th + C(1.0) : m.th;
    const C p1 = (rho * th) * C(T(K) / T(27)), p2 = p1 * C(0.25);  // w p
    const C hu = C(-3.0) * usq;
    C PA1, PA2;
    if constexpr (DEV) {
      // w (Es - b/6) + w p (-3 u^2) + w (p theta - 1/3)(3 e^2 - 2)/2
      const C pt = fma_(rho * m.th, m.th + C(2.0), m.r0) * C(T(K) / T(27));
      PA1 = fma_(p1, hu, fma_(C(0.5), pt, m.es * C(T(K) / T(9))));
      PA2 = fma_(p2, hu, fma_(C(0.5), pt, m.es * C(T(K) / T(36))));
    } else {
      PA1 = p1 * fma_(C(0.5), th, hu);
      PA2 = p2 * fma_(C(2.0), th, hu);
    }
    q.HA[0] = fma_(Es, q.A[0], PA1);
    q.HA[1] = fma_(Es, q.A[1], PA2);
    q.HB[0] = fma_(Es, q.B[0], C(9.0) * p1);
    q.HB[1] = fma_(Es, q.B[1], C(9.0) * p2);
    q.HL[0] = fma_(Es, q.L[0], C(3.0) * p1);
    q.HL[1] = fma_(Es, q.L[1], C(3.0) * p2);
  } else {
    q.HA[0] = DEV ? fma_(Es, q.A[0], m.es * C(T(K) / T(9))) : Es * q.A[0];
    q.HA[1] = DEV ? fma_(Es, q.A[1], m.es * C(T(K) / T(36))) : Es * q.A[1];
    q.HB[0] = Es * q.B[0];
    q.HB[1] = Es * q.B[1];
    q.HL[0] = Es * q.L[0];
    q.HL[1] = Es * q.L[1];
  }
}

// Collision (Eq. 34 with +(1 - w_f/2) C', Eq. 36 or Eq. 38; MRT: Eq. 44) of a
// node from its pairs, its moments and the undivided differences of q = -Q,
// dx = q_x(x+1) - q_x(x-1), dy = q_y(y+1) - q_y(y-1).  v: f*, h* (deviations
// for deviation storage).
//
// C' = C_a (Eq. 49) + F_a.  With a = -dx / 24 and b = -dy / 24, C_a / 2 is
// a - 2 b on the pair (1, 3), b - 2 a on (2, 4) and a + b on the diagonals
// (the rest population follows from the conserved sum).
// HEQ: at a wall node, v[19..26] take h^eq of the moving directions for the wall rules.
// n = (f - f^eq) + C'/2 has no mass and no momentum; in it
//   f* = f^eq + C'/2 + (1 - w_f) n          (BGK),
//   f* = f^eq + C'/2 + M^-1 (1 - S) M n     (MRT),
// and Eq. 36's coupling is kz Z n.
template <class C, int M, bool DEV, int K = 1, bool HEQ = false>
__device__ __forceinline__ void pair_collide(const Phys<typename Scalar<C>::T>& k, int mu_law,
                                             const Pairs<C>& q, const Mom<C>& m, C dx, C dy, C* v,
                                             bool wall = false) {
  using MD = Mode<M>;
  using T = typename Scalar<C>::T;
  constexpr int A[4] = {1, 2, 5, 6};
  const C rho = DEV ? m.r0 + C(1.0) : m.r0;
  C wf, wh, kz;
  pair_rates<C, M>(k, mu_law, rho, DEV ? m.th + C(1.0) : m.th, wf, wh, kz);
  Shells<C> e;
  pair_shells<C, MD::total, DEV, K>(k, rho, m, e);
  // half of C' = C_a + F_a: even parts c[], odd parts of F_a g1 (axis y), g2
  // (diagonals); F_a = w_a [3 e.a + 9 (e.u)(e.a) - 3 u.a], a = (0, ay)
  C c[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] = C(0.0);
  if constexpr (MD::corr) {
    const C a = dx * C(T(-1) / T(24)), b = dy * C(T(-1) / T(24));
    c[0] = fma_(C(-2.0), b, a);
    c[1] = fma_(C(-2.0), a, b);
    c[2] = a + b;
    c[3] = c[2];
  }
  C g1 = C(0.0), g2 = C(0.0);
  if constexpr (MD::force) {
    const C ay = rho * C(-0.5 * K * k.g);  // half of a_y
    const C gx = ay * m.ux, gy = ay * m.uy;
    c[0] = fma_(C(T(-1) / T(3)), gy, c[0]);
    c[1] = fma_(C(T(2) / T(3)), gy, c[1]);
    c[2] = fma_(C(0.25), gx, fma_(C(T(1) / T(6)), gy, c[2]));
    c[3] = fma_(C(-0.25), gx, fma_(C(T(1) / T(6)), gy, c[3]));
    g1 = ay * C(T(1) / T(3));
    g2 = ay * C(T(1) / T(12));
  }
  // pair by pair, so that few values are live at a time: twice n (even and odd
  // parts), h relaxed with Eq. 36's coupling, and (BGK) f relaxed
  const C zc = MD::zfull ? C(-0.5) * e.usq : C(0.0);  // Z = e.u + zc
  const C wh1 = fma_(C(-0.5), wh, C(0.5));
  const C wf1 = fma_(C(-0.5), wf, C(0.5));
  const C kzh = C(0.5) * kz;
  C nE[4], nO[4], bE[4], bO[4];
  C sE = C(0.0), shE = C(0.0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = A[i], o = opp(A[i]), s = i >> 1;
    const C e2 = e.eu[i] * e.eu[i];
    const C fe = fma_(e.B[s], e2, e.A[s]), fo = e.L[s] * e.eu[i];
    const C g = i == 1 ? g1 : g2;
    const bool cf = MD::corr || MD::force, gf = MD::force && i > 0;
    nE[i] = fma_(C(-2.0), cf ? fe - c[i] : fe, q.S[i]);
    nO[i] = fma_(C(-2.0), gf ? fo - g : fo, q.D[i]);
    bE[i] = cf ? fe + c[i] : fe;
    bO[i] = gf ? fo + g : fo;
    const C he = fma_(e.HB[s], e2, e.HA[s]), ho = e.HL[s] * e.eu[i];
    if constexpr (HEQ) {
      if (wall) {
        v[18 + a] = he + ho;
        v[18 + o] = he - ho;
      }
    }
    // h* = h^eq + (1 - w_h)(h - h^eq)
    C hE = fma_(wh1, fma_(C(-2.0), he, q.Sh[i]), he);
    C hO = fma_(wh1, fma_(C(-2.0), ho, q.Dh[i]), ho);
    if constexpr (MD::total) {
      if constexpr (MD::zfull) {
        hE = fma_(kzh, fma_(e.eu[i], nO[i], zc * nE[i]), hE);
        hO = fma_(kzh, fma_(e.eu[i], nE[i], zc * nO[i]), hO);
      } else {
        hE = fma_(kzh, e.eu[i] * nO[i], hE);
        hO = fma_(kzh, e.eu[i] * nE[i], hO);
      }
    }
    v[9 + a] = hE + hO;
    v[9 + o] = hE - hO;
    shE = i == 0 ? hE : shE + hE;
    if constexpr (!MD::mrt) {
      const C fE = fma_(wf1, nE[i], bE[i]), fO = fma_(wf1, nO[i], bO[i]);
      v[a] = fE + fO;
      v[o] = fE - fO;
      sE = i == 0 ? fE : sE + fE;
    }
  }
  if constexpr (MD::mrt) {
    // the even moments e, eps, pxx, pxy and the odd ones q_x, q_y of n (rows
    // of M; n_0 from the vanishing mass), relaxed, and M^-1 of them
    const C se = k.se > T(0) ? C(k.se) : wf, seps = k.seps > T(0) ? C(k.seps) : wf;
    const C sq = k.sq > T(0) ? C(k.sq) : wf;
    const C one = C(1.0);
    const C sa = nE[0] + nE[1], sd = nE[2] + nE[3];
    const C re = (one - se) * fma_(C(2.0), sd, sa);           // e / 3
    const C rp = (one - seps) * fma_(C(2.0), sa, sd);         // -eps / 3
    const C rx = (one - sq) * fma_(C(-2.0), nO[0], nO[2] - nO[3]);  // q_x
    const C ry = (one - sq) * fma_(C(-2.0), nO[1], nO[2] + nO[3]);  // q_y
    const C w1 = C(0.5) * wf1;
    const C pp = w1 * (nE[0] - nE[1]), pq = w1 * (nE[2] - nE[3]);  // pxx / 4, pxy / 4
    const C ax = fma_(C(T(1) / T(6)), rp, re * C(T(-1) / T(12)));
    const C dg = fma_(C(T(-1) / T(12)), rp, re * C(T(1) / T(6)));
    const C x2 = rx * C(T(1) / T(12)), y2 = ry * C(T(1) / T(12));
    const C fE[4] = {bE[0] + (ax + pp), bE[1] + (ax - pp), bE[2] + (dg + pq), bE[3] + (dg - pq)};
    const C fO[4] = {fma_(C(-2.0), x2, bO[0]), fma_(C(-2.0), y2, bO[1]), bO[2] + (x2 + y2),
                     bO[3] + (y2 - x2)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[A[i]] = fE[i] + fO[i];
      v[opp(A[i])] = fE[i] - fO[i];
    }
    sE = (fE[0] + fE[1]) + (fE[2] + fE[3]);
  }
  v[0] = fma_(C(-2.0), sE, K == 1 ? m.r0 : m.r0 * C((double)K));
  v[9] = fma_(C(-2.0), shE, m.sh);
}

}  // namespace lbm
