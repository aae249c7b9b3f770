// linear.cuh -- the unsplit classic step of the constant-coefficient linear
// systems (scalar advection, linear acoustics) in strength form, shared by the
// 2D and 3D fused kernels.
//
// The waves of these systems are multiples of fixed eigenvectors, so the
// fluctuations and limited corrections of a face (Eq. (fluxdiff),
// Eq. (lwflux)) are scalars, and what enters a cell across its two d-faces,
// S_d = (A^+dQ - F)_{i-1/2} + (A^-dQ + F)_{i+1/2}, has a single component
// that the transverse solvers see: the pressure (acoustics) or the scalar
// itself (advection).  With tau_d = dt/dx_d S_d of that component the
// transverse and double-transverse terms (Sec. 2.1; LeVeque 1997) become
// stencils on scalars.  For acoustics, with nu_g = c dt/dx_g, Z the
// impedance, L_g f = 2 f(X) - f(X-g) - f(X+g), D_g f = f(X+g) - f(X-g):
//   A_dg = -tau_d / 2 + nu_e/12 L_e tau_d       (e the third direction, 3D)
//   p   -= nu_g/2 L_g A_dg,   u_g -= nu_g/(2 Z) D_g A_dg     for each g != d
// (the split of S_d in e has pressure -+c/2 S_d, the split of the result in g
// likewise, and E^- and E^+ differ only in the sign of that component).  For
// advection L_g/2 nu_g is the upwind difference of the velocity's sign and
// there is no second component.  The algebra is exact; only the rounding
// differs from splitting vectors face by face.
#pragma once

#include "kernels.h"
#include "riemann.cuh"

namespace claw {

// products that the compiler may not fuse into a neighbouring sum: the fused
// multiply-adds below are written out, so that every kernel and tile shape
// rounds alike
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }

// Limited strength phi(u/a) a of a wave of strength a whose upwind neighbour
// has strength u; with half = true (the MC limiter only) half of it,
// min(|a + u|/4, |a|, |u|) with the common sign, whose factor 2 the caller
// folds into its coefficient.
__device__ __forceinline__ float mc_half(float u, float a) {
  const float x = mulr(0.25f, a + u);
  const float lo = fminf(fminf(x, a), u), hi = fmaxf(fmaxf(x, a), u);
  return fmaxf(lo, 0.f) + fminf(hi, 0.f);
}
// FP64: one addition on the FP64 pipe (the scarce unit); the quarter is an
// exponent decrement (a sum below 2^-1019 counts as zero) and the minimum and
// the sign test run on the bit patterns
__device__ __forceinline__ double mc_half(double u, double a) {
  const double s = a + u;
  const int ah = __double2hiint(a), uh = __double2hiint(u), sh = __double2hiint(s) & 0x7fffffff;
  const unsigned long long am = (unsigned long long)fbits(a) & 0x7fffffffffffffffULL;
  const unsigned long long um = (unsigned long long)fbits(u) & 0x7fffffffffffffffULL;
  const unsigned long long qm =
      sh >= 0x00400000
          ? ((unsigned long long)(unsigned)(sh - 0x00200000) << 32) | (unsigned)__double2loint(s)
          : 0ULL;
  unsigned long long m = am < um ? am : um;
  m = m < qm ? m : qm;
  if ((ah ^ uh) < 0) m = 0ULL;
  return __longlong_as_double((long long)(m | ((unsigned long long)(unsigned)(ah & 0x80000000) << 32)));
}
// phi(u/a) a of the other limiters.  FP64: minima, maxima and doublings on
// the bit patterns (of minmod and superbee nothing runs on the FP64 pipe); van
// Leer's 2 u a / (u + a) by one Halley step from the hardware reciprocal where
// the sum is well inside the normal range, else by division
__device__ __forceinline__ float limit_general(int lim, float u, float a) {
  return limited_strength<float>(lim, u, a);
}
__device__ __forceinline__ double limit_general(int lim, double u, double a) {
  if (lim == CLAW_LIM_NONE) return a;
  using U = unsigned long long;
  const U m = 0x7fffffffffffffffULL, am = (U)fbits(a) & m, um = (U)fbits(u) & m;
  const U lo = am < um ? am : um, hi = am < um ? um : am;
  U g;
  if (lim == CLAW_LIM_MINMOD) {
    g = lo;
  } else if (lim == CLAW_LIM_SUPERBEE) {
    // max(min(2|u|, |a|), min(|u|, 2|a|)) = min(2 lo, hi); a value below
    // 2^-1022 doubles as a denormal (a shift)
    const U two = lo >= 0x0010000000000000ULL ? lo + 0x0010000000000000ULL : lo << 1;
    g = two < hi ? two : hi;
  } else {
    const double au = fabs(u), aa = fabs(a), s = au + aa;
    double r = 0.0;
    if (am == 0 || um == 0) {
      // no correction (and no division where the flow is at rest)
    } else if ((unsigned)(__double2hiint(s) - 0x10000000) < 0x60000000u) {
      double y;
      asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
      const double e = fma(-s, y, 1.0);
      r = (2.0 * au) * (aa * fma(y, fma(e, e, e), y));
    } else {
      r = FM<double>::div(2.0 * au * aa, s);
    }
    g = (U)fbits(r) & m;
  }
  if ((__double2hiint(a) ^ __double2hiint(u)) < 0 || am == 0 || um == 0) g = 0ULL;
  return __longlong_as_double((long long)(g | ((U)fbits(a) & ~m)));
}
template <bool FAST, typename R>
__device__ __forceinline__ R lin_limit(int lim, R u, R a) {
  if (FAST || lim == CLAW_LIM_MC) return mc_half(u, a);
  return limit_general(lim, u, a);
}

// Per-attempt constants of one direction (computed once per block)
template <typename R>
struct LinK {
  R c;    // acoustics: c dt/dx / 2; advection: max(v, 0) dt/dx
  R cm;   // advection: min(v, 0) dt/dx
  R cf;   // coefficient of the limited strength (0 for order 1)
  R t0;   // transverse: acoustics nu/2; advection max(v, 0) dt/dx
  R t1;   // transverse: acoustics nu/(2 Z); advection -min(v, 0) dt/dx
  R d1;   // double transverse, acoustics: nu/6 - 1/2
  R d2;   // double transverse, acoustics: -nu/12
  R iz;   // acoustics: 1 / Z
};

template <class RP, typename R>
struct Lin;
// systems that have the strength form
template <class RP, typename R>
struct is_linear_rp {
  static constexpr bool value = false;
};
template <typename R, int ND>
struct is_linear_rp<RpAcoustics<R, ND>, R> {
  static constexpr bool value = true;
};
template <typename R, int ND>
struct is_linear_rp<RpAdvection<R, ND>, R> {
  static constexpr bool value = true;
};

// acoustics: b_1 = Z du - dp (left-going), b_2 = Z du + dp (right-going), in
// units of 2 Z times the wave strengths.  A face keeps
//   t_p = cf b_p limited,  p = (c b_2 - t_2, t_1),  m = (t_2, c b_1 - t_1)
// and a cell between faces i, i+1 takes
//   (X, Y) = p_i + m_{i+1};  tau = X + Y,  Z omega = X - Y
// (pressure and normal-velocity components of dt/dx S).
template <typename R, int ND>
struct Lin<RpAcoustics<R, ND>, R> {
  static constexpr int M = ND + 1, NS = 2;
  static constexpr bool VEL = true;  // the normal velocity takes part
  __device__ static void consts(const MConsts<R>& C, int d, R dtdx, LinK<R>& k) {
    const R nu = C.aco_c * dtdx;
    k.c = R(0.5) * nu;
    k.cm = R(0);
    const R cf = k.c * (R(0.5) * (R(1) - nu));
    k.cf = C.order == 2 ? (C.lim == CLAW_LIM_MC ? R(2) * cf : cf) : R(0);
    k.t0 = k.c;
    k.t1 = nu * C.aco_h;
    k.d1 = nu * (R(1) / R(6)) - R(0.5);
    k.d2 = nu * (R(-1) / R(12));
    k.iz = R(2) * C.aco_h;
  }
  __device__ static R speed(const MConsts<R>& C, int) { return (R)fabs(C.aco_c); }
  // strengths of the face between states (pl, ul) and (pr, ur)
  __device__ static __forceinline__ void strength(const MConsts<R>& C, R pl, R ul, R pr, R ur,
                                                  R (&b)[NS]) {
    const R dp = pr - pl, du = ur - ul;
    b[0] = fma(C.aco_Z, du, -dp);
    b[1] = fma(C.aco_Z, du, dp);
  }
  // the upwind neighbour's strength of family s: the face below (l) or above (r)
  __device__ static __forceinline__ R upwind(const LinK<R>&, int s, R l, R r) {
    return s == 0 ? r : l;
  }
  // what the face gives the cell above it (p) and the cell below it (m), from
  // its strengths and their upwind neighbours
  template <bool FAST>
  __device__ static __forceinline__ void face(const LinK<R>& k, int lim, const R (&b)[NS],
                                              const R (&up)[NS], R (&p)[NS], R (&m)[NS]) {
    p[1] = mulr(k.cf, lin_limit<FAST>(lim, up[0], b[0]));
    m[0] = mulr(k.cf, lin_limit<FAST>(lim, up[1], b[1]));
    p[0] = fma(k.c, b[1], -m[0]);
    m[1] = fma(k.c, b[0], -p[1]);
  }
  // tau and Z omega of a cell from its lower face's p and its upper face's m
  __device__ static __forceinline__ void cell(const R (&p)[NS], const R (&m)[NS], R& tau, R& zo) {
    const R X = p[0] + m[0], Y = p[1] + m[1];
    tau = X + Y;
    zo = X - Y;
  }
  // tau without the corrections (transverse mode 1)
  __device__ static __forceinline__ R plain(const LinK<R>& k, const R (&bl)[NS],
                                            const R (&bu)[NS]) {
    return mulr(k.c, bl[1] + bu[0]);
  }
  // the normal velocity after the d-faces' updates
  __device__ static __forceinline__ R normal(const LinK<R>& k, R u, R zo) {
    return fma(-k.iz, zo, u);
  }
  // A_dg from tau_d and its neighbours in e
  __device__ static __forceinline__ R second(const LinK<R>& k, R t, R lo, R hi) {
    return fma(k.d1, t, mulr(k.d2, lo + hi));
  }
  // transverse update of (p, u_g) from the scalar a and its neighbours in g
  __device__ static __forceinline__ void apply(const LinK<R>& k, R a, R lo, R hi, R& p, R& u) {
    p = fma(-k.t0, fma(R(2), a, -(lo + hi)), p);
    u = fma(-k.t1, hi - lo, u);
  }
};

// advection: the strength is the jump b; a face keeps t = cf b limited and
//   p = max(v, 0) dt/dx b - t,  m = min(v, 0) dt/dx b + t;  tau = p_i + m_{i+1}
template <typename R, int ND>
struct Lin<RpAdvection<R, ND>, R> {
  static constexpr int M = 1, NS = 1;
  static constexpr bool VEL = false;
  __device__ static void consts(const MConsts<R>& C, int d, R dtdx, LinK<R>& k) {
    const R v = C.p[d], a = (R)fabs(v) * dtdx;
    k.c = v > R(0) ? a : R(0);
    k.cm = v < R(0) ? -a : R(0);
    const R cf = R(0.5) * a * (R(1) - a);
    k.cf = C.order == 2 ? (C.lim == CLAW_LIM_MC ? R(2) * cf : cf) : R(0);
    k.t0 = k.c;
    k.t1 = -k.cm;
    k.d1 = k.d2 = k.iz = R(0);
  }
  __device__ static R speed(const MConsts<R>& C, int d) { return (R)fabs(C.p[d]); }
  __device__ static __forceinline__ void strength(const MConsts<R>&, R pl, R, R pr, R,
                                                  R (&b)[NS]) {
    b[0] = pr - pl;
  }
  __device__ static __forceinline__ R upwind(const LinK<R>& k, int, R l, R r) {
    return k.c > R(0) ? l : r;
  }
  template <bool FAST>
  __device__ static __forceinline__ void face(const LinK<R>& k, int lim, const R (&b)[NS],
                                              const R (&up)[NS], R (&p)[NS], R (&m)[NS]) {
    const R t = mulr(k.cf, lin_limit<FAST>(lim, up[0], b[0]));
    p[0] = fma(k.c, b[0], -t);
    m[0] = fma(k.cm, b[0], t);
  }
  __device__ static __forceinline__ void cell(const R (&p)[NS], const R (&m)[NS], R& tau, R& zo) {
    tau = p[0] + m[0];
    zo = R(0);
  }
  __device__ static __forceinline__ R plain(const LinK<R>& k, const R (&bl)[NS],
                                            const R (&bu)[NS]) {
    return fma(k.c, bl[0], mulr(k.cm, bu[0]));
  }
  __device__ static __forceinline__ R normal(const LinK<R>&, R u, R) { return u; }
  __device__ static __forceinline__ R second(const LinK<R>& k, R t, R lo, R hi) {
    return fma(R(1) / R(6), fma(k.t0, t - lo, mulr(k.t1, t - hi)), mulr(R(-0.5), t));
  }
  __device__ static __forceinline__ void apply(const LinK<R>& k, R a, R lo, R hi, R& p, R&) {
    p = fma(-k.t0, a - lo, fma(-k.t1, a - hi, p));
  }
};

// non-finite test on the bit pattern (no FP64-pipe instruction)
__device__ __forceinline__ int not_finite(double x) {
  return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000;
}
__device__ __forceinline__ int not_finite(float x) {
  return (__float_as_int(x) & 0x7f800000) == 0x7f800000;
}

}  // namespace claw
