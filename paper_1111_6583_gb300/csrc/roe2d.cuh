// roe2d.cuh -- the 2D classic step of the systems with Roe solvers (shallow
// water) in strength form, one launch per attempt (two for a dimensionally
// split step).
//
// The waves of a face are W^p = al_p r_p with the Roe eigenvectors r_p of its
// geometry g (velocities, sound speed).  Keeping al and g in place of the wave
// vectors,
//   theta_p = (al_up r_up . r) / (al r . r),
//   A^-dQ + F = sum_p k_p r_p, k_p = s^-_p al_p + t_p  (A^+dQ - F: s^+ al - t),
// with t_p = 1/2 |s_p| (1 - dt/dx |s_p|) phi al_p, and the transverse split of
// such a sum follows from its strengths: in the frame of the other direction
// its acoustic strengths are (k_0 + k_2)/2 -+ k_1/(2c) and its shear strength
// c (k_2 - k_0).  The same sums as with wave vectors in fewer operations
// (about 125 per face against some 200).  What a cell receives from its two
// faces in a direction is added before it is moved on: with B^- and B^+ the
// splits of a row's x fluctuations, the y-face above row R gets
// H = B^+(R) + B^-(R+1), and the row dt^2/(2 dx dy) (H(R+1/2) - H(R-1/2)).
//
// Layout as in linear2d.cuh: a warp owns a strip of columns (one per lane in
// FP64; two in FP32, whose arithmetic runs on packed pairs) and walks a chunk
// of rows; x neighbours by shuffles, y neighbours in registers, no barrier in
// the walk.  With row r loaded it limits y-face r - 1 and finishes row r - 2.
//
// What bounds it: FP64 the FP64 pipe (87 % busy; 280 instructions per column
// and row against 318, the rest is the halo of 28 owned columns in 32);
// FP32 latency and issue at 12 warps per SM (registers held to 168: 16-warp
// and 14-warp caps spill and measured 368 us at 4096^2 against 340, no cap, 10
// warps, 392).  Dam break FP32 4096^2 664 -> 342 us/step, 1024^2 57 -> 45 us,
// FP64 1024^2 861 -> 754 us, 64 x 59 111 -> 72 us against the shared-memory
// row walk of classic2d_kernel.
#pragma once

#include "linear2d.cuh"
#include "vec.cuh"

namespace claw {

// 1/a for a >= 1 or a sum of square roots (never near the range's ends).
// FP64: one Halley step from the hardware seed (20 bits): error about one
// rounding in three FP64 instructions; FP32: the hardware approximation
__device__ __forceinline__ double rcp_safe(double a) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-a, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float rcp_safe(float a) { return rcp_approx(a); }
template <class V>
__device__ __forceinline__ V vrcp_safe(V a) {
  using S = typename VecOf<V>::S;
  return vmap([](S x) { return rcp_safe(x); }, a);
}

// larger of two speeds (a NaN speed makes the results NaN too, which are
// reported; FP32 drops it here, FP64 compares bit patterns)
__device__ __forceinline__ float max_speed(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double max_speed(double a, double b) { return max_nonneg(a, b); }
// b where s > 0, else a, by value
template <class V>
__device__ __forceinline__ V vpick(V s, V b, V a) {
  using S = typename VecOf<V>::S;
  return vmap([](S x, S y, S z) { return gt0(x) ? y : z; }, s, b, a);
}
// a where s < 0, else b
template <class V>
__device__ __forceinline__ V vneg_pick(V s, V a, V b) {
  using S = typename VecOf<V>::S;
  return vmap([](S x, S y, S z) { return lt0(x) ? y : z; }, s, a, b);
}
template <bool FAST, class V>
__device__ __forceinline__ V vlim(int lim, V u, V a) {
  using R = typename VecOf<V>::S;
  return vmap([lim](R x, R y) { return lin_limit<FAST>(lim, x, y); }, u, a);
}

template <class V, class RP>
struct RoeSys;

// ---------------------------------------------------------------------------
// shallow water: q = (h, hu, hv); p = (sqrt h, u sqrt h, v sqrt h).  The
// strengths of the two gravity waves are kept doubled (A_0, A_2 = 2 al), that
// of the shear wave as it is; the sums k are doubled, and transverse parts
// come four times (their factors are folded into the caller's dt/dx).
// ---------------------------------------------------------------------------
template <class V, typename R>
struct RoeSys<V, RpSW<R, 2>> {
  using RP = RpSW<R, 2>;
  static constexpr int M = 3, MW = 3, NP = 3, NG = 6, NX = 3;
  // un - c, un + c, ut, un, c, 1/c; the limiter's view of a neighbour: the
  // first NX (of the face above the first, of the face below the last wave)
  enum { S0, S2, UT, UN, CS, RC };
  // values of the limiter's view that only the face above / below supplies
  // when the first wave moves down and the last one up
  __device__ static constexpr bool above_only(int k) { return k == S0; }
  __device__ static constexpr bool below_only(int k) { return k == S2; }
  __device__ static __forceinline__ void prep(const MConsts<R>&, const V (&q)[M], V (&p)[NP]) {
    const V il = vrsq(q[0]);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = vmul(q[k], il);
  }
  // Split of a face's waves by direction, with the entropy fix (the tests and
  // formulas of RpSW::solve_pc): zm = doubled strengths of A^-dQ
  __device__ static void split(const MConsts<R>& C, R hl, R hul, R hr, R hur, const R (&A)[3], R un,
                               R c, R (&zm)[3]) {
    const R s[3] = {un - c, un, un + c};
    const R z[3] = {s[0] * A[0], R(2) * un * A[1], s[2] * A[2]};
#pragma unroll
    for (int p = 0; p < 3; ++p) zm[p] = lt0(s[p]) ? z[p] : R(0);
    if (!C.entropy_fix) return;
    const R a0 = R(0.5) * A[0], a2 = R(0.5) * A[2];
    const R hm = hl + a0, hum = hul + a0 * s[0];
    if (RP::minus_neg(C, hl, hul) && RP::minus_pos(C, hm, hum)) {
      const R l0 = RP::template sonic<0>(C, hl, hul, 0), l1 = RP::template sonic<0>(C, hm, hum, 0);
      if (l0 < R(0) && l1 > R(0)) {
        const R beta = FM<R>::div(l1 - s[0], l1 - l0);
        zm[0] = beta * l0 * A[0];
        zm[1] = zm[2] = R(0);
        return;
      }
    }
    const R hm2 = hr - a2, hum2 = hur - a2 * s[2];
    if (RP::plus_pos(C, hr, hur) && RP::plus_neg(C, hm2, hum2)) {
      const R m0 = RP::template sonic<0>(C, hm2, hum2, 1), m1 = RP::template sonic<0>(C, hr, hur, 1);
      if (m0 < R(0) && m1 > R(0)) {
        const R beta = FM<R>::div(m1 - s[2], m1 - m0);
        zm[2] = z[2] - (R(1) - beta) * m1 * A[2];
        zm[0] = z[0];
        zm[1] = z[1];
      }
    }
  }
  // the state beside a gravity wave, (h, hu) + A/2 (1, s), has (hu)^2 < g h^3
  // for certain: in FP32 on the values' leading bits (FP64: no instruction of
  // the scarce pipe) with a margin above their error; NaN: no
  __device__ static __forceinline__ bool slow_wave(R g, R h, R A, R hu, R s) {
    const float a = lead_f32(h), b = 0.5f * lead_f32(A), c = lead_f32(hu), d = b * lead_f32(s);
    const float hm = (a + b) - 4e-6f * (fabsf(a) + fabsf(b));
    const float m = fabsf(c + d) + 8e-6f * (fabsf(c) + fabsf(d));
    return hm > 0.f && m * m < 0.9999f * (float)g * (hm * hm * hm);
  }
  // The normal solve: strengths, geometry; returns whether every lane is
  // plainly subsonic (|un|, |ut| < c, and the states beside the first and last
  // waves too, so that no entropy fix applies).  Otherwise zm holds the split.
  template <int DIR>
  __device__ static __forceinline__ bool solve(const MConsts<R>& C, const V (&ql)[M],
                                               const V (&pl)[NP], const V (&qr)[M],
                                               const V (&pr)[NP], V (&A)[MW], V (&g)[NG],
                                               V (&zm)[MW]) {
    constexpr int n = 1 + DIR, t = 2 - DIR, N = VecOf<V>::N;
    const V iden = vrcp_safe(vadd(pl[0], pr[0]));
    const V un = vmul(vadd(pl[n], pr[n]), iden), ut = vmul(vadd(pl[t], pr[t]), iden);
    const V gh = vmul(V(R(0.5) * C.g), vadd(ql[0], qr[0]));
    const V rc = vrsq(gh), c = vmul(gh, rc);
    const V s0 = vsub(un, c), s2 = vadd(un, c);
    g[UN] = un;
    g[UT] = ut;
    g[CS] = c;
    g[RC] = rc;
    g[S0] = s0;
    g[S2] = s2;
    const V d0 = vsub(qr[0], ql[0]);
    // w = (un dh - d(hu_n)) / c = al_0 - al_2
    const V w = vmul(vfma(un, d0, vsub(ql[n], qr[n])), rc);
    A[0] = vadd(d0, w);
    A[1] = vnfma(ut, d0, vsub(qr[t], ql[t]));
    A[2] = vsub(d0, w);
    R x[9][N];
    vget(un, x[0]);
    vget(ut, x[1]);
    vget(c, x[2]);
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i) ok = ok && less_mag(x[0][i], x[1][i], x[2][i]);
    if (C.entropy_fix) {
      if constexpr (N == 1) {
        ok = ok && slow_wave(C.g, ql[0], A[0], ql[n], s0) && slow_wave(C.g, qr[0], -A[2], qr[n], s2);
      } else {
        const V half = V(R(0.5)), a0 = vmul(half, A[0]), a2 = vmul(half, A[2]);
        const V hm = vadd(ql[0], a0), hum = vfma(a0, s0, ql[n]);
        const V hm2 = vsub(qr[0], a2), hum2 = vnfma(a2, s2, qr[n]);
        const V gg = V(R(0.9999) * C.g);
        const V e1 = vnfma(hum, hum, vmul(vmul(hm, hm), vmul(hm, gg)));
        const V e2 = vnfma(hum2, hum2, vmul(vmul(hm2, hm2), vmul(hm2, gg)));
        float a, b, u, v;
        e1.get(a, b);
        e2.get(u, v);
        ok = ok && fminf(fminf(a, b), fminf(u, v)) > 0.f;
      }
    }
    const bool sub = __all_sync(0xffffffffu, ok);
    if (!sub) {
      R A_[3][N], m[3][N];
      vget(ql[0], x[3]);
      vget(ql[n], x[4]);
      vget(qr[0], x[5]);
      vget(qr[n], x[6]);
#pragma unroll
      for (int k = 0; k < 3; ++k) vget(A[k], A_[k]);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const R av[3] = {A_[0][i], A_[1][i], A_[2][i]};
        R mv[3];
        split(C, x[3][i], x[4][i], x[5][i], x[6][i], av, x[0][i], x[2][i], mv);
#pragma unroll
        for (int k = 0; k < 3; ++k) m[k][i] = mv[k];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) zm[k] = vput(m[k]);
    }
    return sub;
  }
  // |un|, |ut| < c
  __device__ static __forceinline__ bool less_mag(float a, float b, float c) {
    return fmaxf(fabsf(a), fabsf(b)) < c;
  }
  __device__ static __forceinline__ bool less_mag(double a, double b, double c) {
    const unsigned long long k = 0x7fffffffffffffffULL, x = (unsigned long long)fbits(a) & k,
                             y = (unsigned long long)fbits(b) & k;
    return (x > y ? x : y) < (unsigned long long)fbits(c) && fbits(c) > 0;
  }
  // |un| + c = max(|s0|, |s2|)
  __device__ static __forceinline__ V speed(const V (&g)[NG]) {
    return vmap([](R a, R b) { return max_speed((R)fabs(a), (R)fabs(b)); }, g[S0], g[S2]);
  }
  // strengths (doubled) of what the face gives the cell below it (km, A^-dQ + F)
  // and above it (kp, A^+dQ - F), limited with the views of the faces below (b)
  // and above (a); FAST or MC: hal = 1 with half limited strengths, else 1/2
  template <bool FAST>
  __device__ static __forceinline__ void strengths(int lim, R hal, R hl, const V (&g)[NG],
                                                   const V (&A)[MW], const V (&zm)[MW], bool sub,
                                                   const V (&bg)[NX], const V (&bA)[MW],
                                                   const V (&ag)[NX], const V (&aA)[MW],
                                                   V (&km)[MW], V (&kp)[MW]) {
    const V one = V(R(1)), H = V(hal), nl = V(-hl);
    const V un = g[UN], ut = g[UT], s0 = g[S0], s2 = g[S2], un2 = vadd(un, un);
    V u0, v0, a0, u2, v2, a2;  // speed, tangential velocity and strength upwind of waves 0, 2
    if (sub) {
      u0 = ag[S0]; v0 = ag[UT]; a0 = aA[0];
      u2 = bg[S2]; v2 = bg[UT]; a2 = bA[2];
    } else {
      u0 = vpick(s0, bg[S0], ag[S0]); v0 = vpick(s0, bg[UT], ag[UT]); a0 = vpick(s0, bA[0], aA[0]);
      u2 = vpick(s2, bg[S2], ag[S2]); v2 = vpick(s2, bg[UT], ag[UT]); a2 = vpick(s2, bA[2], aA[2]);
    }
    const V tt = vfma(ut, ut, one);
    const V n0 = vfma(s0, s0, tt), n2 = vfma(s2, s2, tt);
    const V d0 = vfma(s0, u0, vfma(ut, v0, one)), d2 = vfma(s2, u2, vfma(ut, v2, one));
    const V w0 = vmul(vmul(a0, d0), vrcp_safe(n0)), w2 = vmul(vmul(a2, d2), vrcp_safe(n2));
    const V L0 = vlim<FAST>(lim, w0, A[0]), L1 = vlim<FAST>(lim, vpick(un, bA[1], aA[1]), A[1]),
            L2 = vlim<FAST>(lim, w2, A[2]);
    const V y1 = vmul(vfma(nl, vabs(un), H), L1);
    if (sub) {
      // s0 < 0 < s2: t_0 = -s0 y0, t_2 = s2 y2
      const V y0 = vmul(vfma(V(hl), s0, H), L0), y2 = vmul(vfma(nl, s2, H), L2);
      km[0] = vmul(s0, vsub(A[0], y0));
      kp[0] = vmul(s0, y0);
      km[2] = vmul(s2, y2);
      kp[2] = vmul(s2, vsub(A[2], y2));
      const V p = vmul(un2, y1), z = vmul(un2, vsub(A[1], y1));
      km[1] = vneg_pick(un, z, p);
      kp[1] = vneg_pick(un, p, z);
    } else {
      const V r0 = vabs(s0), r2 = vabs(s2);
      const V t0 = vmul(vmul(vfma(nl, r0, H), L0), r0), t1 = vmul(y1, vabs(un2)),
              t2 = vmul(vmul(vfma(nl, r2, H), L2), r2);
      km[0] = vadd(zm[0], t0);
      km[1] = vadd(zm[1], t1);
      km[2] = vadd(zm[2], t2);
      kp[0] = vsub(vsub(vmul(s0, A[0]), zm[0]), t0);
      kp[1] = vsub(vsub(vmul(un2, A[1]), zm[1]), t1);
      kp[2] = vsub(vsub(vmul(s2, A[2]), zm[2]), t2);
    }
  }
  // the same without the corrections (transverse mode 1)
  __device__ static __forceinline__ void plain(const V (&g)[NG], const V (&A)[MW],
                                               const V (&zm)[MW], bool sub, V (&km)[MW],
                                               V (&kp)[MW]) {
    const V un = g[UN], un2 = vadd(un, un), zero = V(R(0));
    const V z0 = vmul(g[S0], A[0]), z1 = vmul(un2, A[1]), z2 = vmul(g[S2], A[2]);
    km[0] = sub ? z0 : zm[0];
    km[1] = sub ? vneg_pick(un, z1, zero) : zm[1];
    km[2] = sub ? zero : zm[2];
    kp[0] = vsub(z0, km[0]);
    kp[1] = vsub(z1, km[1]);
    kp[2] = vsub(z2, km[2]);
  }
  // sum_p k_p r_p (doubled)
  template <int DIR>
  __device__ static __forceinline__ void vec(const V (&g)[NG], const V (&k)[MW], V (&o)[M]) {
    constexpr int n = 1 + DIR, t = 2 - DIR;
    const V kap = vadd(k[0], k[2]);
    o[0] = kap;
    o[n] = vfma(g[UN], kap, vmul(g[CS], vsub(k[2], k[0])));
    o[t] = vfma(kap, g[UT], k[1]);
  }
  // transverse parts of sum_p k_p r_p (four times)
  template <int DIR>
  __device__ static __forceinline__ void trans(const V (&g)[NG], bool sub, const V (&k)[MW],
                                               V (&bm)[M], V (&bp)[M]) {
    constexpr int n = 1 + DIR, t = 2 - DIR;
    const V un = g[UN], ut = g[UT], c = g[CS];
    const V kap = vadd(k[0], k[2]), w = vmul(k[1], g[RC]);
    const V b0 = vsub(kap, w), b2 = vadd(kap, w);
    // shear strength c (k_2 - k_0) times its speed ut
    const V m = vmul(vadd(ut, ut), vmul(c, vsub(k[2], k[0])));
    V mm, mp;
    vsplit(ut, m, mm, mp);
    const V l0 = vsub(ut, c), l2 = vadd(ut, c), z0 = vmul(l0, b0), z2 = vmul(l2, b2);
    if (sub) {
      bm[0] = z0;
      bm[t] = vmul(z0, l0);
      bm[n] = vfma(z0, un, mm);
      bp[0] = z2;
      bp[t] = vmul(z2, l2);
      bp[n] = vfma(z2, un, mp);
    } else {
      V m0, m2, p0, p2;
      vsplit(l0, z0, m0, p0);
      vsplit(l2, z2, m2, p2);
      bm[0] = vadd(m0, m2);
      bm[t] = vfma(m0, l0, vmul(m2, l2));
      bm[n] = vfma(bm[0], un, mm);
      bp[0] = vadd(p0, p2);
      bp[t] = vfma(p0, l0, vmul(p2, l2));
      bp[n] = vfma(bp[0], un, mp);
    }
  }
};

// ---------------------------------------------------------------------------
// the walk
// ---------------------------------------------------------------------------
__host__ __device__ constexpr RegTile roe_tile(int prec, int bw) {
  // FP64: one column per lane, two or four warps per block; FP32: pairs, one
  // or two warps
  return prec == 0 ? RegTile{1, bw == 128 ? 4 : 2, bw == 128 ? 112 : 56}
                   : RegTile{2, bw == 128 ? 2 : 1, bw == 128 ? 120 : 60};
}

template <class RP, class V, int NWB, bool FAST>
__global__ void __launch_bounds__(32 * NWB, VecOf<V>::N == 1 ? 0 : 12 / NWB)
    roe2d_kernel(const Member* __restrict__ members, const Tile* __restrict__ tiles,
                 const MConsts<typename VecOf<V>::S> C, int H, int sweep) {
  using R = typename VecOf<V>::S;
  using SY = RoeSys<V, RP>;
  constexpr int M = SY::M, MW = SY::MW, NP = SY::NP, NG = SY::NG, NX = SY::NX;
  constexpr int N = VecOf<V>::N, WL = 32 * N;
  const Tile tl = tiles ? tiles[blockIdx.x] : Tile{0, (int)blockIdx.x};
  const Member& mb = members[tl.member];
  DevCtl* ctl = mb.ctl;
  pdl_enter();  // (the tables above do not change between attempts)
  if (ctl->done) return;  // the whole block
  const int lane = threadIdx.x & 31;
  const R lx = dt_over_dx<R>(ctl, 0), ly = dt_over_dx<R>(ctl, 1);
  const R hal = C.order == 2 ? ((FAST || C.lim == CLAW_LIM_MC) ? R(1) : R(0.5)) : R(0);
  const R hlx = hal * lx, hly = hal * ly;
  // sums are doubled, transverse parts four times
  const V nlx = V(R(-0.5) * lx), nly = V(R(-0.5) * ly), kxy = V(R(0.125) * lx * ly),
          nkxy = V(R(-0.125) * lx * ly);
  const int cur = ctl->cur, nbuf = ctl->nbuf;
  const int nx = mb.nx, ny = mb.ny;
  const Classic2dLayout L = classic2d_layout(nx, ny, NWB * (WL - 4), H);
  const int c0 = (tl.tile % L.nsx) * L.TX + (threadIdx.x >> 5) * (WL - 4), ch = tl.tile / L.nsx;
  const int r0 = (int)(((long long)ch * ny) / L.nch);
  const int r1 = (int)(((long long)(ch + 1) * ny) / L.nch);
  const bool dox = sweep != 2, doy = sweep != 1;
  const int mode = FAST ? 2 : (sweep == 0 ? C.transverse : 0);
  const int lim = C.lim;
  const R* __restrict__ q = (const R*)step_input(mb, cur, nbuf, sweep == 2 ? 1 : 0);
  R* __restrict__ qo = (R*)mb.q[(cur + (sweep == 2 ? 2 : 1)) % nbuf];
  const size_t plane = (size_t)nx * ny;
  const int g0c = c0 - 2 + N * lane;
  const bool inner = g0c >= 0 && g0c + N <= nx;
  const bool vec = N > 1 && (nx & 1) == 0 && (((size_t)q | (size_t)qo) & (2 * sizeof(R) - 1)) == 0;
  // (plain values: packing them into pairs here would wait for the loads)
  auto load = [&](int r, R (&v)[M][N]) {
    if (inner && r >= 0 && r < ny) {
      const R* p = q + (size_t)r * nx + g0c;
#pragma unroll
      for (int k = 0; k < M; ++k) ld_pair<N>(p + k * plane, vec, v[k][0], v[k][N - 1]);
    } else {
#pragma unroll
      for (int c = 0; c < N; ++c) {
        R s[M];
        load_cell<M, R>(C, q, nx, ny, min(g0c + c, nx + 1), r, RP::WALL_X, RP::WALL_Y, s);
#pragma unroll
        for (int k = 0; k < M; ++k) v[k][c] = s[k];
      }
    }
  };

  // columns whose lower y-face / x-face speeds count here
  bool ownx[N], owny[N];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    const int l = N * lane + c;
    ownx[c] = l >= 2 && l <= WL - 2 && g0c + c <= nx;
    owny[c] = l >= 2 && l < WL - 2 && g0c + c < nx;
  }
  const V zero = V(R(0));
  // rows r-1, r-2: state and increments so far; row r-1's prepared values
  V q1[M], q2[M], p1[NP], D1[M], D2[M];
  // y-face r-1; the limiter's view of face r-2; what face r-2 gives the row
  // above it (the vector and its x splits); upward y splits of row r-1
  V al1[MW], g1[NG], zm1[MW], al2[MW], g2[NX];
  bool sub1 = false;
  V pv[M], pbm[M], pbp[M], By1[M];
#pragma unroll
  for (int k = 0; k < M; ++k) q1[k] = q2[k] = D1[k] = D2[k] = pv[k] = pbm[k] = pbp[k] = By1[k] = zero;
#pragma unroll
  for (int k = 0; k < NP; ++k) p1[k] = zero;
#pragma unroll
  for (int p = 0; p < MW; ++p) al1[p] = zm1[p] = al2[p] = zero;
#pragma unroll
  for (int k = 0; k < NG; ++k) g1[k] = zero;
#pragma unroll
  for (int k = 0; k < NX; ++k) g2[k] = zero;
  R smx = R(0), smy = R(0);
  int bad = 0;
  R qn[M][N];
  if (c0 < nx) load(r0 - 2, qn);
  for (int r = c0 < nx ? r0 - 2 : r1 + 2; r <= r1 + 1; ++r) {
    V q0[M], p0[NP], D0[M];
#pragma unroll
    for (int k = 0; k < M; ++k) {
      q0[k] = vput(qn[k]);
      D0[k] = zero;
    }
    if (r <= r1) load(r + 1, qn);
    SY::prep(C, q0, p0);
    if (doy) {
      // y-face r (rows r-1, r)
      V al[MW], g[NG], zm[MW];
#pragma unroll
      for (int p = 0; p < MW; ++p) zm[p] = zero;
      const bool sub = SY::template solve<1>(C, q1, p1, q0, p0, al, g, zm);
      if (r >= r0 && r <= r1) {
        R s[N];
        vget(SY::speed(g), s);
#pragma unroll
        for (int c = 0; c < N; ++c)
          if (owny[c]) smy = max_speed(smy, s[c]);
      }
      // limit face r-1; what it gives rows r-2 and r-1
      V km[MW], kp[MW], mv[M], ga[NX];
#pragma unroll
      for (int k = 0; k < NX; ++k) ga[k] = g[k];
      SY::template strengths<FAST>(lim, hal, hly, g1, al1, zm1, sub1, g2, al2, ga, al, km, kp);
      SY::template vec<1>(g1, km, mv);
#pragma unroll
      for (int k = 0; k < M; ++k) D2[k] = vfma(nly, vadd(pv[k], mv[k]), D2[k]);
      SY::template vec<1>(g1, kp, pv);
      if (mode) {
        if (!FAST && mode == 1) SY::plain(g1, al1, zm1, sub1, km, kp);
        V bm[M], bp[M];
        SY::template trans<1>(g1, sub1, km, bm, bp);
#pragma unroll
        for (int k = 0; k < M; ++k) {
          // x-faces of row r-2
          const V h = vadd(vleft(vadd(pbp[k], bp[k])), vadd(pbm[k], bm[k]));
          D2[k] = vfma(kxy, vsub(vright(h), h), D2[k]);
        }
        SY::template trans<1>(g1, sub1, kp, pbm, pbp);
      }
      sub1 = sub;
#pragma unroll
      for (int p = 0; p < MW; ++p) {
        al2[p] = al1[p];
        al1[p] = al[p];
        zm1[p] = zm[p];
      }
#pragma unroll
      for (int k = 0; k < NX; ++k) g2[k] = g1[k];
#pragma unroll
      for (int k = 0; k < NG; ++k) g1[k] = g[k];
    }
    if (dox && r >= r0 - 1 && r <= r1) {
      // x-face below each column of row r
      V ql[M], pl[NP], al[MW], g[NG], zm[MW], km[MW], kp[MW], mv[M], pw[M];
#pragma unroll
      for (int k = 0; k < M; ++k) ql[k] = vleft(q0[k]);
#pragma unroll
      for (int k = 0; k < NP; ++k) pl[k] = vleft(p0[k]);
#pragma unroll
      for (int p = 0; p < MW; ++p) zm[p] = zero;
      const bool sub = SY::template solve<0>(C, ql, pl, q0, p0, al, g, zm);
      if (r >= r0 && r < r1) {
        R s[N];
        vget(SY::speed(g), s);
#pragma unroll
        for (int c = 0; c < N; ++c)
          if (ownx[c]) smx = max_speed(smx, s[c]);
      }
      {
        V bg[NX], bal[MW], ag[NX], aal[MW];
#pragma unroll
        for (int k = 0; k < NX; ++k) {
          bg[k] = sub && SY::above_only(k) ? zero : vleft(g[k]);
          ag[k] = sub && SY::below_only(k) ? zero : vright(g[k]);
        }
#pragma unroll
        for (int p = 0; p < MW; ++p) {
          bal[p] = sub && p == 0 ? zero : vleft(al[p]);
          aal[p] = sub && p == MW - 1 ? zero : vright(al[p]);
        }
        SY::template strengths<FAST>(lim, hal, hlx, g, al, zm, sub, bg, bal, ag, aal, km, kp);
      }
      SY::template vec<0>(g, km, mv);
      SY::template vec<0>(g, kp, pw);
#pragma unroll
      for (int k = 0; k < M; ++k) D0[k] = vmul(nlx, vadd(pw[k], vright(mv[k])));
      if (mode) {
        if (!FAST && mode == 1) SY::plain(g, al, zm, sub, km, kp);
        V bmm[M], bpm[M], bmp[M], bpp[M];
        SY::template trans<0>(g, sub, km, bmm, bpm);
        SY::template trans<0>(g, sub, kp, bmp, bpp);
#pragma unroll
        for (int k = 0; k < M; ++k) {
          // y-face between rows r-1 and r
          const V h = vadd(By1[k], vadd(bmp[k], vright(bmm[k])));
          D1[k] = vfma(kxy, h, D1[k]);
          D0[k] = vfma(nkxy, h, D0[k]);
          By1[k] = vadd(bpp[k], vright(bpm[k]));
        }
      }
    }
    if (r - 2 >= r0) {
      R o[M][N];
#pragma unroll
      for (int k = 0; k < M; ++k) vget(vadd(q2[k], D2[k]), o[k]);
      const int l = N * lane;
      if (l >= 2 && l < WL - 2 && g0c < nx) {
        const bool two = N > 1 && g0c + 1 < nx;
#pragma unroll
        for (int k = 0; k < M; ++k) {
          const R a = o[k][0], b = o[k][N - 1];
          bad |= not_finite(a);
          if (two) bad |= not_finite(b);
          st_pair(qo + k * plane + (size_t)(r - 2) * nx + g0c, two, vec, a, b);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < M; ++k) {
      q2[k] = q1[k];
      q1[k] = q0[k];
      D2[k] = D1[k];
      D1[k] = D0[k];
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) p1[k] = p0[k];
  }
  finish_attempt<R>(ctl, smx, smy, bad, mb.ntiles, sweep != 1);
}

}  // namespace claw
