// medium2d.cuh -- the 2D classic step of acoustics in a varying medium
// (RpAcousticsVC: aux rho, c per cell, optionally a capacity kappa) in
// strength form, one launch per attempt (two for a dimensionally split step).
//
// The waves of a face are a_1 (-Z_l, 1) and a_2 (Z_r, 1), so theta_1 is the
// ratio of strengths times (1 + Z_l Z_r) / (1 + Z_l^2) (theta_2: 1 + Z_r^2),
// and what enters a cell across its two d-faces, S_d, has pressure and normal
// velocity only.  With tau_d = dt/dx_d S_d,p / kappa the transverse split of a
// cell's fluctuations into its e-faces depends on tau_d alone; the face
// between cells X-e and X receives
//   G_p = -1/2 (c_X Z_X tau(X-e) - c_{X-e} Z_{X-e} tau(X)) / (Z_{X-e} + Z_X)
//   G_u = -1/2 (c_X tau(X-e) + c_{X-e} tau(X)) / (Z_{X-e} + Z_X).
// The same sums as splitting each fluctuation vector on its own; only the
// rounding differs.
//
// Layout as in linear2d.cuh: a warp owns a strip of columns and walks a chunk
// of rows; x neighbours by shuffles, y neighbours in registers.
// With row r loaded it has tau_x of row r, tau_y of row r - 2 and finishes
// row r - 2.  Fused multiply-adds are written out, so every shape gives the
// same bits.
//
// What bounds it: FP32 issue and latency (43 % issue at 1024^2, one wave of
// 1026 warps), FP64 the FP64 pipe.  1024^2 with capacity FP32 211 -> 42
// us/step, FP64 973 -> 370 us, 301 x 280 FP64 110 -> 81 us against a record of
// seven vectors per face written by two sweeps and gathered by an update.
#pragma once

#include "linear2d.cuh"

namespace claw {

// one cell's medium: impedance, sound speed, c Z, 1/kappa, 1/(1 + Z^2)
template <typename R>
struct Med {
  R Z, c, cz, ik, w;
};

// per-direction constants: dt/dx, dt/(2 dx), order (1/2, or 1 with MC's half
// strengths; 0 for first order)
template <typename R>
struct MedK {
  R lam, hl, hal;
};

// p (to the cell above) and m (to the cell below) of a face, components
// pressure and normal velocity, from its strengths and the upwind ones
template <bool FAST, typename R>
__device__ __forceinline__ void med_face(const MedK<R>& k, int lim, const Med<R>& l,
                                         const Med<R>& r, const R (&a)[2], const R (&up)[2],
                                         R (&p)[2], R (&m)[2]) {
  // the upwind faces: above for the wave of speed -c_l, below for c_r (sound
  // speeds are not negative; one of zero carries no correction)
  const R g = fma(l.Z, r.Z, R(1));
  const R u1 = mulr(mulr(up[0], g), l.w);
  const R u2 = mulr(mulr(up[1], g), r.w);
  const R dtc = mulr(k.hl, l.ik + r.ik);  // dt/dx times the mean 1/kappa
  const R t1 = mulr(mulr(mulr(k.hal, l.c), fma(-dtc, l.c, R(1))), lin_limit<FAST>(lim, u1, a[0]));
  const R t2 = mulr(mulr(mulr(k.hal, r.c), fma(-dtc, r.c, R(1))), lin_limit<FAST>(lim, u2, a[1]));
  const R F0 = fma(r.Z, t2, -mulr(l.Z, t1)), Fn = t1 + t2;
  p[0] = fma(r.cz, a[1], -F0);
  p[1] = fma(r.c, a[1], -Fn);
  m[0] = fma(l.cz, a[0], F0);
  m[1] = fma(-l.c, a[0], Fn);
}
// largest Courant speed of a face's waves: each uses the capacity of the cell
// it moves into
template <typename R>
__device__ __forceinline__ R med_speed(const Med<R>& l, const Med<R>& r) {
  return max_nonneg((R)fabs(mulr(l.c, l.ik)), (R)fabs(mulr(r.c, r.ik)));
}

template <class RP, typename R, int BW, bool FAST>
__global__ void __launch_bounds__(32 * reg_tile(sizeof(R) == 8 ? 0 : 1, BW).warps)
    medium2d_kernel(const Member* __restrict__ members, const Tile* __restrict__ tiles,
                    const MConsts<R> C, int H, int sweep) {
  constexpr RegTile RT = reg_tile(sizeof(R) == 8 ? 0 : 1, BW);
  constexpr int M = 3, MA = 2, N = RT.n, WL = 32 * N;  // columns per lane, per warp
  constexpr unsigned FULL = 0xffffffffu;
  const Tile tl = tiles ? tiles[blockIdx.x] : Tile{0, (int)blockIdx.x};
  const Member& mb = members[tl.member];
  DevCtl* ctl = mb.ctl;
  pdl_enter();  // (the tables above do not change between attempts)
  if (ctl->done) return;  // the whole block
  const int lane = threadIdx.x & 31;
  MedK<R> K[2];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    K[d].lam = dt_over_dx<R>(ctl, d);
    K[d].hl = R(0.5) * K[d].lam;
    K[d].hal = C.order == 2 ? (C.lim == CLAW_LIM_MC ? R(1) : R(0.5)) : R(0);
  }
  const int cur = ctl->cur, nbuf = ctl->nbuf;
  const int nx = mb.nx, ny = mb.ny;
  const Classic2dLayout L = classic2d_layout(nx, ny, RT.tx, H);
  const int c0 = (tl.tile % L.nsx) * L.TX + (threadIdx.x >> 5) * (WL - 4), ch = tl.tile / L.nsx;
  const int r0 = (int)(((long long)ch * ny) / L.nch);
  const int r1 = (int)(((long long)(ch + 1) * ny) / L.nch);
  const bool dox = sweep != 2, doy = sweep != 1;
  const int mode = FAST ? 2 : (sweep == 0 ? C.transverse : 0);
  const int lim = C.lim;
  const R* __restrict__ q = (const R*)step_input(mb, cur, nbuf, sweep == 2 ? 1 : 0);
  R* __restrict__ qo = (R*)mb.q[(cur + (sweep == 2 ? 2 : 1)) % nbuf];
  const R* __restrict__ aux = (const R*)mb.aux;
  const size_t plane = (size_t)nx * ny;
  const int g0 = c0 - 2 + N * lane;
  const bool inner = g0 >= 0 && g0 + N <= nx;
  const bool capa = C.capa >= 0;
  const bool vec =
      (nx & 1) == 0 && (((size_t)q | (size_t)qo | (size_t)aux) & (2 * sizeof(R) - 1)) == 0;
  // fields of a row: p, u, v, rho, c, kappa
  auto load = [&](int r, R (&v)[N][6]) {
    if (inner && r >= 0 && r < ny) {
      const size_t off = (size_t)r * nx + g0;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        if (k == 5 && !capa) break;
        const R* p = (k < 3 ? q + k * plane : aux + (k - 3) * plane) + off;
#pragma unroll
        for (int c = 0; c < N; c += 2) ld_pair<N>(p + c, vec, v[c][k], v[c + (N > 1)][k]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const int col = min(g0 + c, nx + 1);
        R s[M], a[MA];
        load_cell<M, R>(C, q, nx, ny, col, r, RP::WALL_X, RP::WALL_Y, s);
        load_aux<MA, R>(C, aux, nx, ny, col, r, a);
        v[c][0] = s[0];
        v[c][1] = s[1];
        v[c][2] = s[2];
        v[c][3] = a[0];
        v[c][4] = a[1];
        if (capa) v[c][5] = load_aux_field<R>(C, aux, nx, ny, col, r, C.capa);
      }
    }
  };
  auto shup = [&](const Med<R>& m) {
    Med<R> o;
    o.Z = __shfl_up_sync(FULL, m.Z, 1);
    o.c = __shfl_up_sync(FULL, m.c, 1);
    o.ik = __shfl_up_sync(FULL, m.ik, 1);
    o.w = __shfl_up_sync(FULL, m.w, 1);
    o.cz = mulr(o.c, o.Z);
    return o;
  };

  // per column: increments so far (rows r-1, r-2; added to the state once, when
  // the row is finished), media of rows r-1, r-2,
  // 1/(Z_l + Z_r) of the lower x-face of row r-1, r-2, tau_x of row r-1;
  // y-faces: strengths of faces r-1, r-2, what face r-2 gives the cell above
  R q1[N][M], q2[N][M], acc1[N][M], acc2[N][M], iz1[N], iz2[N], tx1[N], ya1[N][2], ya2[N][2], yp2[N][2], pz[N], vz[N];
  Med<R> m1[N], m2[N];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    iz1[c] = iz2[c] = tx1[c] = pz[c] = vz[c] = R(0);
    m1[c] = m2[c] = Med<R>{R(1), R(0), R(0), R(0), R(0)};
#pragma unroll
    for (int k = 0; k < M; ++k) acc1[c][k] = acc2[c][k] = q1[c][k] = q2[c][k] = R(0);
#pragma unroll
    for (int s = 0; s < 2; ++s) ya1[c][s] = ya2[c][s] = yp2[c][s] = R(0);
  }
  int bad = 0;
  R smx = R(0), smy = R(0);
  R qn[N][6];
  if (c0 < nx) load(r0 - 2, qn);
  for (int r = c0 < nx ? r0 - 2 : r1 + 2; r <= r1 + 1; ++r) {
    R q0[N][M], acc0[N][M], tx[N], ty[N], iz[N];
    Med<R> m0[N];
#pragma unroll
    for (int c = 0; c < N; ++c) {
#pragma unroll
      for (int k = 0; k < M; ++k) {
        q0[c][k] = qn[c][k];
        acc0[c][k] = R(0);
      }
      m0[c].c = qn[c][4];
      m0[c].Z = mulr(qn[c][3], qn[c][4]);
      m0[c].cz = mulr(m0[c].c, m0[c].Z);
      m0[c].ik = capa ? FM<R>::rcp(qn[c][5]) : R(1);
      m0[c].w = FM<R>::rcp(fma(m0[c].Z, m0[c].Z, R(1)));
      tx[c] = ty[c] = iz[c] = R(0);
    }
    if (r <= r1) load(r + 1, qn);
    const bool xrow = r >= r0 - 1 && r <= r1;
    // y direction: face r (rows r-1, r), limit face r-1, tau_y of row r-2;
    // then face r's transverse part of tau_x (rows r-1 and r)
    R izy[N];
    if (doy) {
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R p = q0[c][0], v = q0[c][2];
        izy[c] = FM<R>::rcp(m1[c].Z + m0[c].Z);
        R a[2], fp[2], fm[2];
        const R dp = p - pz[c], du = v - vz[c];
        a[0] = mulr(fma(m0[c].Z, du, -dp), izy[c]);
        a[1] = mulr(fma(m1[c].Z, du, dp), izy[c]);
        const R up[2] = {a[0], ya2[c][1]};
        med_face<FAST>(K[1], lim, m2[c], m1[c], ya1[c], up, fp, fm);
        const R li = mulr(K[1].lam, m2[c].ik);
        ty[c] = mulr(li, yp2[c][0] + fm[0]);
        acc2[c][0] -= ty[c];
        acc2[c][2] = fma(-li, yp2[c][1] + fm[1], acc2[c][2]);
        if (!FAST && mode == 1) ty[c] = mulr(li, fma(m2[c].cz, ya2[c][1], mulr(m2[c].cz, ya1[c][0])));
        const int l = N * lane + c;
        if (l >= 2 && l < WL - 2 && g0 + c < nx && r >= r0 && r <= r1)
          smy = max_nonneg(smy, med_speed(m1[c], m0[c]));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          ya2[c][s] = ya1[c][s];
          ya1[c][s] = a[s];
          yp2[c][s] = fp[s];
        }
        pz[c] = p;
        vz[c] = v;
      }
    }
    // x direction, row r
    if (dox && xrow) {
      R a[N][2], fp[N][2], fm[N + 1][2];
      const Med<R> ml = shup(m0[N - 1]);
      const R pl = __shfl_up_sync(FULL, q0[N - 1][0], 1);
      const R ul = __shfl_up_sync(FULL, q0[N - 1][1], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R Zl = c == 0 ? ml.Z : m0[c > 0 ? c - 1 : 0].Z;
        iz[c] = FM<R>::rcp(Zl + m0[c].Z);
        const R dp = q0[c][0] - (c == 0 ? pl : q0[c > 0 ? c - 1 : 0][0]);
        const R du = q0[c][1] - (c == 0 ? ul : q0[c > 0 ? c - 1 : 0][1]);
        a[c][0] = mulr(fma(m0[c].Z, du, -dp), iz[c]);
        a[c][1] = mulr(fma(Zl, du, dp), iz[c]);
      }
      const R bl = __shfl_up_sync(FULL, a[N - 1][1], 1), bu = __shfl_down_sync(FULL, a[0][0], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R up[2] = {c == N - 1 ? bu : a[c < N - 1 ? c + 1 : 0][0],
                         c == 0 ? bl : a[c > 0 ? c - 1 : 0][1]};
        const Med<R> lm = c == 0 ? ml : m0[c > 0 ? c - 1 : 0];
        med_face<FAST>(K[0], lim, lm, m0[c], a[c], up, fp[c], fm[c]);
        const int l = N * lane + c;
        if (l >= 2 && l <= WL - 2 && g0 + c <= nx && r >= r0 && r < r1)
          smx = max_nonneg(smx, med_speed(lm, m0[c]));
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) fm[N][s] = __shfl_down_sync(FULL, fm[0][s], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R li = mulr(K[0].lam, m0[c].ik);
        tx[c] = mulr(li, fp[c][0] + fm[c + 1][0]);
        acc0[c][0] = -tx[c];
        acc0[c][1] = mulr(-li, fp[c][1] + fm[c + 1][1]);
        if (!FAST && mode == 1)
          tx[c] = mulr(li, fma(m0[c].cz, a[c][1], mulr(m0[c].cz, c == N - 1 ? bu : a[c < N - 1 ? c + 1 : 0][0])));
      }
    }
    if (mode) {
      // y-faces r from tau_x of rows r-1, r
      if (r >= r0 && r <= r1) {
#pragma unroll
        for (int c = 0; c < N; ++c) {
          const R h0 = mulr(izy[c], fma(m0[c].cz, tx1[c], -mulr(m1[c].cz, tx[c])));
          const R hv = mulr(izy[c], fma(m0[c].c, tx1[c], mulr(m1[c].c, tx[c])));
          const R lb = mulr(K[1].hl, m1[c].ik), la = mulr(K[1].hl, m0[c].ik);
          acc1[c][0] = fma(lb, h0, acc1[c][0]);
          acc1[c][2] = fma(lb, hv, acc1[c][2]);
          acc0[c][0] = fma(-la, h0, acc0[c][0]);
          acc0[c][2] = fma(-la, hv, acc0[c][2]);
        }
      }
      // x-faces of row r-2 from tau_y
      R h0[N + 1], hu[N + 1];
      const R tl_ = __shfl_up_sync(FULL, ty[N - 1], 1);
      const R cl_ = __shfl_up_sync(FULL, m2[N - 1].c, 1);
      const R czl = __shfl_up_sync(FULL, m2[N - 1].cz, 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R t = c == 0 ? tl_ : ty[c > 0 ? c - 1 : 0];
        const R cm = c == 0 ? cl_ : m2[c > 0 ? c - 1 : 0].c;
        const R zm = c == 0 ? czl : m2[c > 0 ? c - 1 : 0].cz;
        h0[c] = mulr(iz2[c], fma(m2[c].cz, t, -mulr(zm, ty[c])));
        hu[c] = mulr(iz2[c], fma(m2[c].c, t, mulr(cm, ty[c])));
      }
      h0[N] = __shfl_down_sync(FULL, h0[0], 1);
      hu[N] = __shfl_down_sync(FULL, hu[0], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R li = mulr(K[0].hl, m2[c].ik);
        acc2[c][0] = fma(li, h0[c + 1] - h0[c], acc2[c][0]);
        acc2[c][1] = fma(li, hu[c + 1] - hu[c], acc2[c][1]);
      }
    }
    if (r - 2 >= r0) {
#pragma unroll
      for (int c = 0; c < N; c += 2) {
        const int l = N * lane + c;
        if (l >= 2 && l < WL - 2 && g0 + c < nx) {
          const bool two = N > 1 && g0 + c + 1 < nx;
#pragma unroll
          for (int k = 0; k < M; ++k) {
            const R a = q2[c][k] + acc2[c][k], b = q2[c + (N > 1)][k] + acc2[c + (N > 1)][k];
            bad |= not_finite(a);
            if (two) bad |= not_finite(b);
            st_pair(qo + k * plane + (size_t)(r - 2) * nx + (g0 + c), two, vec, a, b);
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < N; ++c) {
      tx1[c] = tx[c];
      iz2[c] = iz1[c];
      iz1[c] = iz[c];
      m2[c] = m1[c];
      m1[c] = m0[c];
#pragma unroll
      for (int k = 0; k < M; ++k) {
        acc2[c][k] = acc1[c][k];
        acc1[c][k] = acc0[c][k];
        q2[c][k] = q1[c][k];
        q1[c][k] = q0[c][k];
      }
    }
  }
  finish_attempt<R>(ctl, smx, smy, bad, mb.ntiles, sweep != 1);
}

}  // namespace claw
