// classic3d.cuh -- 3D unsplit Clawpack-classic step (LeVeque 1997): normal
// solves, limited corrections, transverse and double-transverse propagation,
// for scalar advection and linear acoustics, in one launch per attempt.
//
// In strength form (linear.cuh) a direction's sums reduce to one scalar per
// cell, tau_d, on which the transverse terms are stencils, so a step needs no
// face records: the state is read once (plus tile halos) and written once.
//
// Layout.  A warp holds 32 consecutive cells of one x line (lanes 2 .. 29 own
// theirs), a block's NW warps consecutive y lines (warps 2 .. NW-3 own theirs)
// and the block walks a segment of z planes.  x neighbours come by warp
// shuffles, y neighbours through shared memory (two barriers per plane), z
// neighbours are the thread's own values of earlier planes: with plane k
// loaded, tau_x and tau_y of plane k, tau_z of plane k-2 and the finished
// cells of plane k-2.  Every cell is computed by the same instructions
// wherever its tile starts, and written by one thread, so results do not
// depend on the tiling or on scheduling: batches and servers match single
// solves bit for bit.
//
// What bounds it: FP64 the FP64 pipe (83 % of its peak at 112 x 120 x 128);
// FP32 instruction issue (73 % active, 64 registers, two blocks per SM; the
// halo lines and planes are computed again by each tile).  Acoustics 256^3
// FP32 1.85 -> 0.447 ms/step, 128^3 FP64 3.01 -> 0.753 ms, 24^3 FP32 124 -> 26
// us, against three face sweeps and an update over per-face records (560 B
// per cell and step in FP32; now 32 B plus the tile halos).
#pragma once

#include "kernels.h"
#include "linear.cuh"
#include "riemann.cuh"

namespace claw {

// cell (i, j, k) of q[M][nz][ny][nx] with ghost remap: x rule, then y rule on
// the x-remapped value, then z rule (corners defined as x, y, z fills in turn)
template <int M, typename R>
__device__ __forceinline__ void load_cell3(const MConsts<R>& C, const R* __restrict__ q, int nx,
                                           int ny, int nz, int i, int j, int k, int wall0,
                                           int wall1, int wall2, R (&out)[M]) {
  int fz, iz, fy, iy, fx, ix;
  const int kk = bc_map(k, nz, C.bc_lo[2], C.bc_hi[2], fz, iz);
  const int jj = bc_map(j, ny, C.bc_lo[1], C.bc_hi[1], fy, iy);
  const int ii = bc_map(i, nx, C.bc_lo[0], C.bc_hi[0], fx, ix);
  if (iz || iy || ix) {
    // an inflow rule at any level replaces the value below it
#pragma unroll
    for (int c = 0; c < M; ++c) out[c] = C.inflow[c];
    if (iz) return;
    if (iy) {
#pragma unroll
      for (int c = 0; c < M; ++c)
        if (fz && c == wall2) out[c] = -out[c];
      return;
    }
  } else {
    const size_t plane = (size_t)nx * ny * nz;
    const size_t off = ((size_t)kk * ny + jj) * nx + ii;
#pragma unroll
    for (int c = 0; c < M; ++c) out[c] = __ldg(q + c * plane + off);
#pragma unroll
    for (int c = 0; c < M; ++c)
      if (fx && c == wall0) out[c] = -out[c];
  }
#pragma unroll
  for (int c = 0; c < M; ++c) {
    if (fy && c == wall1) out[c] = -out[c];
    if (fz && c == wall2) out[c] = -out[c];
  }
}

// owned cells per warp, lines per block (all but the outer two on each side
// own theirs), and the longest segment of z planes a block walks
constexpr int kXOwn3d = 28;
constexpr int kXSweepLines = 16;
constexpr int kZSeg3d = 64;

struct Layout3 {
  int nxc, nyb, nzs;  // blocks along x and y, segments along z
};
// The number of z segments that makes waves x planes walked least: a block
// walks its own planes and four more, and the GPU holds about two blocks per
// SM in FP32 and one in FP64.  Any number gives the same bits.
inline Layout3 layout3d(int nx, int ny, int nz, int prec) {
  Layout3 L;
  L.nxc = (nx + kXOwn3d - 1) / kXOwn3d;
  L.nyb = (ny + kXSweepLines - 4 - 1) / (kXSweepLines - 4);
  const long long slots = prec == 0 ? 152 : 304, per = (long long)L.nxc * L.nyb;
  long long best = 0;
  L.nzs = 1;
  for (int s = (nz + kZSeg3d - 1) / kZSeg3d; s <= nz; s += s < 16 ? 1 : s / 4) {
    const long long cost = (per * s + slots - 1) / slots * ((nz + s - 1) / s + 4);
    if (best == 0 || cost < best) {
      best = cost;
      L.nzs = s;
    }
  }
  return L;
}
inline int classic3d_blocks(const Layout3& L) { return L.nxc * L.nyb * L.nzs; }

// owner columns of block bx, lines of block by, planes of segment bz
struct Tile3 {
  int x0, y0, z0, z1;
};
__host__ __device__ inline Tile3 tile3d(int t, int nz, const Layout3& L) {
  const int bx = t % L.nxc, by = (t / L.nxc) % L.nyb, bz = t / (L.nxc * L.nyb);
  Tile3 T;
  T.x0 = bx * kXOwn3d;
  T.y0 = by * (kXSweepLines - 4);
  T.z0 = (int)((long long)bz * nz / L.nzs);
  T.z1 = (int)((long long)(bz + 1) * nz / L.nzs);
  return T;
}

// FAST: the MC limiter, second order and transverse mode 2 fixed at compile time
template <class RP, typename R, bool FAST>
__global__ void __launch_bounds__(32 * kXSweepLines, sizeof(R) == 4 ? 2 : 1)
    classic3d_kernel(const Member* __restrict__ members, const MConsts<R> C, const Layout3 L) {
  using LS = Lin<RP, R>;
  constexpr int M = RP::M, NS = LS::NS, NW = kXSweepLines;
  constexpr bool VEL = LS::VEL;
  constexpr unsigned FULL = 0xffffffffu;
  // per line and lane of the newest plane: pressure (or the scalar) and y
  // velocity, tau_x, and tau_z two planes back
  __shared__ R s_p[NW][32], s_v[VEL ? NW : 1][32], s_tx[NW][32], s_tz[NW][32];
  // y-faces: what they give the cell below; the y-transverse scalar
  __shared__ R s_m[NS][NW][32], s_ay[NW][32];
  __shared__ LinK<R> K[3];
  __shared__ int s_done, s_cur, s_nbuf;
  const Member& mb = members[0];
  DevCtl* ctl = mb.ctl;
  pdl_enter();
  if (threadIdx.x < 3) LS::consts(C, threadIdx.x, dt_over_dx<R>(ctl, threadIdx.x), K[threadIdx.x]);
  if (threadIdx.x == 32) {
    s_done = ctl->done;
    s_cur = ctl->cur;
    s_nbuf = ctl->nbuf;
  }
  __syncthreads();
  if (s_done) return;
  const int nx = mb.nx, ny = mb.ny, nz = mb.nz;
  const Tile3 T = tile3d(blockIdx.x, nz, L);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // cells past the second ghost layer load that layer (no owner reads them)
  const int i = min(T.x0 - 2 + lane, nx + 1), j = min(T.y0 - 2 + w, ny + 1);
  const bool own = lane >= 2 && lane <= 29 && T.x0 - 2 + lane < nx && w >= 2 && w <= NW - 3 &&
                   T.y0 - 2 + w < ny;
  const bool row_in = w >= 1 && w <= NW - 2;   // lines whose tau_x, tau_z are read
  const bool row_own = w >= 2 && w <= NW - 3;
  const bool row_face = w >= 2 && w <= NW - 2;  // lines whose lower y-face is read
  const R* __restrict__ q = (const R*)mb.q[s_cur];
  R* __restrict__ qo = (R*)mb.q[(s_cur + 1) % s_nbuf];
  const size_t plane = (size_t)nx * ny, vol = plane * nz;
  // the thread's column remapped once (plain: an interior column)
  const bool plain = i >= 0 && i < nx && j >= 0 && j < ny;
  const size_t col = plain ? (size_t)j * nx + i : 0;
  auto load = [&](int k, R (&v)[M]) {
    if (plain && k >= 0 && k < nz) {
#pragma unroll
      for (int c = 0; c < M; ++c) v[c] = __ldg(q + c * vol + (size_t)k * plane + col);
    } else {
      load_cell3<M, R>(C, q, nx, ny, nz, i, j, k, RP::WALL_X, 2, 3, v);
    }
  };
  const int lim = C.lim;
  const int mode = FAST ? 2 : C.transverse;
  constexpr int U = VEL ? 1 : 0, V = VEL ? 2 : 0, Wc = VEL ? 3 : 0;

  // values of earlier planes: the state less its normal updates of planes
  // k-1, k-2; tau_x, tau_y (transverse form), the z-transverse scalar
  R acc1[M], acc2[M], tx1 = 0, tx2 = 0, tx3 = 0, ty1 = 0, ty2 = 0, ty3 = 0;
  R az1 = 0, az2 = 0, az3 = 0;
  // z-faces: strengths of faces k-1 and k-2, what face k-2 gives the cell above
  R zb1[NS], zb2[NS], zp2[NS], pz = 0, wz = 0;
#pragma unroll
  for (int c = 0; c < M; ++c) acc1[c] = acc2[c] = R(0);
#pragma unroll
  for (int s = 0; s < NS; ++s) zb1[s] = zb2[s] = zp2[s] = R(0);
  int bad = 0;
  R qn[M];
  load(T.z0 - 2, qn);
  for (int k = T.z0 - 2; k <= T.z1 + 1; ++k) {
    R acc0[M];
#pragma unroll
    for (int c = 0; c < M; ++c) acc0[c] = qn[c];
    if (k <= T.z1) load(k + 1, qn);
    const R p = acc0[0], u = acc0[U], v = acc0[V], wv = acc0[Wc];
    const bool xy = k >= T.z0 - 1 && k <= T.z1;  // planes whose tau_x, tau_y are read
    // x direction, plane k
    R tx = R(0), tz = R(0), zoz = R(0), tzT = R(0);
    if (row_in) {
      if (xy) {
        R b[NS], up[NS], fp[NS], fm[NS], mu[NS], zo;
        const R pl = __shfl_up_sync(FULL, p, 1), ul = VEL ? __shfl_up_sync(FULL, u, 1) : R(0);
        LS::strength(C, pl, ul, p, u, b);
#pragma unroll
        for (int s = 0; s < NS; ++s)
          up[s] = LS::upwind(K[0], s, __shfl_up_sync(FULL, b[s], 1),
                             __shfl_down_sync(FULL, b[s], 1));
        LS::template face<FAST>(K[0], lim, b, up, fp, fm);
#pragma unroll
        for (int s = 0; s < NS; ++s) mu[s] = __shfl_down_sync(FULL, fm[s], 1);
        LS::cell(fp, mu, tx, zo);
        acc0[0] -= tx;
        if (VEL) acc0[U] = LS::normal(K[0], acc0[U], zo);
        if (!FAST && mode == 1) {
          R bu[NS];
#pragma unroll
          for (int s = 0; s < NS; ++s) bu[s] = __shfl_down_sync(FULL, b[s], 1);
          tx = LS::plain(K[0], b, bu);
        }
      }
      // z direction: face k (cells k-1, k), limit face k-1, tau_z of cell k-2
      R zb[NS], up[NS], fp[NS], fm[NS];
      LS::strength(C, pz, wz, p, wv, zb);
#pragma unroll
      for (int s = 0; s < NS; ++s) up[s] = LS::upwind(K[2], s, zb2[s], zb[s]);
      LS::template face<FAST>(K[2], lim, zb1, up, fp, fm);
      LS::cell(zp2, fm, tz, zoz);
      tzT = (!FAST && mode == 1) ? LS::plain(K[2], zb2, zb1) : tz;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        zb2[s] = zb1[s];
        zb1[s] = zb[s];
        zp2[s] = fp[s];
      }
      pz = p;
      wz = wv;
    }
    s_p[w][lane] = p;
    if (VEL) s_v[w][lane] = v;
    if (mode) {
      s_tx[w][lane] = tx;
      s_tz[w][lane] = tzT;
    }
    __syncthreads();
    // y direction, plane k: the line's lower y-face
    R yp[NS], yT = R(0);
    if (row_face && xy) {
      R b[NS], bl[NS], bu[NS], up[NS], fm[NS];
      const R p1 = s_p[w - 1][lane], p2 = s_p[w - 2][lane], p3 = s_p[w + 1][lane];
      const R v1 = VEL ? s_v[w - 1][lane] : R(0), v2 = VEL ? s_v[w - 2][lane] : R(0),
              v3 = VEL ? s_v[w + 1][lane] : R(0);
      LS::strength(C, p2, v2, p1, v1, bl);
      LS::strength(C, p1, v1, p, v, b);
      LS::strength(C, p, v, p3, v3, bu);
#pragma unroll
      for (int s = 0; s < NS; ++s) up[s] = LS::upwind(K[1], s, bl[s], bu[s]);
      LS::template face<FAST>(K[1], lim, b, up, yp, fm);
#pragma unroll
      for (int s = 0; s < NS; ++s) s_m[s][w][lane] = fm[s];
      if (!FAST && mode == 1) yT = LS::plain(K[1], b, bu);
    }
    R axz = R(0), azx = R(0);
    if (mode && row_in) {
      // scalars A_dg: (d, g) = (x, z) of plane k and (z, x), (z, y), (x, y) of k-2
      if (row_own) {
        axz = LS::second(K[1], tx, s_tx[w - 1][lane], s_tx[w + 1][lane]);
        azx = LS::second(K[1], tzT, s_tz[w - 1][lane], s_tz[w + 1][lane]);
      }
      const R lo = __shfl_up_sync(FULL, tzT, 1), hi = __shfl_down_sync(FULL, tzT, 1);
      s_ay[w][lane] = LS::second(K[0], tzT, lo, hi) + LS::second(K[2], tx2, tx3, tx1);
    }
    __syncthreads();
    R ty = R(0), az = R(0);
    if (row_own) {
      if (xy) {
        R mu[NS], zo;
#pragma unroll
        for (int s = 0; s < NS; ++s) mu[s] = s_m[s][w + 1][lane];
        LS::cell(yp, mu, ty, zo);
        acc0[0] -= ty;
        if (VEL) acc0[V] = LS::normal(K[1], acc0[V], zo);
        if (!FAST && mode == 1) ty = yT;
      }
      const int r = k - 2;
      R out[M];
#pragma unroll
      for (int c = 0; c < M; ++c) out[c] = acc2[c];
      out[0] -= tz;
      if (VEL) out[Wc] = LS::normal(K[2], out[Wc], zoz);
      if (mode) {
        // (y, z) of plane k; (y, x) of plane k-2
        const R lo = __shfl_up_sync(FULL, ty, 1), hi = __shfl_down_sync(FULL, ty, 1);
        az = axz + LS::second(K[0], ty, lo, hi);
        const R ax = azx + LS::second(K[2], ty2, ty3, ty1);
        const R xl = __shfl_up_sync(FULL, ax, 1), xh = __shfl_down_sync(FULL, ax, 1);
        LS::apply(K[0], ax, xl, xh, out[0], out[U]);
        LS::apply(K[1], s_ay[w][lane], s_ay[w - 1][lane], s_ay[w + 1][lane], out[0], out[V]);
        LS::apply(K[2], az2, az3, az1, out[0], out[Wc]);
      }
      if (own && r >= T.z0) {
        const size_t off = (size_t)r * plane + col;
#pragma unroll
        for (int c = 0; c < M; ++c) {
          bad |= not_finite(out[c]);
          qo[c * vol + off] = out[c];
        }
      }
    }
    tx3 = tx2;
    tx2 = tx1;
    tx1 = tx;
    ty3 = ty2;
    ty2 = ty1;
    ty1 = ty;
    az3 = az2;
    az2 = az1;
    az1 = az;
#pragma unroll
    for (int c = 0; c < M; ++c) {
      acc2[c] = acc1[c];
      acc1[c] = acc0[c];
    }
  }
  finish_attempt<R>(ctl, LS::speed(C, 0), LS::speed(C, 1), bad, mb.ntiles, true, LS::speed(C, 2));
}

template <class RP, typename R>
__global__ void __launch_bounds__(256)
    maxspeed3_kernel(const Member* __restrict__ members, const MConsts<R> C) {
  constexpr int M = RP::M, MW = RP::MW;
  const Member& mb = members[0];
  DevCtl* ctl = mb.ctl;
  const int nx = mb.nx, ny = mb.ny, nz = mb.nz;
  const long long ncell = (long long)nx * ny * nz;
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  R sm[3] = {R(0), R(0), R(0)};
  if (id < ncell) {
    const int i = (int)(id % nx), j = (int)((id / nx) % ny), k = (int)(id / ((long long)nx * ny));
    const R* q = (const R*)mb.q[ctl->cur];
    const int c3[3] = {i, j, k};
    const int n3[3] = {nx, ny, nz};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      for (int side = 0; side < (c3[d] == n3[d] - 1 ? 2 : 1); ++side) {
        int l[3] = {i, j, k}, r[3] = {i, j, k};
        l[d] += side - 1;
        r[d] += side;
        R a[M], b[M], W[MW][M], s[MW], am[M], ap[M], x[RP::NCTX];
        load_cell3<M, R>(C, q, nx, ny, nz, l[0], l[1], l[2], RP::WALL_X, 2, 3, a);
        load_cell3<M, R>(C, q, nx, ny, nz, r[0], r[1], r[2], RP::WALL_X, 2, 3, b);
        if (d == 0) RP::template solve<0>(C, a, b, nullptr, nullptr, W, s, am, ap, x);
        else if (d == 1) RP::template solve<1>(C, a, b, nullptr, nullptr, W, s, am, ap, x);
        else RP::template solve<2>(C, a, b, nullptr, nullptr, W, s, am, ap, x);
#pragma unroll
        for (int p = 0; p < MW; ++p) sm[d] = nanmax(sm[d], (R)fabs(s[p]));
      }
    }
  }
  finish_attempt<R>(ctl, sm[0], sm[1], 0, 0, false, sm[2]);
}

}  // namespace claw
