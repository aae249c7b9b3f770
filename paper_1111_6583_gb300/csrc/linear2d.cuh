// linear2d.cuh -- the 2D classic step of the constant-coefficient linear
// systems (advection, acoustics) in strength form (linear.cuh), one launch per
// attempt (two for a dimensionally split step).
//
// A warp owns a strip of columns (one, two or four per lane, two halo columns
// on each side; reg_tile) and walks a chunk of rows: x neighbours are the
// lane's own columns or come by warp shuffles, y neighbours are the lane's
// values of earlier rows, so there is no shared-memory exchange and no
// barrier in the walk.  With row R loaded the warp has tau_x of row R, tau_y of row R - 2
// and finishes row R - 2.  Products and sums are written as explicit fused
// multiply-adds, so every strip width and chunk height gives the same bits.
//
// What bounds it: FP64 the FP64 pipe (67 % on average at 1000 x 750 in one
// wave of two-column warps; about 45 FP64 instructions per column and row
// against some 250 of the vector form); FP32 issue and latency (53 % issue at
// 4096 x 3072, 154 registers), small grids the latency of an attempt.
// Acoustics 1000 x 750 FP64 368 -> 122 us/step, 64^2 FP64 63 -> 28 us, 700 x
// 650 FP64 superbee 231 -> 83 us, 1024^2 FP32 38.6 -> 26.2 us against the
// shared-memory row walk of classic2d_kernel.  Rows collect increments and add
// them to the state once (errors as the row walk's; updating the state term by
// term cost 12 to 22 % more error and saved 5 % of the time).
#pragma once

#include "kernels.h"
#include "linear.cuh"

namespace claw {

// two consecutive values (8-byte aligned FP32, 16-byte aligned FP64)
__device__ __forceinline__ void ld2(const float* p, float& a, float& b) {
  const float2 t = __ldg((const float2*)p);
  a = t.x;
  b = t.y;
}
__device__ __forceinline__ void ld2(const double* p, double& a, double& b) {
  const double2 t = __ldg((const double2*)p);
  a = t.x;
  b = t.y;
}
__device__ __forceinline__ void st2(float* p, float a, float b) { *(float2*)p = make_float2(a, b); }
__device__ __forceinline__ void st2(double* p, double a, double b) {
  *(double2*)p = make_double2(a, b);
}

// one column or a pair of a row
template <int N, typename R>
__device__ __forceinline__ void ld_pair(const R* p, bool vec, R& a, R& b) {
  if (N > 1 && vec) {
    ld2(p, a, b);
  } else {
    a = __ldg(p);
    if (N > 1) b = __ldg(p + 1);
  }
}
template <typename R>
__device__ __forceinline__ void st_pair(R* p, bool two, bool vec, R a, R b) {
  if (two && vec) {
    st2(p, a, b);
  } else {
    p[0] = a;
    if (two) p[1] = b;
  }
}

// sweep: 0 the unsplit step (slot 0 -> 1); dimensional splitting: 1 the x
// sweeps (slot 0 -> 1), 2 the y sweeps (slot 1 -> 2).  FAST: the MC limiter,
// second order and transverse mode 2 fixed at compile time.
template <class RP, typename R, int BW, bool FAST>
__global__ void __launch_bounds__(32 * reg_tile(sizeof(R) == 8 ? 0 : 1, BW).warps)
    linear2d_kernel(const Member* __restrict__ members, const Tile* __restrict__ tiles,
                    const MConsts<R> C, int H, int sweep) {
  using LS = Lin<RP, R>;
  constexpr RegTile RT = reg_tile(sizeof(R) == 8 ? 0 : 1, BW);
  constexpr int M = RP::M, NS = LS::NS, N = RT.n, WL = 32 * N;  // columns per lane, per warp
  constexpr bool VEL = LS::VEL;
  constexpr int U = VEL ? 1 : 0, V = VEL ? 2 : 0;
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ LinK<R> K[2], T[2];
  const Tile tl = tiles ? tiles[blockIdx.x] : Tile{0, (int)blockIdx.x};
  const Member& mb = members[tl.member];
  DevCtl* ctl = mb.ctl;
  pdl_enter();  // (the tables above do not change between attempts)
  if (ctl->done) return;  // the whole block
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 2) {
    LS::consts(C, lane, dt_over_dx<R>(ctl, lane), K[lane]);
    T[lane] = K[lane];  // transverse terms act on -tau/2
    T[lane].t0 *= R(-0.5);
    T[lane].t1 *= R(-0.5);
  }
  __syncthreads();
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
  const size_t plane = (size_t)nx * ny;
  // the lane's columns g0 .. g0 + N - 1; columns past the second ghost column
  // load that column (nothing reads them)
  const int g0 = c0 - 2 + N * lane;
  const bool inner = g0 >= 0 && g0 + N <= nx;
  // pairs of columns start on even columns: aligned when the rows are
  const bool vec = (nx & 1) == 0 && (((size_t)q | (size_t)qo) & (2 * sizeof(R) - 1)) == 0;
  auto load = [&](int r, R (&v)[N][M]) {
    if (inner && r >= 0 && r < ny) {
      const R* p = q + (size_t)r * nx + g0;
#pragma unroll
      for (int k = 0; k < M; ++k) {
#pragma unroll
        for (int c = 0; c < N; c += 2)
          ld_pair<N>(p + k * plane + c, vec, v[c][k], v[c + (N > 1)][k]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < N; ++c)
        load_cell<M, R>(C, q, nx, ny, min(g0 + c, nx + 1), r, RP::WALL_X, RP::WALL_Y, v[c]);
    }
  };

  // per column: the increments of rows R-1, R-2 so far (added to the state once,
  // when the row is finished, so that they round at their own size); tau_x of rows
  // R-1 .. R-3; y-face strengths of faces R-1, R-2, what face R-2 gives the
  // cell above it; (p, v) of row R-1
  R q1[N][M], q2[N][M], acc1[N][M], acc2[N][M], tx1[N], tx2[N], tx3[N], zb1[N][NS], zb2[N][NS], zp2[N][NS];
  R pz[N], vz[N];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    tx1[c] = tx2[c] = tx3[c] = pz[c] = vz[c] = R(0);
#pragma unroll
    for (int k = 0; k < M; ++k) acc1[c][k] = acc2[c][k] = q1[c][k] = q2[c][k] = R(0);
#pragma unroll
    for (int s = 0; s < NS; ++s) zb1[c][s] = zb2[c][s] = zp2[c][s] = R(0);
  }
  int bad = 0;
  R qn[N][M];
  if (c0 < nx) load(r0 - 2, qn);
  // (a warp whose strip starts past the grid has nothing to do)
  for (int r = c0 < nx ? r0 - 2 : r1 + 2; r <= r1 + 1; ++r) {
    R q0[N][M], acc0[N][M], tx[N], ty[N], zo[N];
#pragma unroll
    for (int c = 0; c < N; ++c) {
#pragma unroll
      for (int k = 0; k < M; ++k) {
        q0[c][k] = qn[c][k];
        acc0[c][k] = R(0);
      }
      tx[c] = ty[c] = zo[c] = R(0);
    }
    if (r <= r1) load(r + 1, qn);
    // y direction: face r (rows r-1, r), limit face r-1, tau_y of row r-2
    if (doy) {
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const R p = q0[c][0], v = q0[c][V];
        R zb[NS], up[NS], fp[NS], fm[NS];
        LS::strength(C, pz[c], vz[c], p, v, zb);
#pragma unroll
        for (int s = 0; s < NS; ++s) up[s] = LS::upwind(K[1], s, zb2[c][s], zb[s]);
        LS::template face<FAST>(K[1], lim, zb1[c], up, fp, fm);
        LS::cell(zp2[c], fm, ty[c], zo[c]);
        acc2[c][0] -= ty[c];
        if (VEL) acc2[c][V] = LS::normal(K[1], acc2[c][V], zo[c]);
        if (!FAST && mode == 1) ty[c] = LS::plain(K[1], zb2[c], zb1[c]);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          zb2[c][s] = zb1[c][s];
          zb1[c][s] = zb[s];
          zp2[c][s] = fp[s];
        }
        pz[c] = p;
        vz[c] = v;
      }
    }
    // x direction, row r
    if (dox && r >= r0 - 1 && r <= r1) {
      R b[N][NS], fp[N][NS], fm[N + 1][NS], bl[NS], bu[NS];
      {
        const R pl = __shfl_up_sync(FULL, q0[N - 1][0], 1);
        const R ul = VEL ? __shfl_up_sync(FULL, q0[N - 1][U], 1) : R(0);
        LS::strength(C, pl, ul, q0[0][0], q0[0][U], b[0]);
      }
#pragma unroll
      for (int c = 1; c < N; ++c)
        LS::strength(C, q0[c - 1][0], q0[c - 1][U], q0[c][0], q0[c][U], b[c]);
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        bl[s] = __shfl_up_sync(FULL, b[N - 1][s], 1);
        bu[s] = __shfl_down_sync(FULL, b[0][s], 1);
      }
#pragma unroll
      for (int c = 0; c < N; ++c) {
        R up[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s)
          up[s] = LS::upwind(K[0], s, c == 0 ? bl[s] : b[c > 0 ? c - 1 : 0][s],
                             c == N - 1 ? bu[s] : b[c < N - 1 ? c + 1 : 0][s]);
        LS::template face<FAST>(K[0], lim, b[c], up, fp[c], fm[c]);
      }
#pragma unroll
      for (int s = 0; s < NS; ++s) fm[N][s] = __shfl_down_sync(FULL, fm[0][s], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        R z;
        LS::cell(fp[c], fm[c + 1], tx[c], z);
        acc0[c][0] = -tx[c];
        if (VEL) acc0[c][U] = LS::normal(K[0], R(0), z);
        if (!FAST && mode == 1) tx[c] = LS::plain(K[0], b[c], c == N - 1 ? bu : b[c < N - 1 ? c + 1 : 0]);
      }
    }
    // transverse terms and the finished row r - 2
    if (mode) {
      const R tl_ = __shfl_up_sync(FULL, ty[N - 1], 1), tr_ = __shfl_down_sync(FULL, ty[0], 1);
#pragma unroll
      for (int c = 0; c < N; ++c) {
        LS::apply(T[0], ty[c], c == 0 ? tl_ : ty[c > 0 ? c - 1 : 0],
                  c == N - 1 ? tr_ : ty[c < N - 1 ? c + 1 : 0], acc2[c][0], acc2[c][U]);
        LS::apply(T[1], tx2[c], tx3[c], tx1[c], acc2[c][0], acc2[c][V]);
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
      tx3[c] = tx2[c];
      tx2[c] = tx1[c];
      tx1[c] = tx[c];
#pragma unroll
      for (int k = 0; k < M; ++k) {
        acc2[c][k] = acc1[c][k];
        acc1[c][k] = acc0[c][k];
        q2[c][k] = q1[c][k];
        q1[c][k] = q0[c][k];
      }
    }
  }
  finish_attempt<R>(ctl, dox ? LS::speed(C, 0) : R(0), doy ? LS::speed(C, 1) : R(0), bad, mb.ntiles,
                    sweep != 1);
}

}  // namespace claw
