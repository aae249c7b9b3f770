// sharpclaw.cuh -- fused SharpClaw stage kernel (Sec. 2 method of lines;
// Sec. 2.1: WENO reconstruction, normal Riemann problems only in multi-D).
//
// One launch = one Runge-Kutta stage for every member of a tile table.  A
// block stages a TX x TY tile of Q^(k) plus an RW-cell halo (ghost remap in
// the load), reconstructs left/right interface values by WENO of order
// 2 RW - 1 (component- or
// characteristic-wise, projection at the Roe state of each interface), solves
// the interface Riemann problems and the in-cell problems (total fluctuation
// A dQ_i), forms L(Q) = -(A^+dQ_{i-1/2} + A^-dQ_{i+1/2} + A dQ_i)/dx summed
// over directions, and writes the stage's linear combinations (StageOp: the
// Shu-Osher SSP-RK3 or the low-storage SSP(10,4) stages).  The last stage's
// last block runs the CFL controller.
#pragma once

#include <type_traits>

#include "async_copy.cuh"
#include "kernels.h"
#include "riemann.cuh"
#include "vec.cuh"
#include "weno_hi.cuh"

namespace claw {

// Both Jiang-Shu WENO5 values at the interface between cells c and d of six
// cell averages a .. f, from their five first differences D: the left-biased
// value at the right edge of c is c + nl / dl, the right-biased one at the
// left edge of d is d - nr / dr.  The two share the candidates and second
// differences of the stencils (b, c, d) and (c, d, e).  Differences in place
// of averages take fewer operations (58 against 86 per pair) and cancel once,
// before the products.  Smoothness indicators are kept times 4 (eps4 = 4 eps)
// and candidates times 6 (the 6 moves to the denominator).
template <typename V, typename R>
__device__ __forceinline__ void weno5_diff(const V (&D)[5], R eps4, V& nl, V& dl, V& nr, V& dr) {
  const V two = V(R(2)), mtwo = V(R(-2)), k13 = V(R(13) / R(3)), e4 = V(eps4);
  const V t0 = vsub(D[1], D[0]), t1 = vsub(D[2], D[1]), t2 = vsub(D[3], D[2]),
          t3 = vsub(D[4], D[3]);
  const V h0 = vfma(vmul(k13, t0), t0, e4), h1 = vfma(vmul(k13, t1), t1, e4),
          h2 = vfma(vmul(k13, t2), t2, e4), h3 = vfma(vmul(k13, t3), t3, e4);
  const V u0 = vfma(two, D[1], t0), u1 = vadd(D[1], D[2]), u2 = vfma(mtwo, D[2], t2);
  const V v0 = vfma(mtwo, D[3], t3), v1 = vadd(D[2], D[3]), v2 = vfma(two, D[2], t1);
  const V e0 = vfma(u0, u0, h0), e1 = vfma(u1, u1, h1), e2 = vfma(u2, u2, h2);
  const V g0 = vfma(v0, v0, h3), g1 = vfma(v1, v1, h2), g2 = vfma(v2, v2, h1);
  // weights d_k / beta_k^2 (1/10, 6/10, 3/10) times the product of the three
  auto side = [&](V e0, V e1, V e2, V p0, V p1, V p2, V& n, V& d) {
    const V s1 = vmul(e1, e1), s2 = vmul(e2, e2), a = vmul(vmul(V(R(3)), e0), e0);
    const V s12 = vmul(s1, s2), b = vadd(s2, s2);
    n = vfma(a, vfma(b, p1, vmul(s1, p2)), vmul(s12, p0));
    d = vmul(V(R(6)), vfma(a, vadd(b, s1), s12));
  };
  const V five = V(R(5)), four = V(R(4)), mone = V(R(-1));
  side(e0, e1, e2, vfma(five, D[1], vmul(mtwo, D[0])), vfma(two, D[2], D[1]),
       vfma(four, D[2], vmul(mone, D[3])), nl, dl);
  side(g0, g1, g2, vfma(five, D[3], vmul(mtwo, D[4])), vfma(two, D[2], D[3]),
       vfma(four, D[2], vmul(mone, D[1])), nr, dr);
}

// n / d for N pairs.  FP64: the reciprocals from the hardware seed and one
// step of Halley's iteration (x y = 1 - e: y (1 + e + e^2), error e^3 of a
// seed good to 20 bits, so correct to about one rounding: three FP64
// instructions against about eight of a division), taken only when every
// divisor is well inside the normal range, else N divisions.
template <typename R, int N>
__device__ __forceinline__ void div_many(const R (&n)[N], const R (&d)[N], R (&q)[N]) {
  if constexpr (sizeof(R) == 8) {
    bool normal = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
      normal = normal && (unsigned)(__double2hiint(d[i]) - 0x10000000) < 0x60000000u;
    if (normal) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d[i]));
        const double e = fma(-d[i], y, 1.0);
        q[i] = n[i] * fma(y, fma(e, e, e), y);
      }
      return;
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) q[i] = FM<R>::div(n[i], d[i]);
}

// the WENO5 pairs of M fields from their differences w[field][5]: corrections
// to the average of the cell on each side (um: add to c, up: subtract from d)
template <typename R, int M>
__device__ __forceinline__ void weno5_fields(const R (&w)[M][5], R eps, R (&um)[M], R (&up)[M]) {
  R nn[2 * M], dd[2 * M], vv[2 * M];
  const R eps4 = R(4) * eps;
  if constexpr (sizeof(R) == 4) {
    // two fields per packed instruction (an odd last field alone)
#pragma unroll
    for (int k = 0; k + 1 < M; k += 2) {
      F2 D[5], a, b, c, d;
#pragma unroll
      for (int j = 0; j < 5; ++j) D[j] = F2(w[k][j], w[k + 1][j]);
      weno5_diff<F2, float>(D, eps4, a, b, c, d);
      a.get(nn[k], nn[k + 1]);
      b.get(dd[k], dd[k + 1]);
      c.get(nn[M + k], nn[M + k + 1]);
      d.get(dd[M + k], dd[M + k + 1]);
    }
    if constexpr (M % 2 == 1)
      weno5_diff<R, R>(w[M - 1], eps4, nn[M - 1], dd[M - 1], nn[2 * M - 1], dd[2 * M - 1]);
  } else {
#pragma unroll
    for (int k = 0; k < M; ++k)
      weno5_diff<R, R>(w[k], eps4, nn[k], dd[k], nn[M + k], dd[M + k]);
  }
  div_many<R, 2 * M>(nn, dd, vv);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    um[k] = vv[k];
    up[k] = vv[M + k];
  }
}

// WENO of order 2 RW - 1 (7 .. 17; WENO5 takes weno5_diff): left-biased value at the right edge of cell
// v[o + RW - 1] from v[o .. o + 2 RW - 2] (REV: the mirrored stencil, value at
// the left edge of cell v[o + RW], read from v[o + 2 RW - 1] downwards).
template <int RW, bool REV, typename R, int NV>
__device__ __forceinline__ R weno_edge(const R (&w)[NV], R eps) {
  constexpr int n = 2 * RW - 1;
  R v[n];
#pragma unroll
  for (int j = 0; j < n; ++j) v[j] = REV ? w[n - j] : w[j];
  if constexpr (RW == 4) return weno7<R>(v, eps);
  else if constexpr (RW == 5) return weno9<R>(v, eps);
  else if constexpr (RW == 6) return weno11<R>(v, eps);
  else if constexpr (RW == 7) return weno13<R>(v, eps);
  else if constexpr (RW == 8) return weno15<R>(v, eps);
  else return weno17<R>(v, eps);
}

// Resident blocks the registers are held to (0: the compiler's choice).  The
// FP32 WENO5 stage waits on its tile loads and barriers, and more warps pay
// for the few spills: with four 256-thread blocks per SM (64 registers)
// 1500 x 700 shock-bubble 270 us/step, three or five 295, left to the compiler
// (80 registers) 310; six 128-thread blocks (80 registers) suit small grids.
template <typename R, int TX, int TY, int RW>
__host__ __device__ constexpr int sharp_minb() {
  return sizeof(R) == 4 && RW == 3 && TY > 1 ? (TX * TY == 256 ? 4 : 6) : 0;
}
// Values of the interfaces' Roe averages kept per cell.  FP64: they save some
// 30 of 560 FP64 instructions per interface; FP32: forming them at each
// interface is cheaper than another barrier and its shared memory (270 against
// 280 us/step).
template <class RP, typename R, int RW>
__host__ __device__ constexpr int sharp_ncp() {
  return RW == 3 && sizeof(R) == 8 ? char_prep_n<RP>() : 0;
}

// static shared memory of sharp_stage_kernel (the arrays declared in it)
template <class RP, typename R, int ND, int TX, int TY, int RW>
constexpr size_t sharp_smem_bytes() {
  constexpr int M = RP::M, MA = RP::MA, G = RW;
  constexpr int MAS = MA > 0 ? MA : 1;
  constexpr int HX = TX + 2 * G, HY = (ND == 2) ? TY + 2 * G : 1;
  constexpr bool kStageRows = TX * TY <= 128;
  constexpr int A = 16 / (int)sizeof(R), OX = kStageRows ? (A - G % A) % A : 0;
  constexpr int HXP0 = (OX + HX + A - 1) / A * A;
  constexpr int HXP = !kStageRows ? HX : ((HXP0 / A) % 2 == 1 ? HXP0 : HXP0 + A);
  constexpr int NE = (ND == 2) ? (TX + 1) * TY + TX * (TY + 1) : TX + 1;
  constexpr int NCP = sharp_ncp<RP, R, RW>();
  return sizeof(R) * ((size_t)M * HY * HXP + (size_t)MAS * (MA > 0 ? HY * HXP : 1) +
                      (size_t)HY * HX + (size_t)(NCP > 0 ? NCP * HY * HX : 1) +
                      4 * (size_t)M * NE + 3) +
         3 * sizeof(int) + 8;
}

template <class RP, typename R, int ND, int TX, int TY, int RW>
__global__ void __launch_bounds__(TX * TY, sharp_minb<R, TX, TY, RW>())
    sharp_stage_kernel(const Member* __restrict__ members, const Tile* __restrict__ tiles,
                       int ntiles_total, const MConsts<R> C, const StageOp op) {
  constexpr int M = RP::M, MW = RP::MW, MA = RP::MA, NC = RP::NCTX;
  constexpr int MAS = MA > 0 ? MA : 1;
  constexpr int NT = TX * TY;
  constexpr int G = RW;        // ghost / halo width
  constexpr int NS = 2 * RW;   // cells around an interface
  constexpr int HX = TX + 2 * G, HY = (ND == 2) ? TY + 2 * G : 1;
  // interface slots: the x-interfaces (TX + 1 per row) first, then the
  // y-interfaces (TY + 1 per column)
  constexpr int NEX = (ND == 2) ? (TX + 1) * TY : TX + 1;
  constexpr int NEY = (ND == 2) ? TX * (TY + 1) : 0;
  constexpr int NE = NEX + NEY;
  // staged rows: a tile row of a field is HXP values from the 16-byte
  // boundary at or below the halo's first cell; cell hi of the halo sits at
  // column OX + hi (tiles start at multiples of TX, a multiple of A)
  // Staged rows, for tiles of 128 threads or fewer (with 256-thread tiles
  // the staging state spilled and the copies measured slower than the
  // cell-by-cell loads in FP32: 0.64-0.71 against 0.61 ms per shock-bubble
  // step); rows padded to an odd number of 16-byte units, so that a column
  // of cells spreads over the shared-memory banks (the y-interface phase
  // reads down columns).  Without staging the rows are HX values, OX = 0.
  constexpr bool kStageRows = TX * TY <= 128;
  constexpr int A = 16 / (int)sizeof(R), OX = kStageRows ? (A - G % A) % A : 0;
  constexpr int HXP0 = (OX + HX + A - 1) / A * A;
  constexpr int HXP = !kStageRows ? HX : ((HXP0 / A) % 2 == 1 ? HXP0 : HXP0 + A);
  static_assert(!kStageRows || TX % A == 0, "tile columns start on 16-byte boundaries");
  __shared__ __align__(16) R Qt[M][HY][HXP];
  __shared__ __align__(16) R At[MAS][MA > 0 ? HY : 1][MA > 0 ? HXP : 1];
  __shared__ __align__(8) unsigned long long s_bar;  // completes the staging copies
  __shared__ R Kt[HY][HX];  // capacity kappa (when the method has one)
  // per-cell part of the interfaces' Roe averages (WENO5, characteristic form)
  constexpr int NCP = sharp_ncp<RP, R, RW>(), NCPS = NCP > 0 ? NCP : 1;
  __shared__ R Pc[NCPS][NCP > 0 ? HY : 1][NCP > 0 ? HX : 1];
  __shared__ R EL[M][NE];  // left edge value of the cell right of an interface
  __shared__ R ER[M][NE];  // right edge value of the cell left of an interface
  __shared__ R FM[M][NE];  // A^- dQ at the interface
  __shared__ R FP[M][NE];  // A^+ dQ at the interface
  __shared__ int s_done, s_cur, s_nbuf;
  __shared__ R s_dt, s_idn[2];

  const int tid = threadIdx.x;
  const int ti = tid % TX, tj = tid / TX;
  [[maybe_unused]] unsigned phase = 0u;  // parity of the staging barrier's phase
  if constexpr (kStageRows) {
    if (tid == 0) {
      mbar_init(smem_u32(&s_bar), 1u);
      fence_mbar_init();
    }
  }

  pdl_enter();
  for (int it = blockIdx.x; it < ntiles_total; it += gridDim.x) {
    const Tile tl = tiles ? tiles[it] : Tile{0, it};
    const Member& mb = members[tl.member];
    DevCtl* ctl = mb.ctl;
    if (tid == 0) {
      s_done = ctl->done;
      s_dt = (R)ctl->dt;
      s_idn[0] = (R)ctl->idx[0];  // 1/dx, divided once on the host
      s_idn[1] = (R)ctl->idx[1];
      s_cur = ctl->cur;
      s_nbuf = ctl->nbuf;
    }
    __syncthreads();
    if (s_done) {
      __syncthreads();
      continue;
    }
    const int nx = mb.nx, ny = (ND == 2) ? mb.ny : 1;
    const int nsx = (nx + TX - 1) / TX;
    const int c0 = (tl.tile % nsx) * TX;
    const int r0 = (ND == 2) ? (tl.tile / nsx) * TY : 0;
    const int cur = s_cur;
    const int nb = s_nbuf;
    const R* __restrict__ qk = (const R*)step_input(mb, cur, nb, op.in);
    const R* __restrict__ qa = (const R*)step_input(mb, cur, nb, op.sa);
    const R* __restrict__ qb = (const R*)step_input(mb, cur, nb, op.sb);
    R* __restrict__ qo = (R*)mb.q[(cur + op.out) % nb];
    R* __restrict__ qo2 = op.out2 >= 0 ? (R*)mb.q[(cur + op.out2) % nb] : nullptr;
    const R* __restrict__ aux = (const R*)mb.aux;
    const size_t plane = (size_t)nx * ny;

    // stage Q^(k) (and aux) with a G-cell halo.  A tile whose halo rows lie
    // inside the grid, with 16-byte aligned fields and rows, arrives by
    // bulk asynchronous copies, one per row and field (HXP values each, the
    // corners and the padding included), completing on the block's
    // barrier; the others (and methods with a capacity field) are loaded
    // cell by cell with the ghost-cell remap, corners skipped in 2D.
    int bad = 0;
    const int xa = c0 - G - OX;  // first staged column
    bool staged = false;
    if constexpr (kStageRows)
      staged = C.capa < 0 && xa >= 0 && xa + HXP <= nx &&
               (ND == 1 || (r0 - G >= 0 && r0 + TY + G <= ny)) &&
               ((size_t)nx * sizeof(R)) % 16 == 0 && ((size_t)qk & 15) == 0 &&
               (MA == 0 || ((size_t)aux & 15) == 0);
    if (staged) {
      const unsigned bar = smem_u32(&s_bar);
      constexpr int NCP = (M + MA) * HY;
      constexpr unsigned RB = HXP * sizeof(R);
      if (tid == 0) mbar_arrive_expect_tx(bar, NCP * RB);
      // a block's later tile refills rows that its previous tile read
      // (those reads precede the barriers of finish_attempt)
      if (it != (int)blockIdx.x && tid < NCP) fence_proxy_async_smem();
      for (int cp = tid; cp < NCP; cp += NT) {
        const int f = cp / HY, hj = cp % HY;
        const int r = (ND == 2) ? r0 - G + hj : 0;
        const R* src = f < M ? qk + (size_t)f * plane + (size_t)r * nx + xa
                             : aux + (size_t)(f - M) * plane + (size_t)r * nx + xa;
        R* dst = f < M ? &Qt[f][hj][0] : &At[MA > 0 ? f - M : 0][MA > 0 ? hj : 0][0];
        bulk_g2s(smem_u32(dst), src, RB, bar);
      }
      const bool got = mbar_wait_bounded(bar, phase);
      if (__syncthreads_or(!got)) {
        // a copy did not complete in time: wait (bounded) for the rest,
        // report CLAW_ETIMEOUT through the control block, compute nothing
        mbar_wait_bounded(bar, phase);
        bad = 2;
      }
      phase ^= 1u;
    } else {
      for (int idx = tid; idx < HX * HY; idx += NT) {
        const int hi = idx % HX, hj = idx / HX;
        if (ND == 2) {
          const bool xin = hi >= G && hi < G + TX, yin = hj >= G && hj < G + TY;
          if (!xin && !yin) continue;
        }
        const int c = c0 - G + hi, r = (ND == 2) ? r0 - G + hj : 0;
        R v[M];
        load_cell<M, R>(C, qk, nx, ny, min(c, nx + G - 1), (ND == 2) ? min(r, ny + G - 1) : 0,
                        RP::WALL_X, RP::WALL_Y, v);
#pragma unroll
        for (int k = 0; k < M; ++k) Qt[k][hj][OX + hi] = v[k];
        if (MA > 0) {
          R a[MAS];
          load_aux<MA, R>(C, aux, nx, ny, min(c, nx + G - 1),
                          (ND == 2) ? min(r, ny + G - 1) : 0, a);
#pragma unroll
          for (int k = 0; k < MA; ++k) At[k][MA > 0 ? hj : 0][MA > 0 ? OX + hi : 0] = a[k];
        }
        if (C.capa >= 0)
          Kt[hj][hi] = load_aux_field<R>(C, aux, nx, ny, min(c, nx + G - 1),
                                         (ND == 2) ? min(r, ny + G - 1) : 0, C.capa);
      }
      __syncthreads();
    }
    const bool skip = bad != 0;
    if constexpr (NCP > 0) {
      if (C.char_decomp) {
        // the cells beside an interface: one more than the tile on each side
        constexpr int WX = TX + 2, WY = (ND == 2) ? TY + 2 : 1;
        for (int idx = tid; idx < WX * WY; idx += NT) {
          const int hi = G - 1 + idx % WX, hj = (ND == 2) ? G - 1 + idx / WX : 0;
          const bool xin = hi >= G && hi < G + TX, yin = ND == 1 || (hj >= G && hj < G + TY);
          if (!xin && !yin) continue;  // corners (not loaded cell by cell)
          R v[M], p[NCPS];
#pragma unroll
          for (int k = 0; k < M; ++k) v[k] = Qt[k][hj][OX + hi];
          RP::char_prep(C, v, p);
#pragma unroll
          for (int k = 0; k < NCP; ++k) Pc[k][hj][hi] = p[k];
        }
        __syncthreads();
      }
    }

    R L[M];
#pragma unroll
    for (int k = 0; k < M; ++k) L[k] = R(0);
    R smx = R(0), smy = R(0);

    // (a, b) every interface of both directions, each by one thread:
    // reconstruction of its two edge values, then its Riemann problem
    // (q^R_{a-1}, q^L_a) from the same thread's edge values
    auto interface = [&](auto dirc, int le, int e) {
      constexpr int dir = decltype(dirc)::value;
      const int na = (dir == 0) ? TX + 1 : TY + 1;
      const int a = le % na, b = le / na;
      R cell[NS][M];
#pragma unroll
      for (int k6 = 0; k6 < NS; ++k6) {
        // cells a-RW .. a+RW-1 along the line
        const int hi = (dir == 0) ? a + k6 : G + b;
        const int hj = (dir == 0) ? ((ND == 2) ? G + b : 0) : a + k6;
#pragma unroll
        for (int k = 0; k < M; ++k) cell[k6][k] = Qt[k][hj][OX + hi];
      }
      R wm[M], wp[M];
      if constexpr (RW == 3) {
        // WENO5 on the differences of the six cells (of their characteristic
        // components: the projection is linear); corrections to the two cells
        R df[5][M], w[M][5], um[M], up[M];
#pragma unroll
        for (int k6 = 0; k6 < 5; ++k6)
#pragma unroll
          for (int k = 0; k < M; ++k) df[k6][k] = cell[k6 + 1][k] - cell[k6][k];
        if (C.char_decomp) {
          R x[NC];
          if constexpr (NCP > 0) {
            const int hil = (dir == 0) ? G + a - 1 : G + b, hir = (dir == 0) ? G + a : G + b;
            const int hjl = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a - 1;
            const int hjr = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a;
            R pl[NCPS], pr[NCPS];
#pragma unroll
            for (int k = 0; k < NCP; ++k) {
              pl[k] = Pc[k][hjl][hil];
              pr[k] = Pc[k][hjr][hir];
            }
            RP::template char_ctx_pc<dir>(C, cell[RW - 1], cell[RW], pl, pr, x);
          } else {
            RP::template char_ctx<dir>(C, cell[RW - 1], cell[RW], x);
          }
#pragma unroll
          for (int k6 = 0; k6 < 5; ++k6) {
            R v[M];
            RP::template to_char<dir>(C, x, df[k6], v);
#pragma unroll
            for (int k = 0; k < M; ++k) w[k][k6] = v[k];
          }
          weno5_fields<R, M>(w, C.weno_eps, um, up);
          RP::template from_char<dir>(C, x, um, wm);
          RP::template from_char<dir>(C, x, up, wp);
        } else {
#pragma unroll
          for (int k = 0; k < M; ++k)
#pragma unroll
            for (int k6 = 0; k6 < 5; ++k6) w[k][k6] = df[k6][k];
          weno5_fields<R, M>(w, C.weno_eps, wm, wp);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
          wm[k] = cell[RW - 1][k] + wm[k];
          wp[k] = cell[RW][k] - wp[k];
        }
      } else if (C.char_decomp) {
        R x[NC];
        R w[NS][M];
        RP::template char_ctx<dir>(C, cell[RW - 1], cell[RW], x);
#pragma unroll
        for (int k6 = 0; k6 < NS; ++k6) RP::template to_char<dir>(C, x, cell[k6], w[k6]);
        R um[M], up[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
          R line[NS];
#pragma unroll
          for (int k6 = 0; k6 < NS; ++k6) line[k6] = w[k6][k];
          um[k] = weno_edge<RW, false>(line, C.weno_eps);
          up[k] = weno_edge<RW, true>(line, C.weno_eps);
        }
        RP::template from_char<dir>(C, x, um, wm);
        RP::template from_char<dir>(C, x, up, wp);
      } else {
#pragma unroll
        for (int k = 0; k < M; ++k) {
          R line[NS];
#pragma unroll
          for (int k6 = 0; k6 < NS; ++k6) line[k6] = cell[k6][k];
          wm[k] = weno_edge<RW, false>(line, C.weno_eps);
          wp[k] = weno_edge<RW, true>(line, C.weno_eps);
        }
      }
#pragma unroll
      for (int k = 0; k < M; ++k) {
        ER[k][e] = wm[k];
        EL[k][e] = wp[k];
      }
      R al[MAS], ar[MAS];
      if (MA > 0) {
        const int hil = (dir == 0) ? G + a - 1 : G + b, hir = (dir == 0) ? G + a : G + b;
        const int hjl = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a - 1;
        const int hjr = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a;
#pragma unroll
        for (int k = 0; k < MA; ++k) {
          al[k] = At[k][MA > 0 ? hjl : 0][MA > 0 ? OX + hil : 0];
          ar[k] = At[k][MA > 0 ? hjr : 0][MA > 0 ? OX + hir : 0];
        }
      }
      R W[MW][M], s[MW], am[M], ap[M], x[NC];
      RP::template solve<dir>(C, wm, wp, al, ar, W, s, am, ap, x);
#pragma unroll
      for (int k = 0; k < M; ++k) {
        FM[k][e] = am[k];
        FP[k][e] = ap[k];
      }
      // interfaces 0..n of interior lines count for the Courant number
      const int ga = ((dir == 0) ? c0 : r0) + a, gb = ((dir == 0) ? r0 : c0) + b;
      const int nA = (dir == 0) ? nx : ny, nB = (dir == 0) ? ny : nx;
      if (ga <= nA && gb < nB) {
        R m_ = R(0);
        if (C.capa < 0) {
#pragma unroll
          for (int p = 0; p < MW; ++p) m_ = nanmax(m_, (R)fabs(s[p]));
        } else {
          // a wave's Courant number uses the capacity of the cell it enters
          const int hil = (dir == 0) ? G + a - 1 : G + b, hir = (dir == 0) ? G + a : G + b;
          const int hjl = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a - 1;
          const int hjr = (dir == 0) ? ((ND == 2) ? G + b : 0) : G + a;
          const R kl = Kt[hjl][hil], kr = Kt[hjr][hir];
#pragma unroll
          for (int p = 0; p < MW; ++p)
            m_ = nanmax(m_, gt0(s[p]) ? ::claw::FM<R>::div(s[p], kr)
                                      : (lt0(s[p]) ? ::claw::FM<R>::div(-s[p], kl) : R(0)));
        }
        if (dir == 0) smx = nanmax(smx, m_);
        else smy = nanmax(smy, m_);
      }
    };
    // the y-interfaces start on a warp boundary of the loop so that no warp
    // runs both directions' code (slots NEX .. NEXP-1 stay idle)
    constexpr int NEXP = (ND == 2) ? (NEX + 31) / 32 * 32 : NEX;
    for (int t = skip ? NEXP + NEY : tid; t < NEXP + NEY; t += NT) {
      if (t < NEX) interface(std::integral_constant<int, 0>{}, t, t);
      else if constexpr (ND == 2) {
        if (t >= NEXP) interface(std::integral_constant<int, 1>{}, t - NEXP, NEX + t - NEXP);
      }
    }
    __syncthreads();

    // (c) the in-cell Riemann problems (q^L_i, q^R_i) and the cell's L, x then y
    auto incell = [&](auto dirc, int ci, int cj) {
      constexpr int dir = decltype(dirc)::value;
      const int na = (dir == 0) ? TX + 1 : TY + 1;
      const int a = (dir == 0) ? ci : cj, b = (dir == 0) ? cj : ci;
      const int e0 = (dir == 0 ? 0 : NEX) + b * na + a, e1 = e0 + 1;
      R ql[M], qr[M], al[MAS];
#pragma unroll
      for (int k = 0; k < M; ++k) {
        ql[k] = EL[k][e0];
        qr[k] = ER[k][e1];
      }
      if (MA > 0) {
#pragma unroll
        for (int k = 0; k < MA; ++k)
          al[k] = At[k][MA > 0 ? ((ND == 2) ? G + cj : 0) : 0][MA > 0 ? OX + G + ci : 0];
      }
      // total fluctuation A dQ_i = A^- + A^+ of the solve (q^L_i, q^R_i), which
      // for every conservative solver here equals the flux jump
      // f(q^R_i) - f(q^L_i); systems with a non-conservative component
      // (the advected tracer) take the solve itself
      R adq[M];
      if constexpr (incell_solve<RP>::value) {
        R W[MW][M], s_[MW], am[M], ap[M], x[NC];
        RP::template solve<dir>(C, ql, qr, al, al, W, s_, am, ap, x);
#pragma unroll
        for (int k = 0; k < M; ++k) adq[k] = am[k] + ap[k];
      } else {
        R fl[M], fr[M];
        RP::template flux<dir>(C, ql, al, fl);
        RP::template flux<dir>(C, qr, al, fr);
#pragma unroll
        for (int k = 0; k < M; ++k) adq[k] = fr[k] - fl[k];
      }
      // with a capacity the cell's L is -(1/(kappa_i dx)) (...)
      const R idn = s_idn[dir];
      const R idk = C.capa < 0 ? idn
                               : ::claw::FM<R>::div(idn, Kt[(ND == 2) ? G + cj : 0][G + ci]);
#pragma unroll
      for (int k = 0; k < M; ++k) L[k] -= (FP[k][e0] + FM[k][e1] + adq[k]) * idk;
    };
    // thread cidx == tid owns cell (ci, cj) (NT == TX*TY)
    for (int cidx = skip ? TX * TY : tid; cidx < TX * TY; cidx += NT) {
      const int ci = cidx % TX, cj = cidx / TX;
      incell(std::integral_constant<int, 0>{}, ci, cj);
      if constexpr (ND == 2) incell(std::integral_constant<int, 1>{}, ci, cj);
    }
    // (no barrier: the combination below reads only this thread's L and the
    // staged Q^(k); the barriers of finish_attempt precede the next tile)

    // (d) Runge-Kutta stage combination: v = Q^(k) + g dt L, then up to two
    // linear combinations with earlier states
    if (!skip) {
      const int c = c0 + ti, r = r0 + tj;
      if (c < nx && r < ny) {
        const size_t off = (size_t)r * nx + c;
        const R gdt = (R)op.g * s_dt;
        const R a0 = (R)op.a0, a1 = (R)op.a1, b0 = (R)op.b0, b1 = (R)op.b1;
#pragma unroll
        for (int k = 0; k < M; ++k) {
          const R qkv = Qt[k][(ND == 2) ? G + tj : 0][OX + G + ti];
          const R v = qkv + gdt * L[k];
          const R o = (op.a0 != 0.0) ? a0 * qa[k * plane + off] + a1 * v : a1 * v;
          bad |= !isfinite(o);
          qo[k * plane + off] = o;
          if (qo2) {
            const R o2 = (op.b0 != 0.0) ? b0 * qb[k * plane + off] + b1 * v : b1 * v;
            qo2[k * plane + off] = o2;
          }
        }
      }
    }
    finish_attempt<R>(ctl, smx, smy, bad, mb.ntiles, op.last != 0);
  }
}

}  // namespace claw
