// vec.cuh -- arithmetic on one value or on a pair of FP32 values (F2), for code
// written once for both.  The packed instructions (fma/add/mul.rn.f32x2) do two
// FP32 operations per issue slot; minima, selects, reciprocals and shuffles
// work on the halves.
#pragma once

#include "riemann.cuh"

namespace claw {

struct F2 {
  unsigned long long v;
  __device__ __forceinline__ F2() {}
  __device__ __forceinline__ F2(float a, float b) {
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  }
  __device__ __forceinline__ explicit F2(float a) : F2(a, a) {}
  __device__ __forceinline__ void get(float& a, float& b) const {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  }
};

// V's scalar type and number of values
template <class V>
struct VecOf {
  using S = V;
  static constexpr int N = 1;
};
template <>
struct VecOf<F2> {
  using S = float;
  static constexpr int N = 2;
};

__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 vsub(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
template <typename R>
__device__ __forceinline__ R vfma(R a, R b, R c) { return fma(a, b, c); }
template <typename R>
__device__ __forceinline__ R vadd(R a, R b) { return a + b; }
template <typename R>
__device__ __forceinline__ R vsub(R a, R b) { return a - b; }
// products that the compiler may not fuse into a neighbouring sum, so that
// every instantiation rounds alike
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }

// c - a b
__device__ __forceinline__ F2 vnfma(F2 a, F2 b, F2 c) { return vsub(c, vmul(a, b)); }
template <typename R>
__device__ __forceinline__ R vnfma(R a, R b, R c) { return fma(-a, b, c); }

// f on each value (pairs: on both halves)
template <class F>
__device__ __forceinline__ F2 vmap(F f, F2 a) {
  float x, y;
  a.get(x, y);
  return F2(f(x), f(y));
}
template <class F>
__device__ __forceinline__ F2 vmap(F f, F2 a, F2 b) {
  float x, y, u, v;
  a.get(x, y);
  b.get(u, v);
  return F2(f(x, u), f(y, v));
}
template <class F>
__device__ __forceinline__ F2 vmap(F f, F2 a, F2 b, F2 c) {
  float x, y, u, v, p, q;
  a.get(x, y);
  b.get(u, v);
  c.get(p, q);
  return F2(f(x, u, p), f(y, v, q));
}
template <class F, typename R>
__device__ __forceinline__ R vmap(F f, R a) { return f(a); }
template <class F, typename R>
__device__ __forceinline__ R vmap(F f, R a, R b) { return f(a, b); }
template <class F, typename R>
__device__ __forceinline__ R vmap(F f, R a, R b, R c) { return f(a, b, c); }
// a predicate that holds for a value (pairs: for either / for both halves)
template <class F>
__device__ __forceinline__ bool vany(F f, F2 a, F2 b, F2 c) {
  float x, y, u, v, p, q;
  a.get(x, y);
  b.get(u, v);
  c.get(p, q);
  return f(x, u, p) || f(y, v, q);
}
template <class F, typename R>
__device__ __forceinline__ bool vany(F f, R a, R b, R c) { return f(a, b, c); }

// the halves as an array
__device__ __forceinline__ void vget(F2 a, float (&x)[2]) { a.get(x[0], x[1]); }
template <typename R>
__device__ __forceinline__ void vget(R a, R (&x)[1]) { x[0] = a; }
__device__ __forceinline__ F2 vput(const float (&x)[2]) { return F2(x[0], x[1]); }
template <typename R>
__device__ __forceinline__ R vput(const R (&x)[1]) { return x[0]; }

template <class V>
__device__ __forceinline__ V vabs(V a) {
  using S = typename VecOf<V>::S;
  return vmap([](S x) { return (S)fabs(x); }, a);
}
template <class V>
__device__ __forceinline__ V vrsq(V a) {
  using S = typename VecOf<V>::S;
  return vmap([](S x) { return FM<S>::rsqrt(x); }, a);
}
// v where s < 0 (m) and elsewhere (p), 0 in the other one.  FP64 by selects
// (the FP64 pipe is the scarce unit), pairs by one packed subtraction
template <class V>
__device__ __forceinline__ void vsplit(V s, V v, V& m, V& p) {
  using S = typename VecOf<V>::S;
  m = vmap([](S a, S x) { return lt0(a) ? x : S(0); }, s, v);
  if constexpr (VecOf<V>::N == 1) p = lt0(s) ? S(0) : v;
  else p = vsub(v, m);
}

// the value of the column to the left / right (columns run over a warp's
// lanes, a pair's halves first)
__device__ __forceinline__ F2 vleft(F2 a) {
  float x, y;
  a.get(x, y);
  return F2(__shfl_up_sync(0xffffffffu, y, 1), x);
}
__device__ __forceinline__ F2 vright(F2 a) {
  float x, y;
  a.get(x, y);
  return F2(y, __shfl_down_sync(0xffffffffu, x, 1));
}
template <typename R>
__device__ __forceinline__ R vleft(R a) { return __shfl_up_sync(0xffffffffu, a, 1); }
template <typename R>
__device__ __forceinline__ R vright(R a) { return __shfl_down_sync(0xffffffffu, a, 1); }

}  // namespace claw
