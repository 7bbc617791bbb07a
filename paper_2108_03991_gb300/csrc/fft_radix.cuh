// Butterflies of 2, 3, 4, 5 and 8 points in registers.
#pragma once
#include "common.cuh"

namespace bem {

// ---------------------------------------------------------------------------------------
// butterflies (forward: exp(-2 pi i / R); inverse: conjugate)
// ---------------------------------------------------------------------------------------
template <typename V> __device__ __forceinline__ V mul_mi(V a, bool inv) {  // * (-i) or * (+i)
  return inv ? mk(-a.y, a.x) : mk(a.y, -a.x);
}

template <typename V> __device__ __forceinline__ void bfly2(V* v) {
  V a = v[0], b = v[1];
  v[0] = vadd(a, b);
  v[1] = vsub(a, b);
}

template <typename V> __device__ __forceinline__ void bfly3(V* v, bool inv) {
  typedef decltype(v[0].x) R;
  const R h = (R)0.86602540378443864676;  // sin(2 pi / 3)
  V t1 = vadd(v[1], v[2]);
  V d = vsub(v[1], v[2]);
  V t2 = mul_mi(d, inv);
  V m = vfma((R)-0.5, t1, v[0]);
  v[0] = vadd(v[0], t1);
  v[1] = vfma(h, t2, m);
  v[2] = vfma(-h, t2, m);
}

template <typename V> __device__ __forceinline__ void bfly4(V* v, bool inv) {
  V y0 = vadd(v[0], v[2]), y1 = vsub(v[0], v[2]), y2 = vadd(v[1], v[3]);
  V y3 = mul_mi(vsub(v[1], v[3]), inv);
  v[0] = vadd(y0, y2);
  v[1] = vadd(y1, y3);
  v[2] = vsub(y0, y2);
  v[3] = vsub(y1, y3);
}

template <typename V> __device__ __forceinline__ void bfly5(V* v, bool inv) {
  typedef decltype(v[0].x) R;
  const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;  // cos 2pi/5, 4pi/5
  const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;   // sin 2pi/5, 4pi/5
  V t1 = vadd(v[1], v[4]), t2 = vadd(v[2], v[3]), t3 = vsub(v[1], v[4]), t4 = vsub(v[2], v[3]);
  V a1 = vfma(c2, t2, vfma(c1, t1, v[0]));
  V a2 = vfma(c1, t2, vfma(c2, t1, v[0]));
  V b1 = vfma(s2, t4, mk(s1 * t3.x, s1 * t3.y));
  V b2 = vfma(-s1, t4, mk(s2 * t3.x, s2 * t3.y));
  V ib1 = mul_mi(b1, inv), ib2 = mul_mi(b2, inv);  // (-i) b forward
  v[0] = vadd(v[0], vadd(t1, t2));
  v[1] = vadd(a1, ib1);
  v[4] = vsub(a1, ib1);
  v[2] = vadd(a2, ib2);
  v[3] = vsub(a2, ib2);
}

template <typename V> __device__ __forceinline__ void bfly8(V* v, bool inv) {
  typedef decltype(v[0].x) R;
  const R r2 = (R)0.70710678118654752440;
  V e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  bfly4(e, inv);
  bfly4(o, inv);
  // w8^k o[k]: w8 = exp(-i pi/4) forward, its factor 1/sqrt(2) left to the last sums
  V w1 = inv ? mk(o[1].x - o[1].y, o[1].x + o[1].y) : mk(o[1].x + o[1].y, o[1].y - o[1].x);
  V w2 = mul_mi(o[2], inv);
  V w3 = inv ? mk(-(o[3].x + o[3].y), o[3].x - o[3].y) : mk(o[3].y - o[3].x, -(o[3].x + o[3].y));
  v[0] = vadd(e[0], o[0]);
  v[4] = vsub(e[0], o[0]);
  v[1] = vfma(r2, w1, e[1]);
  v[5] = vfma(-r2, w1, e[1]);
  v[2] = vadd(e[2], w2);
  v[6] = vsub(e[2], w2);
  v[3] = vfma(r2, w3, e[3]);
  v[7] = vfma(-r2, w3, e[3]);
}

}  // namespace bem
