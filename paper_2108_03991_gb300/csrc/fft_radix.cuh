// Butterflies of 2, 3, 4, 5 and 8 points in registers.
#pragma once
#include "common.cuh"

namespace bem {

// a + b, a - b, c a + b (c real): in FP32 both parts in one packed instruction (add, fma .f32x2, each part
// rounded as the scalar instruction does), which halves the issue slots of the butterflies' additions
__device__ __forceinline__ unsigned long long f2_pack(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ float2 vadd(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ float2 vfma(float c, float2 a, float2 b) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_pack(make_float2(c, c))), "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return vfma(-1.f, b, a); }
__device__ __forceinline__ double2 vfma(double c, double2 a, double2 b) {
  return make_double2(fma(c, a.x, b.x), fma(c, a.y, b.y));
}
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return csub(a, b); }

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
