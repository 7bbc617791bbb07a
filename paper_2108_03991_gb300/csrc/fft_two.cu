// The grid step's convolution in FP32 for all but small grids (use_two in fft.cu): every transform of length P = A B is two
// register passes with one trip through shared memory between them,
//   n = b + B a, k = ka + A kb:  X[k] = sum_b W_P^(b ka) W_B^(b kb) sum_a W_A^(a ka) x[n],
// the A-point transforms over a with the twiddles W_P^(b ka), then the B-point transforms over b, both
// in place (the spectrum of ka, kb stays at ka (B | 1) + kb; the inverse undoes the passes in
// reverse, so nothing is ever reordered). Three launches over a workspace X[c][kx][z][y] of the
// x-transformed data rows (Px nz ny values a component):
//   x forward : eight rows of one data plane per CTA, read from the grid by the first pass and written
//               kx-major by the second
//   y-z fused : one kx per CTA: y transforms of its nz data rows in shared memory, z transforms of every
//               ky (in registers when Pz is a radix, else as two passes over Pz rows), times Ghat, and
//               back, in place
//   x inverse : the mirror of the first launch
// Bound by the shared-memory pipe at 16 warps per SM (512 x 512 x 8: k_two_yz 66% of its peak, 9% of DRAM's;
// 100 to 128 registers for radices above 16), on small grids by instruction fetch: a value crosses
// shared memory 2 times per line where the forms before (shuffle stages in a warp, 10 shuffles a value;
// radix-8 Stockham passes with a trip per stage; five passes over the whole padded grid where nz > 16;
// or a whole plane per CTA, which leaves SMs without one) took 5 to 25.
// Three components (us): 512 x 512 x 8 399 -> 326, 256 x 256 x 8 101 -> 92, 150 x 90 x 21 242 -> 65, 400 x 300 x
// 12 1,722 -> 219, 96 x 80 x 72 284 -> 100, 200 x 30 x 9 169 -> 26.
// Not kept: every pass through one loop over shared memory, each radix's code once per kernel (782 us
// on 512 x 512 x 8: run-time strides); two or three kx per CTA with 512 threads there (388).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fft_radix.cuh"

namespace bem {

// cos and sin of 2 pi k / M at compile time (Taylor series about 0, |x| <= pi)
constexpr double ct_sin(double x) {
  double t = x, s = x;
  for (int i = 1; i < 20; ++i) {
    t *= -x * x / ((2.0 * i) * (2.0 * i + 1.0));
    s += t;
  }
  return s;
}
constexpr double ct_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int i = 1; i < 20; ++i) {
    t *= -x * x / ((2.0 * i - 1.0) * (2.0 * i));
    s += t;
  }
  return s;
}
template <int M> struct Root {
  float c[M], s[M];
  constexpr Root() : c(), s() {
    for (int k = 0; k < M; ++k) {
      const int q = 2 * k > M ? k - M : k;
      const double x = 6.283185307179586476925 * q / M;
      c[k] = (float)ct_cos(x);
      s[k] = (float)ct_sin(x);
    }
  }
};

template <int M> struct Two { static constexpr int A = 1; };  // M = A * (M / A), both in the list
template <> struct Two<6> { static constexpr int A = 2; };
template <> struct Two<9> { static constexpr int A = 3; };
template <> struct Two<10> { static constexpr int A = 2; };
template <> struct Two<12> { static constexpr int A = 4; };
template <> struct Two<15> { static constexpr int A = 3; };
template <> struct Two<16> { static constexpr int A = 4; };
template <> struct Two<18> { static constexpr int A = 2; };
template <> struct Two<20> { static constexpr int A = 4; };
template <> struct Two<24> { static constexpr int A = 8; };
template <> struct Two<25> { static constexpr int A = 5; };
template <> struct Two<27> { static constexpr int A = 3; };
template <> struct Two<30> { static constexpr int A = 5; };
template <> struct Two<32> { static constexpr int A = 4; };

// M-point butterfly (M of 1, 2, 3, 4, 5, 8) of which only the first N inputs are not zero; the
// cases that occur (N about half of M) without the additions of zeros
template <int M, int N, bool INV> __device__ __forceinline__ void leaf(float2* v) {
  static_assert(N >= 1 && N <= M, "inputs");
  if constexpr (M == 1) {
  } else if constexpr (N == 1) {
#pragma unroll
    for (int k = 1; k < M; ++k) v[k] = v[0];
  } else if constexpr (M == 3 && N == 2) {
    const float h = 0.86602540378443864676f;
    const float2 t = mul_mi(v[1], INV), m = vfma(-0.5f, v[1], v[0]);
    v[0] = vadd(v[0], v[1]);
    v[1] = vfma(h, t, m);
    v[2] = vfma(-h, t, m);
  } else if constexpr (M == 4 && N == 2) {
    const float2 a = v[0], b = v[1], ib = mul_mi(b, INV);
    v[0] = vadd(a, b);
    v[1] = vadd(a, ib);
    v[2] = vsub(a, b);
    v[3] = vsub(a, ib);
  } else if constexpr (M == 5 && N <= 3) {
    const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    const float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
    const float2 p = v[1], q = N == 3 ? v[2] : make_float2(0.f, 0.f);
    const float2 a1 = vfma(c2, q, vfma(c1, p, v[0])), a2 = vfma(c1, q, vfma(c2, p, v[0]));
    const float2 b1 = mul_mi(vfma(s2, q, make_float2(s1 * p.x, s1 * p.y)), INV);
    const float2 b2 = mul_mi(vfma(-s1, q, make_float2(s2 * p.x, s2 * p.y)), INV);
    v[0] = vadd(v[0], vadd(p, q));
    v[1] = vadd(a1, b1);
    v[4] = vsub(a1, b1);
    v[2] = vadd(a2, b2);
    v[3] = vsub(a2, b2);
  } else if constexpr (M == 8 && N <= 4) {
    const float r2 = 0.70710678118654752440f;
    float2 e[4], o[4];
    e[0] = v[0];
    e[1] = N > 2 ? v[2] : make_float2(0.f, 0.f);
    o[0] = v[1];
    o[1] = N > 3 ? v[3] : make_float2(0.f, 0.f);
    leaf<4, 2, INV>(e);
    leaf<4, 2, INV>(o);
    const float2 w1 = INV ? make_float2(o[1].x - o[1].y, o[1].x + o[1].y) : make_float2(o[1].x + o[1].y, o[1].y - o[1].x);
    const float2 w2 = mul_mi(o[2], INV);
    const float2 w3 = INV ? make_float2(-(o[3].x + o[3].y), o[3].x - o[3].y)
                          : make_float2(o[3].y - o[3].x, -(o[3].x + o[3].y));
    v[0] = vadd(e[0], o[0]);
    v[4] = vsub(e[0], o[0]);
    v[1] = vfma(r2, w1, e[1]);
    v[5] = vfma(-r2, w1, e[1]);
    v[2] = vadd(e[2], w2);
    v[6] = vsub(e[2], w2);
    v[3] = vfma(r2, w3, e[3]);
    v[7] = vfma(-r2, w3, e[3]);
  } else {
#pragma unroll
    for (int k = N; k < M; ++k) v[k] = make_float2(0.f, 0.f);
    if constexpr (M == 2) bfly2(v);
    else if constexpr (M == 3) bfly3(v, INV);
    else if constexpr (M == 4) bfly4(v, INV);
    else if constexpr (M == 5) bfly5(v, INV);
    else bfly8(v, INV);
  }
}
template <int I, int N, typename F> __device__ __forceinline__ void each_const(F& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>());
    each_const<I + 1, N>(f);
  }
}
constexpr bool is_leaf(int M) { return M <= 5 || M == 8; }

// natural-order M-point transform in registers of the first NI inputs (the others are zero and are not
// read), its twiddles compile-time constants; outputs that the caller drops cost nothing either
template <int M, bool INV, int NI = M>
__device__ __forceinline__ void dft(float2* v) {
  if constexpr (is_leaf(M)) {
    leaf<M, NI, INV>(v);
  } else {
    constexpr int A = Two<M>::A, B = M / A;
    static_assert(is_leaf(A) && NI >= B, "first level");
    constexpr Root<M> w{};
    float2 u[B][A];
    auto column = [&](auto bc) {
      constexpr int b = decltype(bc)::value, N = (NI - b + B - 1) / B;
#pragma unroll
      for (int a = 0; a < N; ++a) u[b][a] = v[b + B * a];
      leaf<A, N, INV>(u[b]);
#pragma unroll
      for (int k = 1; k < A; ++k)
        if (b > 0) u[b][k] = cmul(u[b][k], make_float2(w.c[b * k], INV ? w.s[b * k] : -w.s[b * k]));
    };
    each_const<0, B>(column);
#pragma unroll
    for (int k = 0; k < A; ++k) {
      float2 t[B];
#pragma unroll
      for (int b = 0; b < B; ++b) t[b] = u[b][k];
      dft<B, INV>(t);
#pragma unroll
      for (int q = 0; q < B; ++q) v[k + A * q] = t[q];
    }
  }
}

#define BEM_RADIX16(X) X(1) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16)
#define BEM_RADIX32(X) X(18) X(20) X(24) X(25) X(27) X(30) X(32)
// f(constant M) for the radix m of the list; kernels whose radices stay below 17 (CLS 16) keep the
// registers of the others out
template <int CLS, typename F> __device__ __forceinline__ void with_radix(int m, F f) {
  switch (m) {
#define BEM_C(M) case M: f(std::integral_constant<int, M>()); break;
    BEM_RADIX16(BEM_C)
    default:
      if constexpr (CLS > 16) {
        switch (m) {
          BEM_RADIX32(BEM_C)
          default: break;
        }
      }
#undef BEM_C
  }
}

static bool is_radix(int m) {
#define BEM_C(M) if (m == M) return true;
  BEM_RADIX16(BEM_C)
  BEM_RADIX32(BEM_C)
#undef BEM_C
  return false;
}

// A >= B with A B = P and the smallest A
static bool two_split(int P, int* A, int* B) {
  for (int a = 1; a <= 32; ++a)
    if (P % a == 0 && P / a <= a && is_radix(a) && is_radix(P / a)) {
      *A = a;
      *B = P / a;
      return true;
    }
  return false;
}

// P >= 2 n - 1: of the A inputs b + B a of a first pass only a < (A + 1) / 2 can hold data, and of the
// outputs of a last pass only those are kept
constexpr int held(int A) { return (A + 1) / 2; }

struct TwoAxis {
  int P, A, B, Bp, pitch;  // Bp = B | 1; pitch: elements of a line in shared memory
};
struct TwoArgs {
  int nx, ny, nz, Pz, gy, gz, zreg, nk;  // zreg: the z transforms run in registers; nk: kx per y-z CTA
  int64_t ng, P3;
  TwoAxis x, y, z;
};
constexpr int kTwoRows = 8;  // rows per CTA of the x passes: 64-byte runs of y in the workspace
constexpr size_t kTwoSmem = 200 * 1024;

template <int CLS>
__global__ void __launch_bounds__(256) k_two_xfwd(const float2* __restrict__ sigma, float2* __restrict__ ws,
                                                  const float2* __restrict__ T, TwoArgs p) {
  extern __shared__ float2 S[];  // [row][ka Bp + b]
  const TwoAxis q = p.x;
  const int y0 = blockIdx.x * kTwoRows, z = blockIdx.y, c = blockIdx.z, nr = min(kTwoRows, p.ny - y0);
  const float2* src = sigma + c * p.ng + ((int64_t)z * p.ny + y0) * p.nx;
  with_radix<CLS>(q.A, [&](auto m) {
    constexpr int A = decltype(m)::value;
    for (int i = threadIdx.x; i < kTwoRows * q.B; i += blockDim.x) {
      const int l = i / q.B, b = i - l * q.B;
      float2 v[A];
#pragma unroll
      for (int a = 0; a < held(A); ++a) {
        const int x = b + q.B * a;
        v[a] = l < nr && x < p.nx ? src[(int64_t)l * p.nx + x] : make_float2(0.f, 0.f);
      }
      dft<A, false, held(A)>(v);
#pragma unroll
      for (int k = 0; k < A; ++k) {
        if (k) v[k] = cmul(v[k], __ldg(T + k * q.B + b));
        S[l * q.pitch + k * q.Bp + b] = v[k];
      }
    }
  });
  __syncthreads();
  float2* dst = ws + c * p.P3 + (int64_t)z * p.ny + y0;
  const int64_t ks = (int64_t)p.nz * p.ny;
  with_radix<CLS>(q.B, [&](auto m) {
    constexpr int B = decltype(m)::value;
    for (int i = threadIdx.x; i < kTwoRows * q.A; i += blockDim.x) {
      const int l = i & (kTwoRows - 1), k = i / kTwoRows;
      float2 v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = S[l * q.pitch + k * q.Bp + b];
      dft<B, false>(v);
      if (l < nr) {
#pragma unroll
        for (int b = 0; b < B; ++b) dst[(k + q.A * b) * ks + l] = v[b];
      }
    }
  });
}

template <int CLS>
__global__ void __launch_bounds__(256) k_two_xinv(const float2* __restrict__ ws, float2* __restrict__ phi,
                                                  const float2* __restrict__ T, TwoArgs p) {
  extern __shared__ float2 S[];
  const TwoAxis q = p.x;
  const int y0 = blockIdx.x * kTwoRows, z = blockIdx.y, c = blockIdx.z, nr = min(kTwoRows, p.ny - y0);
  const float2* src = ws + c * p.P3 + (int64_t)z * p.ny + y0;
  const int64_t ks = (int64_t)p.nz * p.ny;
  with_radix<CLS>(q.B, [&](auto m) {
    constexpr int B = decltype(m)::value;
    for (int i = threadIdx.x; i < kTwoRows * q.A; i += blockDim.x) {
      const int l = i & (kTwoRows - 1), k = i / kTwoRows;
      float2 v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = l < nr ? src[(k + q.A * b) * ks + l] : make_float2(0.f, 0.f);
      dft<B, true>(v);
#pragma unroll
      for (int b = 0; b < B; ++b) S[l * q.pitch + k * q.Bp + b] = cmul(v[b], cconj(__ldg(T + k * q.B + b)));
    }
  });
  __syncthreads();
  float2* dst = phi + c * p.ng + ((int64_t)z * p.ny + y0) * p.nx;
  with_radix<CLS>(q.A, [&](auto m) {
    constexpr int A = decltype(m)::value;
    for (int i = threadIdx.x; i < kTwoRows * q.B; i += blockDim.x) {
      const int l = i / q.B, b = i - l * q.B;
      if (l >= nr) continue;
      float2 v[A];
#pragma unroll
      for (int k = 0; k < A; ++k) v[k] = S[l * q.pitch + k * q.Bp + b];
      dft<A, true>(v);
#pragma unroll
      for (int a = 0; a < held(A); ++a) {
        const int x = b + q.B * a;
        if (x < p.nx) dst[(int64_t)l * p.nx + x] = v[a];
      }
    }
  });
}

template <int CLS>
__global__ void __launch_bounds__(512) k_two_yz(float2* __restrict__ ws, const float2* __restrict__ gs,
                                                const float2* __restrict__ Ty, const float2* __restrict__ Tz,
                                                TwoArgs p) {
  extern __shared__ float2 S[];  // [z][ka Bp + b]
  const TwoAxis q = p.y;
  const int kx0 = blockIdx.x * p.nk, c = blockIdx.y, nk = min(p.nk, p.x.P - kx0);
  const int nl = nk * p.nz;  // lines: the nz rows of kx0, of kx0 + 1, ..., one after another
  float2* X = ws + c * p.P3 + (int64_t)kx0 * p.nz * p.ny;  // [line][y]
  with_radix<CLS>(q.A, [&](auto m) {
    constexpr int A = decltype(m)::value;
    for (int i = threadIdx.x; i < nl * q.B; i += blockDim.x) {
      const int z = i / q.B, b = i - z * q.B;
      float2 v[A];
#pragma unroll
      for (int a = 0; a < held(A); ++a) {
        const int y = b + q.B * a;
        v[a] = y < p.ny ? X[(int64_t)z * p.ny + y] : make_float2(0.f, 0.f);
      }
      dft<A, false, held(A)>(v);
#pragma unroll
      for (int k = 0; k < A; ++k) {
        if (k) v[k] = cmul(v[k], __ldg(Ty + k * q.B + b));
        S[z * q.pitch + k * q.Bp + b] = v[k];
      }
    }
  });
  __syncthreads();
  with_radix<CLS>(q.B, [&](auto m) {
    constexpr int B = decltype(m)::value;
    for (int i = threadIdx.x; i < nl * q.A; i += blockDim.x) {
      const int z = i / q.A, k = i - z * q.A;
      float2* s = S + z * q.pitch + k * q.Bp;
      float2 v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = s[b];
      dft<B, false>(v);
#pragma unroll
      for (int b = 0; b < B; ++b) s[b] = v[b];
    }
  });
  __syncthreads();
  // z transforms, thread = ky = ka + A kb
  if (p.zreg) {
    with_radix<CLS>(p.Pz, [&](auto m) {
      constexpr int M = decltype(m)::value;
      for (int i = threadIdx.x; i < nk * q.P; i += blockDim.x) {
        const int kk = i / q.P, ky = i - kk * q.P, kb = ky / q.A, kx = kx0 + kk;
        float2* s = S + kk * p.nz * q.pitch + (ky - kb * q.A) * q.Bp + kb;
        const int fy = min(ky, q.P - ky);
        const float2* G = gs + (int64_t)min(kx, p.x.P - kx) * p.gz * p.gy;
        float2 v[M];
#pragma unroll
        for (int z = 0; z < held(M); ++z) v[z] = z < p.nz ? s[z * q.pitch] : make_float2(0.f, 0.f);
        dft<M, false, held(M)>(v);
#pragma unroll
        for (int z = 0; z < M; ++z) v[z] = cmul(v[z], __ldg(G + min(z, M - z) * p.gy + fy));
        dft<M, true>(v);
#pragma unroll
        for (int z = 0; z < held(M); ++z)
          if (z < p.nz) s[z * q.pitch] = v[z];
      }
    });
    __syncthreads();
  } else {
    const TwoAxis r = p.z;  // one kx per CTA
    const float2* G = gs + (int64_t)min(kx0, p.x.P - kx0) * p.gz * p.gy;
    with_radix<CLS>(r.A, [&](auto m) {
      constexpr int A = decltype(m)::value;
      for (int i = threadIdx.x; i < r.B * q.P; i += blockDim.x) {
        const int b = i / q.P, ky = i - b * q.P, kb = ky / q.A;
        float2* s = S + (ky - kb * q.A) * q.Bp + kb;
        float2 v[A];
#pragma unroll
        for (int a = 0; a < held(A); ++a) {
          const int z = b + r.B * a;
          v[a] = z < p.nz ? s[z * q.pitch] : make_float2(0.f, 0.f);
        }
        dft<A, false, held(A)>(v);
#pragma unroll
        for (int k = 0; k < A; ++k) {
          if (k) v[k] = cmul(v[k], __ldg(Tz + k * r.B + b));
          s[(b + r.B * k) * q.pitch] = v[k];
        }
      }
    });
    __syncthreads();
    with_radix<CLS>(r.B, [&](auto m) {
      constexpr int B = decltype(m)::value;
      for (int i = threadIdx.x; i < r.A * q.P; i += blockDim.x) {
        const int k = i / q.P, ky = i - k * q.P, kb = ky / q.A;
        float2* s = S + (ky - kb * q.A) * q.Bp + kb + k * r.B * q.pitch;
        const int fy = min(ky, q.P - ky);
        float2 v[B];
#pragma unroll
        for (int b = 0; b < B; ++b) v[b] = s[b * q.pitch];
        dft<B, false>(v);
#pragma unroll
        for (int b = 0; b < B; ++b) {
          const int kz = k + r.A * b;
          v[b] = cmul(v[b], __ldg(G + min(kz, r.P - kz) * p.gy + fy));
        }
        dft<B, true>(v);
#pragma unroll
        for (int b = 0; b < B; ++b) s[b * q.pitch] = cmul(v[b], cconj(__ldg(Tz + k * r.B + b)));
      }
    });
    __syncthreads();
    with_radix<CLS>(r.A, [&](auto m) {
      constexpr int A = decltype(m)::value;
      for (int i = threadIdx.x; i < r.B * q.P; i += blockDim.x) {
        const int b = i / q.P, ky = i - b * q.P, kb = ky / q.A;
        float2* s = S + (ky - kb * q.A) * q.Bp + kb;
        float2 v[A];
#pragma unroll
        for (int k = 0; k < A; ++k) v[k] = s[(b + r.B * k) * q.pitch];
        dft<A, true>(v);
#pragma unroll
        for (int a = 0; a < held(A); ++a) {
          const int z = b + r.B * a;
          if (z < p.nz) s[z * q.pitch] = v[a];
        }
      }
    });
    __syncthreads();
  }
  with_radix<CLS>(q.B, [&](auto m) {
    constexpr int B = decltype(m)::value;
    for (int i = threadIdx.x; i < nl * q.A; i += blockDim.x) {
      const int z = i / q.A, k = i - z * q.A;
      float2* s = S + z * q.pitch + k * q.Bp;
      float2 v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = s[b];
      dft<B, true>(v);
#pragma unroll
      for (int b = 0; b < B; ++b) s[b] = cmul(v[b], cconj(__ldg(Ty + k * q.B + b)));
    }
  });
  __syncthreads();
  with_radix<CLS>(q.A, [&](auto m) {
    constexpr int A = decltype(m)::value;
    for (int i = threadIdx.x; i < nl * q.B; i += blockDim.x) {
      const int z = i / q.B, b = i - z * q.B;
      float2 v[A];
#pragma unroll
      for (int k = 0; k < A; ++k) v[k] = S[z * q.pitch + k * q.Bp + b];
      dft<A, true>(v);
#pragma unroll
      for (int a = 0; a < held(A); ++a) {
        const int y = b + q.B * a;
        if (y < p.ny) X[(int64_t)z * p.ny + y] = v[a];
      }
    }
  });
}

static bool two_args(const aim_ctx* c, TwoArgs* p, size_t* xsm, size_t* ysm) {
  p->nx = c->gn[0];
  p->ny = c->gn[1];
  p->nz = c->gn[2];
  p->Pz = c->gp[2];
  p->ng = c->ng;
  p->P3 = (int64_t)c->gp[0] * c->gp[1] * c->gp[2];
  p->gy = c->gp[1] / 2 + 1;
  p->gz = c->gp[2] / 2 + 1;
  TwoAxis* ax[3] = {&p->x, &p->y, &p->z};
  for (int a = 0; a < 3; ++a) {
    TwoAxis& q = *ax[a];
    q = TwoAxis{c->gp[a], 0, 0, 0, 0};
    if (!two_split(q.P, &q.A, &q.B)) return false;
    q.Bp = q.B | 1;
    // x: eight rows two elements apart fall into different banks (lanes run over rows, then ka)
    q.pitch = a == 0 ? (q.A * q.Bp + 15) / 16 * 16 + 2 : (q.A * q.Bp) | 1;
  }
  p->zreg = is_radix(p->Pz);
  *xsm = (size_t)kTwoRows * p->x.pitch * sizeof(float2);
  const size_t slab = (size_t)(p->zreg ? p->nz : p->Pz) * p->y.pitch * sizeof(float2);
  p->nk = 1;
  // two kx per CTA where both together leave shared memory for three CTAs per SM (registers for four up to
  // radix 16, for two above)
  if (p->zreg && 2 * slab <= 70 * 1024) p->nk = 2;
  *ysm = p->nk * slab;
  return *xsm <= kTwoSmem && *ysm <= kTwoSmem;
}

bool two_path(const aim_ctx* c) {
  TwoArgs p;
  size_t xs, ys;
  return two_args(c, &p, &xs, &ys);
}

// W_P^(b ka) as [ka][b], the two-pass transforms' twiddles
int two_twiddles(aim_ctx* c) {
  TwoArgs p;
  size_t xs, ys;
  if (!two_args(c, &p, &xs, &ys)) return BEM_OK;
  const TwoAxis* ax[3] = {&p.x, &p.y, &p.z};
  for (int a = 0; a < 3; ++a) {
    const TwoAxis& q = *ax[a];
    std::vector<float2> t(q.P);
    for (int k = 0; k < q.A; ++k)
      for (int b = 0; b < q.B; ++b) {
        const double ang = -2.0 * M_PI * (double)((int64_t)k * b % q.P) / q.P;
        t[k * q.B + b] = make_float2((float)std::cos(ang), (float)std::sin(ang));
      }
    BEM_TRY(upload(c, &c->f32.tt[a], t.data(), t.size()));
  }
  return BEM_OK;
}

int two_init_attrs() {
  for (const void* f : {(const void*)k_two_xfwd<16>, (const void*)k_two_xfwd<32>, (const void*)k_two_yz<16>,
                        (const void*)k_two_yz<32>, (const void*)k_two_xinv<16>, (const void*)k_two_xinv<32>})
    BEM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTwoSmem));
  return BEM_OK;
}

// z pass over the padded planes [z][Py][Px] of the plane passes: a thread has one (x, y) line of M = Pz
// points in registers (neighbouring threads neighbouring x: every load and store is coalesced, where
// the shared-memory passes stage a tile and synchronise at every stage). The three passes of 64 x 64 x
// 15, three components, 18.7 -> 14.6 us, of 40 x 40 x 18 10.9 -> 8.2.
template <int M>
__global__ void __launch_bounds__(64) k_two_z(float2* __restrict__ ws, const float2* __restrict__ ghat, int Px, int Py,
                                              int nz, int64_t P3) {
  const int i = blockIdx.x * 64 + threadIdx.x;
  if (i >= Px * Py) return;
  const int y = i / Px, x = i - y * Px, gx = Px / 2 + 1, gy = Py / 2 + 1;
  const int64_t plane = (int64_t)Px * Py;
  float2* s = ws + blockIdx.y * P3 + i;
  const float2* g = ghat + (int64_t)min(y, Py - y) * gx + min(x, Px - x);
  float2 v[M];
#pragma unroll
  for (int z = 0; z < held(M); ++z) v[z] = z < nz ? s[z * plane] : make_float2(0.f, 0.f);
  dft<M, false, held(M)>(v);
#pragma unroll
  for (int z = 0; z < M; ++z) v[z] = cmul(v[z], __ldg(g + (int64_t)min(z, M - z) * gy * gx));
  dft<M, true>(v);
#pragma unroll
  for (int z = 0; z < held(M); ++z)
    if (z < nz) s[z * plane] = v[z];
}

bool two_z_radix(int Pz) { return is_radix(Pz); }

bool two_z(aim_ctx* c, float2* ws, int ncomp, cudaStream_t s) {
  const int Px = c->gp[0], Py = c->gp[1], Pz = c->gp[2];
  const dim3 grid((Px * Py + 63) / 64, ncomp);
  switch (Pz) {
#define BEM_C(M)                                                                                                   \
  case M: k_two_z<M><<<grid, 64, 0, s>>>(ws, c->f32.Ghat, Px, Py, c->gn[2], (int64_t)Px * Py * Pz); return true;
    BEM_RADIX16(BEM_C)
    BEM_RADIX32(BEM_C)
#undef BEM_C
    default: return false;
  }
}

template <int CX, int CY>
static int two_launch(aim_ctx* c, const TwoArgs& p, size_t xsm, size_t ysm, const float2* sigma, float2* phi,
                      int ncomp, float2* ws, cudaStream_t s) {
  PrecBuf<float>& b = c->f32;
  const dim3 gx((p.ny + kTwoRows - 1) / kTwoRows, p.nz, ncomp);
  // threads of the y-z pass: 512 where shared memory leaves room for one CTA per SM
  const int ty = ysm > 100 * 1024 ? 512 : 256;
  const int tx = std::max(64, std::min(256, (int)round_up(kTwoRows * p.x.A, 32)));
  k_two_xfwd<CX><<<gx, tx, xsm, s>>>(sigma, ws, b.tt[0], p);
  k_two_yz<CY><<<dim3((p.x.P + p.nk - 1) / p.nk, ncomp), ty, ysm, s>>>(ws, b.Gs, b.tt[1], b.tt[2], p);
  k_two_xinv<CX><<<gx, tx, xsm, s>>>(ws, phi, b.tt[0], p);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

int two_conv(aim_ctx* c, const float2* sigma, float2* phi, int ncomp, float2* ws, cudaStream_t s) {
  TwoArgs p;
  size_t xsm, ysm;
  if (!two_args(c, &p, &xsm, &ysm)) {
    set_error("two-pass convolution: lengths not supported");
    return BEM_EINVAL;
  }
  const bool bx = p.x.A > 16, by = p.y.A > 16 || (p.zreg ? p.Pz : p.z.A) > 16;
  if (bx) return by ? two_launch<32, 32>(c, p, xsm, ysm, sigma, phi, ncomp, ws, s)
                    : two_launch<32, 16>(c, p, xsm, ysm, sigma, phi, ncomp, ws, s);
  return by ? two_launch<16, 32>(c, p, xsm, ysm, sigma, phi, ncomp, ws, s)
            : two_launch<16, 16>(c, p, xsm, ysm, sigma, phi, ncomp, ws, s);
}

}  // namespace bem
