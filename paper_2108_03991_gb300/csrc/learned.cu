// Learned correction for the preconditioned solve (an extension; the paper's own preconditioner
// is the constraint preconditioner of Qian 2009, Sec. II-C). A 4-layer 3-D convolutional net
// on the AIM grid (3x3x3 kernels, zero padding, no biases, ReLU between layers, channels
// 8 -> 16 -> 16 -> 16 -> 8) maps the projected residual P r (Re/Im of the four grid components,
// scaled by their RMS) to a grid correction that W = P^T interpolates back:
//   M(r) = M_bd r + W net(P r),
// used on the right in flexible GMRES. Weights and activations are BF16, every sum is FP32;
// gradients are FP32. Training minimises |P (W net(P r) - t)|^2 / |P t|^2, t = x - M_bd r, over
// pairs r = A x with x drawn on the device (splitmix64 counter hash, Box-Muller; half of them
// smoothed as grid potentials of random grid sources), with Adam. The error is measured on the
// grid: the block-diagonal part leaves mesh-scale error modes that no grid field represents, and
// the network is meant as a coarse (grid-level) correction beside it.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace bem {

constexpr int kLayers = 4;
constexpr int kCh[kLayers + 1] = {8, 16, 16, 16, 8};
static int wcount(int l) { return kCh[l] * kCh[l + 1] * 27; }
static int woffset(int l) {
  int o = 0;
  for (int i = 0; i < l; ++i) o += wcount(i);
  return o;
}
static int wtotal() { return woffset(kLayers); }

// ---------------------------------------------------------------------------------------
// splitmix64 (Steele, Lea, Flood 2014) as a counter-based hash; Box-Muller normals
// ---------------------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__host__ __device__ __forceinline__ double u01(uint64_t h) {  // (0, 1)
  return ((h >> 11) + 0.5) * (1.0 / 9007199254740992.0);
}
__global__ void k_randn_c(uint64_t seed, int n, float2* out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double u1 = u01(splitmix64(seed ^ (2ull * i))), u2 = u01(splitmix64(seed ^ (2ull * i + 1)));
  double r = sqrt(-2.0 * log(u1)), th = 2.0 * 3.14159265358979323846 * u2;
  out[i] = make_float2((float)(r * cos(th)), (float)(r * sin(th)));
}

// ---------------------------------------------------------------------------------------
// convolution kernels
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_f(float v, float* o) { *o = v; }
__device__ __forceinline__ void from_f(float v, __nv_bfloat16* o) { *o = __float2bfloat16(v); }

// A pass over the grid is cut into tiles of 4 qx by ty by tz points (qx ty tz <= 64, chosen for the
// fewest tiles: tile_of). Two packed FP32 multiply-adds per instruction (fma.rn.f32x2, each half
// rounded as a plain fmaf) leave half the issue slots for the shared-memory loads.
struct Dims {
  int nx, ny, nz;
  int64_t ng;
  int qx, ty, tz;     // tile: quads of points along x, points along y and z
  int ntx, nty, ntz;  // tiles per axis
  int hp, hy, hz;     // halo rows: pitch in floats (a multiple of 4), rows along y and z
};
constexpr int kConvPts = 64;        // quads of points per tile, at most
constexpr int kConvThreads = 128;   // the tile's quads, times two halves of the output channels
constexpr int kGwThreads = 288;     // (input channel, dz, dy) of the weight gradient, times row sets
constexpr int kGwCtas = 456;        // its persistent CTAs (three per SM) and partial sums, at most

typedef unsigned long long f2x;  // two packed FP32
__device__ __forceinline__ f2x pack2(float a, float b) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f2x a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c) {
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// the halo of a tile, C channels [hz][hy][pitch], zero outside the grid; a half-warp per (z, y) row
// of at most 16 values, all channels' loads of it in flight together (one channel at a time spent
// four fifths of a pass waiting for them)
template <int C, typename T>
__device__ __forceinline__ void load_halo(const T* __restrict__ in, const Dims& d, int pitch, int x0,
                                          int y0, int z0, float* s) {
  const int hl = threadIdx.x & 15, nrow = d.hz * d.hy;
  const int x = x0 + hl - 1, w = 4 * d.qx + 2;
  const bool put = hl < pitch, xin = hl < w && x >= 0 && x < d.nx;
  for (int r = threadIdx.x >> 4; r < nrow; r += blockDim.x >> 4) {
    const int y = y0 + r % d.hy - 1, z = z0 + r / d.hy - 1;
    const bool live = xin && y >= 0 && z >= 0 && y < d.ny && z < d.nz;
    const T* src = in + (live ? ((int64_t)z * d.ny + y) * d.nx + x : 0);
    float v[C];
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = live ? to_f(src[c * d.ng]) : 0.f;
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (put) s[(c * nrow + r) * pitch + hl] = v[c];
  }
}

// out[co][p] = act( sum_ci sum_taps w[co][ci][tap] in[ci][p + tap - 1] ) (* mask[co][p] > 0), the sum
// of an output in the order ci, tap. Weights as [ci][tap][co] (k_prep_w). A thread has four
// points along x and half of the output channels: per (ci, dz, dy) it reads six values and 3 CO/2
// weights (broadcast) for 12 CO/2 multiply-adds. Bound by the FP32 pipe (45% active): a layer of 16 to 16
// channels on 35 x 35 x 78 points is 0.66 G multiply-adds (18 us at 36 T/s, 39 measured: 0.86 of a wave
// of CTAs, the shared-memory pipe at 65% of its peak). With one point per thread, 16
// scalar weight loads for 16 multiply-adds, per-channel staging and the weight gradient's two loads
// per multiply-add, a forward and backward pass on that grid took 3.13 ms, a host round trip of
// the input and 14 allocations included; now 0.73 ms.
template <int CI, int CO, typename TI, typename TO, bool RELU>
__global__ void __launch_bounds__(kConvThreads) k_conv(const TI* __restrict__ in,
                                                       const float* __restrict__ w,
                                                       TO* __restrict__ out,
                                                       const __nv_bfloat16* __restrict__ mask, Dims d) {
  constexpr int CH = CO / 2;  // output channels per thread
  extern __shared__ __align__(16) float sm[];
  float* sw = sm;                    // [CI][27][CO]
  float* sin_ = sm + CI * 27 * CO;   // [CI][hz][hy][hp]
  const int bx = blockIdx.x % d.ntx, by = (blockIdx.x / d.ntx) % d.nty, bz = blockIdx.x / (d.ntx * d.nty);
  const int x0 = bx * 4 * d.qx, y0 = by * d.ty, z0 = bz * d.tz;
#pragma unroll 7
  for (int i = threadIdx.x; i < CI * 27 * CO / 4; i += kConvThreads)
    reinterpret_cast<float4*>(sw)[i] = __ldg(reinterpret_cast<const float4*>(w) + i);
  load_halo<CI>(in, d, d.hp, x0, y0, z0, sin_);
  __syncthreads();
  const int half = threadIdx.x / kConvPts, id = threadIdx.x % kConvPts;
  const int q = id % d.qx, ty = (id / d.qx) % d.ty, tz = id / (d.qx * d.ty);
  if (tz >= d.tz) return;
  const int sy = d.hp, sz = d.hp * d.hy;
  const float* base = sin_ + tz * sz + ty * sy + 4 * q;
  const float* wb = sw + half * CH;
  f2x acc[4][CH / 2];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int j = 0; j < CH / 2; ++j) acc[p][j] = 0ull;
  for (int ci = 0; ci < CI; ++ci) {
    const float* sc = base + ci * d.hz * sz;
#pragma unroll
    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        const float* r = sc + dz * sz + dy * sy;
        const float4 a = *reinterpret_cast<const float4*>(r);
        const float2 b = *reinterpret_cast<const float2*>(r + 4);
        const f2x v[6] = {pack2(a.x, a.x), pack2(a.y, a.y), pack2(a.z, a.z),
                          pack2(a.w, a.w), pack2(b.x, b.x), pack2(b.y, b.y)};
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          f2x wv[CH / 2];
#pragma unroll
          for (int j = 0; j < CH / 4; ++j) {
            const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(wb + (dz * 9 + dy * 3 + dx) * CO + 4 * j);
            wv[2 * j] = u.x;
            wv[2 * j + 1] = u.y;
          }
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) acc[p][j] = fma2(wv[j], v[p + dx], acc[p][j]);
        }
      }
    wb += 27 * CO;
  }
  const int x = x0 + 4 * q, y = y0 + ty, z = z0 + tz;
  if (y >= d.ny || z >= d.nz) return;
  const int64_t pt = ((int64_t)z * d.ny + y) * d.nx + x;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (x + p >= d.nx) break;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const float2 u = unpack2(acc[p][j / 2]);
      float v = j & 1 ? u.y : u.x;
      const int64_t o = (half * CH + j) * d.ng + pt + p;
      if (RELU) v = fmaxf(v, 0.f);
      if (mask && !(__bfloat162float(mask[o]) > 0.f)) v = 0.f;
      from_f(v, &out[o]);
    }
  }
}

// part[cta][ci][tap][co] = sum over the CTA's tiles of g[co][p] in[ci][p + tap - 1]. A thread has one
// (ci, dz, dy), the three dx and half of the output channels; it walks the tile's rows along x with
// a sliding window of three inputs, so a point costs one input load and CO / 8 broadcast loads of g
// for 3 CO / 2 multiply-adds. With 8 input channels two sets of threads share the rows. Three CTAs
// per SM (half the channels per thread keep it under 76 registers). The CTAs' sums meet in
// k_gw_reduce.
template <int CI, int CO, typename TI>
__global__ void __launch_bounds__(kGwThreads, 3) k_conv_gw(const TI* __restrict__ in,
                                                        const float* __restrict__ g,
                                                        float* __restrict__ part, Dims d) {
  constexpr int NS = kGwThreads / (CI * 18);  // 1 or 2 sets of rows
  constexpr int CH = CO / 2;                 // output channels per thread
  constexpr int GP = CO + 4;                 // floats per point of g in shared memory
  extern __shared__ __align__(16) float sm[];
  const int tx = 4 * d.qx, npt = tx * d.ty * d.tz;
  const int pitch = tx + 3;  // odd: the lanes' rows (input channel, dz, dy) start in different banks
  float* sg = sm;               // [point][GP]
  float* sin_ = sm + npt * GP;  // [CI][hz][hy][pitch]
  const int set = threadIdx.x / (CI * 18), half = threadIdx.x / (CI * 9) % 2, id = threadIdx.x % (CI * 9);
  const int ci = id / 9, dz = (id % 9) / 3, dy = id % 3;
  f2x acc[3][CH / 2];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < CH / 2; ++j) acc[k][j] = 0ull;
  const int ntile = d.ntx * d.nty * d.ntz;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int x0 = (tile % d.ntx) * tx, y0 = (tile / d.ntx) % d.nty * d.ty, z0 = tile / (d.ntx * d.nty) * d.tz;
    __syncthreads();  // the last tile's readers are done
    load_halo<CI>(in, d, pitch, x0, y0, z0, sin_);
    if (threadIdx.x < npt) {  // npt <= 256
      const int p = threadIdx.x;
      const int x = x0 + p % tx, y = y0 + p / tx % d.ty, z = z0 + p / (tx * d.ty);
      const bool live = x < d.nx && y < d.ny && z < d.nz;
      const float* src = g + (live ? ((int64_t)z * d.ny + y) * d.nx + x : 0);
      float v[CO];
#pragma unroll
      for (int co = 0; co < CO; ++co) v[co] = live ? src[co * d.ng] : 0.f;
#pragma unroll
      for (int co = 0; co < CO; co += 4)
        *reinterpret_cast<float4*>(sg + p * GP + co) = make_float4(v[co], v[co + 1], v[co + 2], v[co + 3]);
    }
    __syncthreads();
    for (int row = set; row < d.ty * d.tz; row += NS) {
      const int ry = row % d.ty, rz = row / d.ty;
      const float* r = sin_ + ((ci * d.hz + rz + dz) * d.hy + ry + dy) * pitch;
      const float* gr = sg + row * tx * GP + half * CH;
      f2x v0 = pack2(r[0], r[0]), v1 = pack2(r[1], r[1]);
#pragma unroll 4
      for (int x = 0; x < tx; ++x) {
        const f2x v2 = pack2(r[x + 2], r[x + 2]);
#pragma unroll
        for (int j = 0; j < CH / 4; ++j) {
          const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(gr + x * GP + 4 * j);
          acc[0][2 * j] = fma2(u.x, v0, acc[0][2 * j]);
          acc[0][2 * j + 1] = fma2(u.y, v0, acc[0][2 * j + 1]);
          acc[1][2 * j] = fma2(u.x, v1, acc[1][2 * j]);
          acc[1][2 * j + 1] = fma2(u.y, v1, acc[1][2 * j + 1]);
          acc[2][2 * j] = fma2(u.x, v2, acc[2][2 * j]);
          acc[2][2 * j + 1] = fma2(u.y, v2, acc[2][2 * j + 1]);
        }
        v0 = v1;
        v1 = v2;
      }
    }
  }
  // the sets' sums meet in shared memory, then one [ci][tap][co] block per CTA goes out
  float* red = sm;  // [CI * 27][CO]
  for (int k = 0; k < NS; ++k) {
    __syncthreads();
    if (set != k) continue;
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int j = 0; j < CH / 2; ++j) {
        float2* o = reinterpret_cast<float2*>(red + (ci * 27 + dz * 9 + dy * 3 + q) * CO + half * CH) + j;
        const float2 v = unpack2(acc[q][j]);
        *o = k == 0 ? v : make_float2(o->x + v.x, o->y + v.y);
      }
  }
  __syncthreads();
  float4* dst = reinterpret_cast<float4*>(part + (int64_t)blockIdx.x * CI * 27 * CO);
  for (int i = threadIdx.x; i < CI * 27 * CO / 4; i += kGwThreads) dst[i] = reinterpret_cast<float4*>(red)[i];
}

// gw[co][ci][tap] += the sum of the ncta partial sums, eight threads per weight in a fixed order
__global__ void __launch_bounds__(256) k_gw_reduce(const float* __restrict__ part, int ncta, int CI,
                                                   int CO, float* __restrict__ gw) {
  __shared__ float s[8][32];
  const int n = CI * CO * 27, lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;  // [ci][tap][co]
  float acc = 0.f;
  if (i < n) {
#pragma unroll 8
    for (int c = k; c < ncta; c += 8) acc += part[(int64_t)c * n + i];
  }
  s[k][lane] = acc;
  __syncthreads();
  if (k == 0 && i < n) {
    for (int q = 1; q < 8; ++q) acc += s[q][lane];
    const int co = i % CO, t = i / CO % 27, ci = i / (CO * 27);
    gw[(co * CI + ci) * 27 + t] += acc;
  }
}

// the passes' weights, all layers at once: BF16-rounded (the network's weights are BF16) as
// wf[ci][tap][co] for the forward pass and wb[co][26 - tap][ci] (transposed, flipped) for the
// backward-data pass
__global__ void k_prep_w(const float* w0, float* wf0, float* wb0) {
  const int l = blockIdx.y, CI = l == 0 ? 8 : 16, CO = l == kLayers - 1 ? 8 : 16;
  const int off = l == 0 ? 0 : (8 * 16 + (l - 1) * 16 * 16) * 27;
  const float* w = w0 + off;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= CI * CO * 27) return;
  const int t = i % 27, ci = (i / 27) % CI, co = i / (27 * CI);
  const float v = __bfloat162float(__float2bfloat16(w[i]));
  wf0[off + (ci * 27 + t) * CO + co] = v;
  wb0[off + (co * 27 + 26 - t) * CI + ci] = v;
}

__global__ void k_adam(float* w, float* m, float* v, const float* g, int n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float gi = g[i];
  float mi = b1 * m[i] + (1.f - b1) * gi, vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---------------------------------------------------------------------------------------
// grid <-> channels
// ---------------------------------------------------------------------------------------
__global__ void k_to_bf16(const float* a, int64_t n, __nv_bfloat16* o) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) o[i] = __float2bfloat16(a[i]);
}
__global__ void k_sumsq(const float2* s, int64_t n, float* out) {
  float acc = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += s[i].x * s[i].x + s[i].y * s[i].y;
  acc = warp_sum(make_float2(acc, 0.f)).x;
  if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}
// x[2c][p] = Re sigma_c(p) / rms, x[2c+1][p] = Im sigma_c(p) / rms (rms over all 8 channels)
__global__ void k_pack(const float2* sig, const float* sumsq, int64_t ng, __nv_bfloat16* x) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= 4 * ng) return;
  const float rms = sqrtf(fmaxf(*sumsq, 1e-30f) / (8.f * ng));
  const int64_t c = i / ng, p = i - c * ng;
  x[2 * c * ng + p] = __float2bfloat16(sig[i].x / rms);
  x[(2 * c + 1) * ng + p] = __float2bfloat16(sig[i].y / rms);
}
// phi_c(p) = rms (out[2c][p] + i out[2c+1][p])
__global__ void k_unpack(const float* out, const float* sumsq, int64_t ng, float2* phi) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= 4 * ng) return;
  const float rms = sqrtf(fmaxf(*sumsq, 1e-30f) / (8.f * ng));
  const int64_t c = i / ng, p = i - c * ng;
  phi[i] = make_float2(rms * out[2 * c * ng + p], rms * out[(2 * c + 1) * ng + p]);
}
// g_out[2c][p] = rms Re gphi_c(p) * scale, g_out[2c+1][p] = rms Im gphi_c(p) * scale
__global__ void k_pack_grad(const float2* gphi, const float* sumsq, const float* tnorm2, int64_t ng,
                            float* g) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= 4 * ng) return;
  const float rms = sqrtf(fmaxf(*sumsq, 1e-30f) / (8.f * ng));
  const float sc = 2.f * rms / fmaxf(*tnorm2, 1e-30f);
  const int64_t c = i / ng, p = i - c * ng;
  g[2 * c * ng + p] = sc * gphi[i].x;
  g[(2 * c + 1) * ng + p] = sc * gphi[i].y;
}
__global__ void k_axpy_c(const float2* a, const float2* b, float sb, int n, float2* o) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = make_float2(a[i].x + sb * b[i].x, a[i].y + sb * b[i].y);
}

// ---------------------------------------------------------------------------------------
// network state
// ---------------------------------------------------------------------------------------
struct Net {
  int nw = 0;
  float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
  float *wf = nullptr, *wb = nullptr;  // the passes' weights (k_prep_w)
  float* part = nullptr;               // [kGwCtas][16 * 16 * 27] partial weight gradients
  __nv_bfloat16* act[kLayers] = {nullptr, nullptr, nullptr, nullptr};  // x, h1, h2, h3
  float* out = nullptr;      // [8][ng]
  float* gbuf[2] = {nullptr, nullptr};  // [16][ng] gradients
  float* scal = nullptr;     // [0] sumsq of the input grid, [1..2] |e|^2, |t|^2
  float2 *sig = nullptr, *phi = nullptr, *g2 = nullptr;  // [4][ng]
  float2 *x = nullptr, *r = nullptr, *t = nullptr, *u = nullptr, *e = nullptr;  // [N]
  int adam_t = 0;
  std::vector<void*> mem;
  char* arena = nullptr;  // one allocation that alloc() hands out (a pass of its own), if any
  size_t left = 0;
  ~Net() { for (void* p : mem) cudaFree(p); }
  static size_t padded(size_t bytes) { return (bytes + 16 + 255) & ~(size_t)255; }
  int reserve(size_t bytes) {
    char* p = nullptr;
    BEM_TRY(alloc(&p, bytes));
    arena = p;
    left = bytes;
    return BEM_OK;
  }
  template <typename T> int alloc(T** p, size_t n) {
    if (arena) {
      const size_t b = padded(n * sizeof(T));
      if (b > left) { set_error("net allocation: workspace too small"); return BEM_ENOMEM; }
      *p = reinterpret_cast<T*>(arena);
      arena += b;
      left -= b;
      return BEM_OK;
    }
    cudaError_t e = cudaMalloc((void**)p, n * sizeof(T) + 16);
    if (e != cudaSuccess) { set_error("net allocation: %s", cudaGetErrorString(e)); return BEM_ENOMEM; }
    mem.push_back(*p);
    return BEM_OK;
  }
};

// The tile with the fewest tiles to cover the grid (each costs the same), then the smallest halo
static Dims dims_of(int nx, int ny, int nz) {
  Dims d;
  d.nx = nx; d.ny = ny; d.nz = nz;
  d.ng = (int64_t)nx * ny * nz;
  const int nq = (nx + 3) / 4;
  int64_t best = INT64_MAX, halo = 0;
  for (int qx = 1; qx <= 3; ++qx)
    for (int ty = 1; ty <= 16; ++ty) {
      const int tz = std::min(kConvPts / (qx * ty), 16);
      if (tz < 1) break;
      const int64_t tiles = (int64_t)((nq + qx - 1) / qx) * ((ny + ty - 1) / ty) * ((nz + tz - 1) / tz);
      const int64_t h = (int64_t)(4 * qx + 4) * (ty + 2) * (tz + 2);
      if (h > 900) continue;  // 16 channels of halo in 58 KB
      if (tiles < best || (tiles == best && h < halo)) {
        best = tiles;
        halo = h;
        d.qx = qx; d.ty = ty; d.tz = tz;
      }
    }
  d.ntx = (nq + d.qx - 1) / d.qx;
  d.nty = (ny + d.ty - 1) / d.ty;
  d.ntz = (nz + d.tz - 1) / d.tz;
  d.hp = 4 * d.qx + 4;
  d.hy = d.ty + 2;
  d.hz = d.tz + 2;
  return d;
}

static size_t halo_bytes(int C, const Dims& d) { return (size_t)C * d.hz * d.hy * d.hp * 4; }
static size_t conv_smem(int CI, int CO, const Dims& d) { return (size_t)CO * CI * 27 * 4 + halo_bytes(CI, d); }
static size_t gw_smem(int CI, int CO, const Dims& d) {
  return std::max((size_t)CO * CI * 27 * 4, (size_t)4 * d.qx * d.ty * d.tz * (CO + 4) * 4 + halo_bytes(CI, d));
}

template <int CI, int CO, typename TI, typename TO, bool RELU>
static int launch_conv(const TI* in, const float* w, TO* out, const __nv_bfloat16* mask, const Dims& d,
                       cudaStream_t s) {
  const size_t sm = conv_smem(CI, CO, d);
  // per call: the attribute belongs to the current device
  BEM_CUDA(cudaFuncSetAttribute(k_conv<CI, CO, TI, TO, RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  BEM_CUDA(cudaFuncSetAttribute(k_conv<CI, CO, TI, TO, RELU>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  k_conv<CI, CO, TI, TO, RELU><<<d.ntx * d.nty * d.ntz, kConvThreads, sm, s>>>(in, w, out, mask, d);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

template <int CI, int CO, typename TI>
static int launch_gw(const TI* in, const float* g, float* part, float* gw, const Dims& d, cudaStream_t s) {
  const size_t sm = gw_smem(CI, CO, d);
  const int ncta = std::min(d.ntx * d.nty * d.ntz, kGwCtas);
  BEM_CUDA(cudaFuncSetAttribute(k_conv_gw<CI, CO, TI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  BEM_CUDA(cudaFuncSetAttribute(k_conv_gw<CI, CO, TI>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  k_conv_gw<CI, CO, TI><<<ncta, kGwThreads, sm, s>>>(in, g, part, d);
  k_gw_reduce<<<(CI * CO * 27 + 31) / 32, 256, 0, s>>>(part, ncta, CI, CO, gw);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

static int prep_weights(Net& n, cudaStream_t s) {
  static_assert(kLayers == 4, "k_prep_w's layer offsets");
  k_prep_w<<<dim3((16 * 16 * 27 + 255) / 256, kLayers), 256, 0, s>>>(n.w, n.wf, n.wb);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// forward: act[0] = x (BF16) given; act[1..3] = ReLU layers (BF16); out (FP32)
static int net_forward(Net& n, const Dims& d, cudaStream_t s) {
  BEM_TRY(prep_weights(n, s));
  const float* w = n.wf;
  BEM_TRY((launch_conv<8, 16, __nv_bfloat16, __nv_bfloat16, true>(n.act[0], w + woffset(0), n.act[1], nullptr, d, s)));
  BEM_TRY((launch_conv<16, 16, __nv_bfloat16, __nv_bfloat16, true>(n.act[1], w + woffset(1), n.act[2], nullptr, d, s)));
  BEM_TRY((launch_conv<16, 16, __nv_bfloat16, __nv_bfloat16, true>(n.act[2], w + woffset(2), n.act[3], nullptr, d, s)));
  BEM_TRY((launch_conv<16, 8, __nv_bfloat16, float, false>(n.act[3], w + woffset(3), n.out, nullptr, d, s)));
  return BEM_OK;
}

// backward from gout = dL/d(out) (FP32 [8][ng], may be n.gbuf[0]) after net_forward with the same
// weights; accumulates n.g; writes dL/dx into gx (FP32 [8][ng]) when gx != nullptr
static int net_backward(Net& n, const Dims& d, const float* gout, float* gx, cudaStream_t s) {
  float* g0 = n.gbuf[0];
  float* g1 = n.gbuf[1];
  const float* w = n.wb;
  // layer 3: 16 -> 8
  BEM_TRY((launch_gw<16, 8, __nv_bfloat16>(n.act[3], gout, n.part, n.g + woffset(3), d, s)));
  BEM_TRY((launch_conv<8, 16, float, float, false>(gout, w + woffset(3), g1, n.act[3], d, s)));
  // layer 2: 16 -> 16
  BEM_TRY((launch_gw<16, 16, __nv_bfloat16>(n.act[2], g1, n.part, n.g + woffset(2), d, s)));
  BEM_TRY((launch_conv<16, 16, float, float, false>(g1, w + woffset(2), g0, n.act[2], d, s)));
  // layer 1: 16 -> 16
  BEM_TRY((launch_gw<16, 16, __nv_bfloat16>(n.act[1], g0, n.part, n.g + woffset(1), d, s)));
  BEM_TRY((launch_conv<16, 16, float, float, false>(g0, w + woffset(1), g1, n.act[1], d, s)));
  // layer 0: 8 -> 16
  BEM_TRY((launch_gw<8, 16, __nv_bfloat16>(n.act[0], g1, n.part, n.g + woffset(0), d, s)));
  if (gx) BEM_TRY((launch_conv<16, 8, float, float, false>(g1, w + woffset(0), gx, nullptr, d, s)));
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

static int net_alloc_grid(Net& n, int64_t ng) {
  BEM_TRY(n.alloc(&n.act[0], 8 * (size_t)ng));
  for (int l = 1; l < kLayers; ++l) BEM_TRY(n.alloc(&n.act[l], 16 * (size_t)ng));
  BEM_TRY(n.alloc(&n.out, 8 * (size_t)ng));
  BEM_TRY(n.alloc(&n.gbuf[0], 16 * (size_t)ng));
  BEM_TRY(n.alloc(&n.gbuf[1], 16 * (size_t)ng));
  BEM_TRY(n.alloc(&n.part, (size_t)kGwCtas * 16 * 16 * 27));
  return BEM_OK;
}

static int net_alloc_weights(Net& n) {
  n.nw = wtotal();
  BEM_TRY(n.alloc(&n.w, n.nw));
  BEM_TRY(n.alloc(&n.m, n.nw));
  BEM_TRY(n.alloc(&n.v, n.nw));
  BEM_TRY(n.alloc(&n.g, n.nw));
  BEM_TRY(n.alloc(&n.wf, n.nw));
  BEM_TRY(n.alloc(&n.wb, n.nw));
  BEM_CUDA(cudaMemset(n.m, 0, n.nw * sizeof(float)));
  BEM_CUDA(cudaMemset(n.v, 0, n.nw * sizeof(float)));
  return BEM_OK;
}

static Net* get_net(aim_ctx* c, int* rc) {
  *rc = BEM_OK;
  if (c->net) return static_cast<Net*>(c->net);
  Net* n = new Net();
  *rc = net_alloc_weights(*n);
  if (*rc == BEM_OK) *rc = net_alloc_grid(*n, c->ng);
  const size_t N = (size_t)c->ne + c->nt;
  if (*rc == BEM_OK) *rc = n->alloc(&n->scal, 8);
  if (*rc == BEM_OK) *rc = n->alloc(&n->sig, 4 * (size_t)c->ng);
  if (*rc == BEM_OK) *rc = n->alloc(&n->phi, 4 * (size_t)c->ng);
  if (*rc == BEM_OK) *rc = n->alloc(&n->g2, 4 * (size_t)c->ng);
  for (float2** p : {&n->x, &n->r, &n->t, &n->u, &n->e})
    if (*rc == BEM_OK) *rc = n->alloc(p, N);
  if (*rc != BEM_OK) {
    delete n;
    return nullptr;
  }
  c->net = n;
  return n;
}

void free_net(aim_ctx* c) {
  delete static_cast<Net*>(c->net);
  c->net = nullptr;
}

// u = W net(P r) (FP32), using the context's grid; scal[0] holds the input grid's sum of squares
static int net_correction(aim_ctx* c, Net& n, const float2* r, float2* u, cudaStream_t s) {
  const Dims d = dims_of(c->gn[0], c->gn[1], c->gn[2]);
  BEM_TRY(project_all<float>(c, r, n.sig, s));
  BEM_CUDA(cudaMemsetAsync(n.scal, 0, sizeof(float), s));
  k_sumsq<<<304, 256, 0, s>>>(n.sig, 4 * c->ng, n.scal);
  k_pack<<<(unsigned)((4 * c->ng + 255) / 256), 256, 0, s>>>(n.sig, n.scal, c->ng, n.act[0]);
  BEM_TRY(net_forward(n, d, s));
  k_unpack<<<(unsigned)((4 * c->ng + 255) / 256), 256, 0, s>>>(n.out, n.scal, c->ng, n.phi);
  BEM_TRY(interp_all<float>(c, n.phi, u, s));
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

int net_apply(aim_ctx* c, const float2* r, float2* z, cudaStream_t s) {
  int rc = BEM_OK;
  Net* n = get_net(c, &rc);
  if (!n) return rc;
  const int N = c->ne + c->nt;
  BEM_TRY(setup_precond(c));
  BEM_TRY(precond_apply<float>(c, r, z, s));
  BEM_TRY(net_correction(c, *n, r, n->u, s));
  k_axpy_c<<<(N + 255) / 256, 256, 0, s>>>(z, n->u, 1.f, N, z);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// one training step over `batch` fresh pairs; returns the mean relative loss
static int net_train_step(aim_ctx* c, Net& n, int batch, float lr, uint64_t seed, float* loss,
                          cudaStream_t s) {
  const Dims d = dims_of(c->gn[0], c->gn[1], c->gn[2]);
  const int N = c->ne + c->nt;
  BEM_CUDA(cudaMemsetAsync(n.g, 0, n.nw * sizeof(float), s));
  double lsum = 0;
  for (int b = 0; b < batch; ++b) {
    if (b % 2 == 0) {
      // white x
      k_randn_c<<<(N + 255) / 256, 256, 0, s>>>(splitmix64(seed * 7919ull + b), N, n.x);
    } else {
      // smooth x: grid potentials of random grid sources, interpolated to the unknowns
      const int64_t n4 = 4 * c->ng;
      k_randn_c<<<(unsigned)((n4 + 255) / 256), 256, 0, s>>>(splitmix64(seed * 7919ull + b), (int)n4,
                                                             n.sig);
      BEM_TRY(fft_conv<float>(c, c->f32, n.sig, n.phi, 4, c->f32.ws, s));
      BEM_TRY(interp_all<float>(c, n.phi, n.x, s));
    }
    BEM_TRY(matvec_graph<float>(c, AIM_OP_SYSTEM, n.x, n.r, s));          // r = A x
    BEM_TRY(precond_apply<float>(c, n.r, n.t, s));                        // t = M_bd r
    k_axpy_c<<<(N + 255) / 256, 256, 0, s>>>(n.x, n.t, -1.f, N, n.t);     // t = x - M_bd r
    BEM_TRY(net_correction(c, n, n.r, n.u, s));                           // u = W net(P r)
    // loss |P e|^2 / |P t|^2 with e = u - t: the error measured on the grid, where the
    // correction lives; gradient w.r.t. the output grid = 2 P W P e / |P t|^2
    BEM_CUDA(cudaMemsetAsync(n.scal + 1, 0, 2 * sizeof(float), s));
    k_axpy_c<<<(N + 255) / 256, 256, 0, s>>>(n.u, n.t, -1.f, N, n.e);     // e = u - t
    BEM_TRY(project_all<float>(c, n.e, n.phi, s));                         // P e
    BEM_TRY(project_all<float>(c, n.t, n.g2, s));                          // P t
    k_sumsq<<<304, 256, 0, s>>>(n.phi, 4 * c->ng, n.scal + 1);
    k_sumsq<<<304, 256, 0, s>>>(n.g2, 4 * c->ng, n.scal + 2);
    BEM_TRY(interp_all<float>(c, n.phi, n.e, s));                          // W P e
    BEM_TRY(project_all<float>(c, n.e, n.phi, s));                         // P W P e
    k_pack_grad<<<(unsigned)((4 * c->ng + 255) / 256), 256, 0, s>>>(n.phi, n.scal, n.scal + 2,
                                                                        c->ng, n.gbuf[0]);
    BEM_TRY(net_backward(n, d, n.gbuf[0], nullptr, s));
    float h[2];
    BEM_CUDA(cudaMemcpyAsync(h, n.scal + 1, 2 * sizeof(float), cudaMemcpyDeviceToHost, s));
    BEM_CUDA(cudaStreamSynchronize(s));
    lsum += h[0] / std::max(h[1], 1e-30f);
  }
  // Adam on the batch-summed gradient: the step m/sqrt(v) does not change when the gradient is
  // scaled, so summing instead of averaging only rescales eps (passed as eps * batch)
  ++n.adam_t;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n.adam_t), c2 = 1.f - std::pow(b2, (float)n.adam_t);
  k_adam<<<(n.nw + 255) / 256, 256, 0, s>>>(n.w, n.m, n.v, n.g, n.nw, lr, b1, b2, 1e-8f * batch,
                                            c1, c2);
  BEM_CUDA(cudaGetLastError());
  *loss = (float)(lsum / batch);
  return BEM_OK;
}

}  // namespace bem

using namespace bem;

extern "C" {

int bem_net_init(aim_ctx* c, uint64_t seed) {
  if (!c) { set_error("bem_net_init: null context"); return BEM_EINVAL; }
  int rc = BEM_OK;
  Net* n = get_net(c, &rc);
  if (!n) return rc;
  std::vector<float> w(n->nw);
  int o = 0;
  for (int l = 0; l < kLayers; ++l) {
    const double sd = std::sqrt(2.0 / (27.0 * kCh[l]));
    for (int i = 0; i < wcount(l); ++i, ++o) {
      double u1 = u01(splitmix64(seed ^ (2ull * o))), u2 = u01(splitmix64(seed ^ (2ull * o + 1)));
      w[o] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(2.0 * M_PI * u2));
    }
  }
  BEM_CUDA(cudaMemcpy(n->w, w.data(), n->nw * sizeof(float), cudaMemcpyHostToDevice));
  BEM_CUDA(cudaMemset(n->m, 0, n->nw * sizeof(float)));
  BEM_CUDA(cudaMemset(n->v, 0, n->nw * sizeof(float)));
  n->adam_t = 0;
  return BEM_OK;
}

int64_t bem_net_weights(aim_ctx* c, float* w, int64_t n, int set) {
  if (!c) { set_error("bem_net_weights: null context"); return BEM_EINVAL; }
  int rc = BEM_OK;
  Net* net = get_net(c, &rc);
  if (!net) return rc;
  if (!w) return net->nw;
  if (n != net->nw) { set_error("bem_net_weights: expected %d weights", net->nw); return BEM_EINVAL; }
  if (set) {
    BEM_CUDA(cudaMemcpy(net->w, w, n * sizeof(float), cudaMemcpyHostToDevice));
    BEM_CUDA(cudaMemset(net->m, 0, n * sizeof(float)));
    BEM_CUDA(cudaMemset(net->v, 0, n * sizeof(float)));
    net->adam_t = 0;
  } else {
    BEM_CUDA(cudaMemcpy(w, net->w, n * sizeof(float), cudaMemcpyDeviceToHost));
  }
  return n;
}

int bem_net_train(aim_ctx* c, int steps, int batch, float lr, uint64_t seed, float* losses,
                  void* stream) {
  if (!c || steps < 1 || batch < 1 || !(lr > 0)) {
    set_error("bem_net_train: bad arguments");
    return BEM_EINVAL;
  }
  int rc = BEM_OK;
  Net* n = get_net(c, &rc);
  if (!n) return rc;
  // the targets x - M_bd A x hold M_bd's own error A_ii^{-1} - X_ii: with inverses built in FP32
  // that is the FP32 LU's error (left residual ~ cond * eps), mesh-scale noise no grid
  // correction can learn, so training builds them in FP64
  BEM_TRY(setup_precond(c, BEM_C64));
  cudaStream_t s = (cudaStream_t)stream;
  for (int k = 0; k < steps; ++k) {
    float l = 0;
    BEM_TRY(net_train_step(c, *n, batch, lr, splitmix64(seed + 1000003ull * k), &l, s));
    if (losses) losses[k] = l;
  }
  return BEM_OK;
}

int bem_net_apply(aim_ctx* c, const void* r, void* z, int correction_only, void* stream) {
  if (!c || !r || !z || r == z) {
    set_error("bem_net_apply: bad arguments");
    return BEM_EINVAL;
  }
  if (!correction_only) return net_apply(c, (const float2*)r, (float2*)z, (cudaStream_t)stream);
  int rc = BEM_OK;
  Net* n = get_net(c, &rc);
  if (!n) return rc;
  return net_correction(c, *n, (const float2*)r, (float2*)z, (cudaStream_t)stream);
}

// Standalone network pass for verification: x [8][ng] FP32 (rounded to BF16 on entry), weights
// FP32 host (rounded to BF16 in the kernels), out [8][ng] FP32; with gout [8][ng] the backward
// pass writes gw (host, FP32, layers one after another) and gx [8][ng] (device).
int bem_convnet_run(int nx, int ny, int nz, const float* w_host, const float* x, const float* gout,
                    float* out, float* gw_host, float* gx, void* stream) {
  if (nx < 1 || ny < 1 || nz < 1 || !w_host || !x || !out) {
    set_error("bem_convnet_run: bad arguments");
    return BEM_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  Net n;
  const Dims d = dims_of(nx, ny, nz);
  n.nw = wtotal();
  const size_t ng = (size_t)d.ng;
  // one allocation for the pass: weights (plain, forward, backward), gradients, activations
  size_t bytes = 4 * Net::padded(n.nw * sizeof(float)) + Net::padded(8 * ng * 2) + 3 * Net::padded(16 * ng * 2);
  if (gout) bytes += 2 * Net::padded(16 * ng * 4) + Net::padded((size_t)kGwCtas * 16 * 16 * 27 * 4);
  BEM_TRY(n.reserve(bytes));
  for (float** p : {&n.w, &n.wf, &n.wb, &n.g}) BEM_TRY(n.alloc(p, n.nw));
  BEM_TRY(n.alloc(&n.act[0], 8 * ng));
  for (int l = 1; l < kLayers; ++l) BEM_TRY(n.alloc(&n.act[l], 16 * ng));
  n.out = out;
  BEM_CUDA(cudaMemcpyAsync(n.w, w_host, n.nw * sizeof(float), cudaMemcpyHostToDevice, s));
  k_to_bf16<<<(unsigned)((8 * ng + 255) / 256), 256, 0, s>>>(x, 8 * (int64_t)ng, n.act[0]);
  BEM_TRY(net_forward(n, d, s));
  if (gout) {
    BEM_TRY(n.alloc(&n.gbuf[0], 16 * ng));
    BEM_TRY(n.alloc(&n.gbuf[1], 16 * ng));
    BEM_TRY(n.alloc(&n.part, (size_t)kGwCtas * 16 * 16 * 27));
    BEM_CUDA(cudaMemsetAsync(n.g, 0, n.nw * sizeof(float), s));
    BEM_TRY(net_backward(n, d, gout, gx, s));
    if (gw_host) BEM_CUDA(cudaMemcpyAsync(gw_host, n.g, n.nw * sizeof(float), cudaMemcpyDeviceToHost, s));
  }
  BEM_CUDA(cudaStreamSynchronize(s));
  return BEM_OK;
}

}  // extern "C"
