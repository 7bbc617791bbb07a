// Sparse internal operators at high frequency (Sec. III-A, third item of the internal problem).
// When the skin depth delta_i = -1/Im k_i is small against an object, L_{k_i} and K_{k_i}
// couple each basis function only to its near neighbours: they are treated as sparse, the pairs
// whose RWG supports lie farther apart than R_cut = 23 delta_i dropped (e^{-23} ~ 1e-10; the
// support distance is bounded from below by the centroid distance less the two triangles'
// centroid-to-vertex radii, nearest of the 2 x 2 triangle pairs), and
//   e = Z_s h = -(1 / (j k0 eps_rc)) L_s^{-1} (K_s + I_x/2) h
// replaces the dense e = Z h of Eq. MFIEinZin. The paper applies L_s^{-1} with a sparse direct
// solver; here the kept pattern of each object is reordered by reverse Cuthill-McKee (host), so
// that L_s becomes a band of half-width b, factorised without pivoting in FP64 (one CTA per
// object), and each product is the sparse rows of K_s + I_x/2 (all objects in one launch) and
// then one CTA per object for a forward and a back substitution, blocked by W columns (each
// column of L and of U stored contiguously, the triangle of a diagonal block replaced by its
// inverse, a block's columns streamed into shared memory by one bulk copy while earlier blocks
// are worked on). C = Y_eq Z stays dense, so j = h - C h is unchanged and e = Z_s h, needed only
// by the I_x e term of the system matvec, runs beside it. The sparse form is used when every object
// qualifies (band and rows below half the dense bytes, b <= 192) and a set-up check of Z_s h
// against the dense FP64 Z h (one probe vector) stays below 1e-8, and below 1e-5 in FP32.
#include <algorithm>
#include <cmath>
#include <complex>
#include <memory>
#include <type_traits>
#include <vector>

#include "bulk.cuh"
#include "common.cuh"

namespace bem {

constexpr double kZspCut = 23.0;     // R_cut / delta
constexpr int kZspBandMax = 192;     // largest half-bandwidth of the product kernel
constexpr size_t kZspSmemMax = 220 * 1024;  // FP64 vector and two 8-column slabs (set-up limit)
constexpr size_t kZspSmemCta = 227 * 1024;  // shared memory of one CTA
constexpr int kZspThreads = 256;  // consumers; one more warp issues the copies
// columns per block of the substitutions: a step solves one block and updates the b rows beside
// it. 32 in FP32; 16 in FP64, where a step is bound by the FP64 rate and wider slabs only take
// shared memory (8 where the vector leaves no room for two 16-column slabs)
constexpr int kZspW32 = 32, kZspW64 = 16, kZspW64s = 8;
constexpr int kZspRing = 256;        // second accumulator, a ring over rows (>= 192 + 32)
constexpr int kZspStages = 3;        // slabs in flight (2 where shared memory leaves no room)
constexpr double kZspCheck = 1e-8;   // set-up check of Z_s h against Z h
constexpr double kZspCheck32 = 1e-5;  // that of the FP32 Z_s h, against the FP64 Z h
constexpr double kZspSame = 1e-13;  // below it Z_s h and Z h are the same product to FP64 rounding
constexpr double kTwoPi = 6.283185307179586476925;

struct ZspObj {
  int e0, n, b, pad;
  int64_t loff;   // offset of the object's n x b column tables of L and U
  int64_t woff;   // offset of its FP64 band (set-up only), n x (2b + 1)
  double ar, ai;  // alpha = -1 / (j k0 eps_rc)
};

struct Zsp {
  std::vector<ZspObj> obj;
  ZspObj* d_obj = nullptr;
  int32_t *d_perm = nullptr, *d_pos = nullptr;  // row e0 + r <-> edge e0 + perm[r], both global
  int32_t *d_row = nullptr, *d_col = nullptr;   // K_s + I_x/2 in permuted row order (CSR)
  int64_t nnz = 0, nband = 0, nwork = 0;
  int bmax = 0, bstore = 0, nmax = 0;  // largest half-bandwidth, largest stored one (>= 31)
  int w64 = kZspW64;                   // columns per block of the FP64 substitutions
  double2* W = nullptr;                          // FP64 bands during set-up
  double2 *kv64 = nullptr, *L64 = nullptr, *U64 = nullptr, *D64 = nullptr;
  float2 *kv32 = nullptr, *L32 = nullptr, *U32 = nullptr, *D32 = nullptr;
  int* d_fail = nullptr;
  int* d_err = nullptr;    // set by a product whose bounded wait timed out
  float2* v32 = nullptr;   // [kMaxBatch][ne] rows of K_s + I_x/2 h, permuted (product scratch)
  double2* v64 = nullptr;
  double check = -1, check32 = -1;  // max over objects of |Z_s h - Z h| / |Z h| at set-up, FP64 and FP32 Z_s
  ~Zsp() {
    if (W) cudaFree(W);
  }
};

// ---------------------------------------------------------------------------------------
// set-up kernels
// ---------------------------------------------------------------------------------------
__global__ void k_tri_radius(const double* verts, const int32_t* tris, const double* cen, int nt,
                             double* rad) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  double r = 0;
  for (int a = 0; a < 3; ++a) {
    const double* v = &verts[3 * tris[3 * t + a]];
    const double dx = v[0] - cen[3 * t], dy = v[1] - cen[3 * t + 1], dz = v[2] - cen[3 * t + 2];
    r = fmax(r, sqrt(dx * dx + dy * dy + dz * dz));
  }
  rad[t] = r;
}

// mask[m n + k] = 1 iff the supports of edges e0 + m and e0 + k come within rcut
__global__ void k_zsp_mask(const double* cen, const double* rad, const int32_t* et, int e0, int n,
                           double rcut, uint8_t* mask) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n * n) return;
  const int m = e0 + (int)(idx / n), k = e0 + (int)(idx % n);
  double d = 1e300;
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      const int t = et[2 * m + a], s = et[2 * k + b];
      const double dx = cen[3 * t] - cen[3 * s], dy = cen[3 * t + 1] - cen[3 * s + 1],
                   dz = cen[3 * t + 2] - cen[3 * s + 2];
      d = fmin(d, fmax(0.0, sqrt(dx * dx + dy * dy + dz * dz) - rad[t] - rad[s]));
    }
  mask[idx] = d <= rcut ? 1 : 0;
}

// the kept entries of L (band of the permuted matrix) and of B = K + I_x/2 (CSR values), from
// the object's dense column-major n x n matrices; one thread per permuted row
__global__ void k_zsp_gather(ZspObj o, const double2* L, const double2* B, const int32_t* perm,
                             const int32_t* pos, const int32_t* row, const int32_t* col,
                             double2* W, double2* kv) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= o.n) return;
  const int w = 2 * o.b + 1;
  const int node = perm[o.e0 + r] - o.e0;
  for (int k = row[o.e0 + r]; k < row[o.e0 + r + 1]; ++k) {
    const int cl = col[k] - o.e0;
    const int64_t src = node + (int64_t)cl * o.n;
    kv[k] = B[src];
    const int j = pos[col[k]] - o.e0;
    W[o.woff + (int64_t)r * w + (j - r + o.b)] = L[src];
  }
}

// LU without pivoting of each object's band (one CTA per object, in place, FP64): W[i][j - i + b]
// holds A_ij; afterwards the strict lower band holds L (unit diagonal) and the rest U.
__global__ void __launch_bounds__(256) k_zsp_lu(const ZspObj* objs, double2* Wall, int* fail) {
  const ZspObj o = objs[blockIdx.x];
  const int n = o.n, b = o.b, w = 2 * b + 1;
  double2* W = Wall + o.woff;
  __shared__ double2 lcol[kZspBandMax], urow[kZspBandMax];
  __shared__ double red[256];
  // scale: the largest diagonal magnitude
  double mx = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double2 d = W[(int64_t)i * w + b];
    mx = fmax(mx, sqrt(d.x * d.x + d.y * d.y));
  }
  red[threadIdx.x] = mx;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  const double tiny = 1e-13 * red[0];
  for (int k = 0; k < n; ++k) {
    const int m = min(b, n - 1 - k);  // rows (and columns) below (right of) the pivot in the band
    double2 p = W[(int64_t)k * w + b];
    const double pm = p.x * p.x + p.y * p.y;
    if (!(sqrt(pm) > tiny)) {
      if (threadIdx.x == 0) atomicExch(&fail[blockIdx.x], 1);
      p = make_double2(red[0], 0.0);
    }
    const double den = p.x * p.x + p.y * p.y;
    const double2 ip = make_double2(p.x / den, -p.y / den);
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
      double2* a = &W[(int64_t)(k + 1 + t) * w + (b - 1 - t)];  // A[k+1+t][k]
      const double2 l = cmul(*a, ip);
      *a = l;
      lcol[t] = l;
      urow[t] = W[(int64_t)k * w + (b + 1 + t)];  // A[k][k+1+t]
    }
    __syncthreads();
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
      const int i = t / m, j = t % m;  // row k+1+i, column k+1+j
      double2* a = &W[(int64_t)(k + 1 + i) * w + (j - i + b)];
      const double2 u = cmul(lcol[i], urow[j]);
      a->x -= u.x;
      a->y -= u.y;
    }
    __syncthreads();
  }
}

template <typename V> __device__ __forceinline__ V to_v(double2 a);
template <> __device__ __forceinline__ double2 to_v<double2>(double2 a) { return a; }
template <> __device__ __forceinline__ float2 to_v<float2>(double2 a) {
  return make_float2((float)a.x, (float)a.y);
}

// column tables for the substitutions: Lc[c][k] = L[c+1+k][c], Uc[c][k] = U[c-1-k][c] (zero
// outside the matrix), D[c] = 1 / U[c][c]; FP64 and FP32 copies
__global__ void k_zsp_extract(const ZspObj* objs, const double2* Wall, double2* L64, double2* U64,
                              double2* D64, float2* L32, float2* U32, float2* D32) {
  const ZspObj o = objs[blockIdx.y];
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int n = o.n, b = o.b, w = 2 * b + 1;
  if (idx >= (int64_t)n * b) return;
  const int c = (int)(idx / b), k = (int)(idx % b);
  const double2* W = Wall + o.woff;
  double2 l = make_double2(0, 0), u = make_double2(0, 0);
  if (c + 1 + k < n) l = W[(int64_t)(c + 1 + k) * w + (b - 1 - k)];
  if (c - 1 - k >= 0) u = W[(int64_t)(c - 1 - k) * w + (b + 1 + k)];
  L64[o.loff + idx] = l;
  U64[o.loff + idx] = u;
  L32[o.loff + idx] = make_float2((float)l.x, (float)l.y);
  U32[o.loff + idx] = make_float2((float)u.x, (float)u.y);
  if (k == 0) {
    const double2 d = W[(int64_t)c * w + b];
    const double den = d.x * d.x + d.y * d.y;
    const double2 id = make_double2(d.x / den, -d.y / den);
    D64[o.e0 + c] = id;
    D32[o.e0 + c] = make_float2((float)id.x, (float)id.y);
  }
}

// Inverses of the triangles inside the W-column diagonal blocks, in place of the triangles: the
// strict lower part of (L_ss)^-1 and the strict upper part of (U_ss)^-1 have as many entries as
// the triangles themselves, so the column tables keep their size and layout (the half-bandwidth
// stored is at least W - 1, so that a block's whole triangle lies in the band). A block's solve is
// then a product, not a chain of W dependent steps. From the FP64 factors; one CTA of 32 threads
// per block, one thread per column.
template <int W, typename V>
__global__ void __launch_bounds__(32) k_zsp_invtri(const ZspObj* objs, const double2* Wall, V* Lc,
                                                   V* Uc) {
  const ZspObj o = objs[blockIdx.y];
  const int n = o.n, b = o.b, w = 2 * b + 1, c0 = W * blockIdx.x;
  if (c0 >= n) return;
  const int nb = min(W, n - c0), t = threadIdx.x;
  const double2* A = Wall + o.woff;
  __shared__ double2 T[W][W + 1], X[W][W + 1];
  for (int i = t; i < nb * nb; i += 32) {
    const int r = i / nb, q = i % nb;
    T[r][q] = A[(int64_t)(c0 + r) * w + (q - r + b)];
  }
  __syncwarp();
  if (t < nb) {  // column t of the unit lower inverse
    X[t][t] = make_double2(1.0, 0.0);
    for (int r = t + 1; r < nb; ++r) {
      double2 acc = make_double2(0.0, 0.0);
      for (int q = t; q < r; ++q) cfma(acc, T[r][q], X[q][t]);
      X[r][t] = make_double2(-acc.x, -acc.y);
      Lc[o.loff + (int64_t)(c0 + t) * b + (r - t - 1)] = to_v<V>(X[r][t]);
    }
    // column t of the upper inverse
    auto inv = [](double2 d) {
      const double den = d.x * d.x + d.y * d.y;
      return make_double2(d.x / den, -d.y / den);
    };
    X[t][t] = inv(T[t][t]);
    for (int r = t - 1; r >= 0; --r) {
      double2 acc = make_double2(0.0, 0.0);
      for (int q = r + 1; q <= t; ++q) cfma(acc, T[r][q], X[q][t]);
      const double2 v = cmul(acc, inv(T[r][r]));
      X[r][t] = make_double2(-v.x, -v.y);
      Uc[o.loff + (int64_t)(c0 + t) * b + (t - r - 1)] = to_v<V>(X[r][t]);
    }
  }
}

__global__ void k_round_kv(const double2* a, float2* b, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_float2((float)a[i].x, (float)a[i].y);
}

// ---------------------------------------------------------------------------------------
// the product e = Z_s h in two launches: the rows of K_s + I_x/2 (all objects' rows in one
// launch, kZspLanes lanes per row), then the substitutions, one CTA per object and right-hand side,
// blocked by W columns: a block is solved as a product with its stored triangle inverse and its
// solved values are applied to the b rows below (above, going back).
// ---------------------------------------------------------------------------------------
template <typename V> __device__ __forceinline__ V vzero() { V v; v.x = 0; v.y = 0; return v; }
template <typename V> __device__ __forceinline__ V one() { V v; v.x = 1; v.y = 0; return v; }
template <typename V> __device__ __forceinline__ V vmul(V a, V b) {
  V r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
constexpr int kZspLanes = 16;  // lanes per row of K_s + I_x/2: four entries each in flight

// v[r] (permuted row r of every object, stride vs per right-hand side) = ((K_s + I_x/2) h)[perm r]
template <typename R>
__global__ void __launch_bounds__(256) k_zsp_rows(const int32_t* __restrict__ row,
                                                  const int32_t* __restrict__ col,
                                                  const typename C2<R>::T* __restrict__ kv,
                                                  const typename C2<R>::T* __restrict__ x, int64_t xs,
                                                  typename C2<R>::T* __restrict__ v, int64_t vs,
                                                  int ne) {
  typedef typename C2<R>::T V;
  const int r = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kZspLanes);
  const int sub = threadIdx.x & (kZspLanes - 1);
  const V* h = x + blockIdx.y * xs;
  V acc = vzero<V>();
  if (r < ne) {
    const int k1 = row[r + 1];
    for (int k = row[r] + sub; k < k1; k += 4 * kZspLanes) {
      // the missing entries of a short last group repeat its first column, with value 0
      int c[4];
      V a[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kk = k + q * kZspLanes;
        c[q] = col[kk < k1 ? kk : k];
        a[q] = kk < k1 ? kv[kk] : vzero<V>();
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(acc, a[q], h[c[q]]);
    }
  }
#pragma unroll
  for (int o = kZspLanes / 2; o > 0; o >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
  }
  if (r < ne && sub == 0) v[blockIdx.y * vs + r] = acc;
}

// One CTA per (right-hand side, object). The serial chain is 2 n / W block steps; a step is two
// products out of shared memory with a barrier after each:
//   solve   x_s = T_s^-1 r_s, eight lanes per row
//   update  r -= (the W columns of the band beside the block) x_s, one lane per row, the columns
//           split between the two halves of the CTA; the halves add into two accumulators (the
//           vector, and a ring of kZspRing rows that covers the band), so they need no reduction
// The slabs of W columns (contiguous, W b entries) arrive by bulk copies kept nst - 1 blocks
// ahead. FP32: bound by moving a ring's 1.7 MB of tables through one SM (13 us at 64 B a clock)
// when rings are few and by HBM when they fill the GPU; FP64 by the FP64 rate (0.2 ms a ring).
// One warp per ring and 8-column blocks solved by shuffles, the form before, was one chain of
// 2 n / 8 steps: e = Z_s h of rings of 912 edges (b = 114), k_zsp_rows included, took 297 us for
// 1 ring, 306 for 36, 380 for 256 (FP64 2,810, 2,895, 3,187 us); now 57, 64, 125 us (FP64 408, 453,
// 979). 2 to 7 slabs in flight take the same time.
// Every wait is bounded; a timeout sets *err and ends the CTA once its copies have landed.
template <typename R, int W>
__global__ void __launch_bounds__(kZspThreads + 32) k_zsp_solve(
    const ZspObj* __restrict__ objs, const int32_t* __restrict__ perm,
    const typename C2<R>::T* __restrict__ Lc, const typename C2<R>::T* __restrict__ Uc,
    const typename C2<R>::T* __restrict__ D, const typename C2<R>::T* __restrict__ vin, int64_t vs,
    typename C2<R>::T* __restrict__ y, int64_t ys, int vbytes, int slab_bytes, int nst, int* err) {
  typedef typename C2<R>::T V;
  extern __shared__ __align__(16) unsigned char zsp_smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(zsp_smem);  // [nst], nst <= 8
  V* xs = reinterpret_cast<V*>(zsp_smem + 64);            // the block's solved values [W]
  V* v1 = xs + W;                                         // second accumulator [kZspRing]
  V* v = v1 + kZspRing;                                   // the running vector
  unsigned char* slabs = reinterpret_cast<unsigned char*>(v) + vbytes;  // nst slots of slab_bytes
  const ZspObj o = objs[blockIdx.y];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = o.n, b = o.b, e0 = o.e0;
  const V* Lo = Lc + o.loff;
  const V* Uo = Uc + o.loff;
  const int nblk = (n + W - 1) / W, nslab = 2 * nblk;
  // slab s: L's columns of block s (forward), then U's of block 2 nblk - 1 - s (going back)
  auto issue = [&](int s, int slot) {
    const int kb = s < nblk ? s : nslab - 1 - s;
    const int c0 = W * kb, nb = min(W, n - c0);
    const uint32_t bytes = (uint32_t)(((size_t)nb * b * sizeof(V) + 15) & ~(size_t)15);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads of the slot
    mbar_arrive_tx(&bar[slot], bytes);
    bulk_g2s(slabs + (size_t)slot * slab_bytes, (s < nblk ? Lo : Uo) + (int64_t)c0 * b, bytes, &bar[slot]);
  };
  const bool producer = tid == kZspThreads;
  if (producer) {
    for (int q = 0; q < nst; ++q) mbar_init(&bar[q], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int q = 0; q < nst && q < nslab; ++q) issue(q, q);
  }
  const V* vi = vin + blockIdx.x * vs + e0;
  for (int r = tid; r < n; r += kZspThreads + 32) v[r] = vi[r];
  for (int r = tid; r < kZspRing; r += kZspThreads + 32) v1[r] = vzero<V>();
  __syncthreads();
  if (warp == kZspThreads / 32) {  // the copies: their issue stays off the consumers' chain
    for (int s = 0; s < nslab; ++s) {
      if (__syncthreads_or(0)) return;
      __syncthreads();
      if (producer && s + nst < nslab) issue(s + nst, s % nst);
    }
    return;
  }
  const int row = tid >> 3, sub = tid & 7;          // solve: row of the block, lane of the row
  const int half = warp >> 2, i0 = (warp & 3) * 32 + lane;  // update: column half, row
  int slot = 0, phase = 0;
  V dn = vzero<V>();  // 1 / U_rr of this thread's row in the next block (read one step ahead)
  auto step = [&](int s, auto dir) -> bool {
    constexpr bool kFwd = decltype(dir)::value;
    const bool ok = mbar_wait(&bar[slot], phase);
    const V* S = reinterpret_cast<const V*>(slabs + (size_t)slot * slab_bytes);  // S[t b + k]: column t, entry k
    const int c0 = W * (kFwd ? s : nslab - 1 - s), nb = min(W, n - c0);
    const V dr = dn;
    if (s + 1 >= nblk && s + 1 < nslab) dn = D[e0 + min(n - 1, W * (nslab - 2 - s) + row)];
    // loads are unconditional (their addresses stay inside this CTA's shared memory) and what
    // does not belong is dropped afterwards, so that a thread's loads are all in flight at once
    V acc = vzero<V>();
    if (row < W) {
#pragma unroll
      for (int q = 0; q < W / 8; ++q) {
        const int t = sub + 8 * q;
        V r = v[c0 + t];
        const V r1 = v1[(c0 + t) & (kZspRing - 1)];
        r.x += r1.x;
        r.y += r1.y;
        const int k = kFwd ? row - t - 1 : t - row - 1;
        V a = S[t * b + max(k, 0)];
        if (t == row) a = kFwd ? one<V>() : dr;
        if (k >= -1 && t < nb && row < nb) cfma(acc, a, r);
      }
    }
#pragma unroll
    for (int q = 4; q > 0; q >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, q);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, q);
    }
    if (sub == 0 && row < W) xs[row] = acc;
    if (__syncthreads_or(!ok)) {
      if (tid == 0) {
        atomicExch(err, 1);
        for (int q = 1; q < nst && s + q < nslab; ++q) {  // the copies in flight
          const int sl = (slot + q) % nst;
          mbar_wait(&bar[sl], sl > slot ? phase : phase ^ 1);
        }
      }
      return false;
    }
    const int live = min(b, kFwd ? n - c0 - W : c0);  // rows beside the block (none below a short one)
    for (int i = i0; i < live; i += 128) {
      // entry k = W - 1 + i - t below the block, t + i above it; k < b belongs to column t
      const int st = kFwd ? b - 1 : b + 1;
      const V* p = S + half * (W / 2) * st + (kFwd ? W - 1 + i : i);
      const int tlo = W + i - b - half * (W / 2), thi = min(nb, b - i) - half * (W / 2);
      const V* x = xs + half * (W / 2);
      V c[2] = {vzero<V>(), vzero<V>()};
#pragma unroll
      for (int q = 0; q < W / 2; ++q) {
        const V a = p[q * st];
        if (kFwd ? q >= tlo : q < thi) cfma(c[q & 1], a, x[q]);
      }
      const int g = kFwd ? c0 + W + i : c0 - 1 - i;
      V* u = half ? &v1[g & (kZspRing - 1)] : &v[g];
      u->x -= c[0].x + c[1].x;
      u->y -= c[0].y + c[1].y;
    }
    if (tid < nb) {
      const V x = xs[tid];
      v1[(c0 + tid) & (kZspRing - 1)] = vzero<V>();
      v[c0 + tid] = x;
    }
    __syncthreads();
    if (++slot == nst) {
      slot = 0;
      phase ^= 1;
    }
    return true;
  };
  for (int s = 0; s < nblk; ++s)
    if (!step(s, std::true_type())) return;
  for (int s = nblk; s < nslab; ++s)
    if (!step(s, std::false_type())) return;
  V al;
  al.x = (R)o.ar;
  al.y = (R)o.ai;
  V* e = y + blockIdx.x * ys;
  for (int r = tid; r < n; r += kZspThreads) e[perm[e0 + r]] = vmul(al, v[r]);
}

// shared memory of k_zsp_solve with nst slabs of w columns
template <typename V> static size_t zsp_smem_bytes(const Zsp* z, int w, int nst) {
  const size_t vbytes = ((size_t)z->nmax * sizeof(V) + 15) & ~(size_t)15;
  return 64 + (size_t)(w + kZspRing) * sizeof(V) + vbytes + ((size_t)nst * w * z->bstore + w) * sizeof(V);  // + w: reads past the last slab, dropped
}

template <typename R>
int zsp_apply(aim_ctx* c, const typename C2<R>::T* h, typename C2<R>::T* e, int nrhs, int64_t hs,
              int64_t es, cudaStream_t s) {
  typedef typename C2<R>::T V;
  Zsp* z = static_cast<Zsp*>(c->zsp);
  if (!z || !c->zsp_ready) {
    set_error("sparse internal operator not built");
    return BEM_EINVAL;
  }
  if (nrhs < 1 || nrhs > kMaxBatch) {
    set_error("sparse internal operator: 1 <= nrhs <= %d", kMaxBatch);
    return BEM_EINVAL;
  }
  const bool f = sizeof(R) == 4;
  V* v = f ? (V*)z->v32 : (V*)z->v64;
  const int ne = c->ne;
  k_zsp_rows<R><<<dim3((unsigned)(((int64_t)ne * kZspLanes + 255) / 256), nrhs), 256, 0, s>>>(
      z->d_row, z->d_col, f ? (const V*)z->kv32 : (const V*)z->kv64, h, hs, v, ne, ne);
  const int w = f ? kZspW32 : z->w64;
  const int nst = zsp_smem_bytes<V>(z, w, kZspStages) <= kZspSmemCta ? kZspStages : 2;
  const size_t sm = zsp_smem_bytes<V>(z, w, nst);
  const int vbytes = (int)(((size_t)z->nmax * sizeof(V) + 15) & ~(size_t)15);
  const int slab_bytes = w * z->bstore * (int)sizeof(V);
  auto launch = [&](auto* kernel) -> int {
    // per call: the attribute belongs to the current device
    BEM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    // the right-hand sides of one object next to each other: they share its tables in L2
    kernel<<<dim3(nrhs, (unsigned)z->obj.size()), kZspThreads + 32, sm, s>>>(
        z->d_obj, z->d_perm, f ? (const V*)z->L32 : (const V*)z->L64,
        f ? (const V*)z->U32 : (const V*)z->U64, f ? (const V*)z->D32 : (const V*)z->D64, v, ne, e,
        es, vbytes, slab_bytes, nst, z->d_err);
    return BEM_OK;
  };
  if constexpr (sizeof(R) == 4) BEM_TRY(launch(&k_zsp_solve<R, kZspW32>));
  else if (z->w64 == kZspW64) BEM_TRY(launch(&k_zsp_solve<R, kZspW64>));
  else BEM_TRY(launch(&k_zsp_solve<R, kZspW64s>));
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

template int zsp_apply<float>(aim_ctx*, const float2*, float2*, int, int64_t, int64_t, cudaStream_t);
template int zsp_apply<double>(aim_ctx*, const double2*, double2*, int, int64_t, int64_t,
                               cudaStream_t);

// ---------------------------------------------------------------------------------------
// set-up
// ---------------------------------------------------------------------------------------
// reverse Cuthill-McKee order of a symmetric pattern (adjacency lists, self loops ignored):
// breadth-first from a minimum-degree vertex of each component, neighbours taken in increasing
// degree, the whole order reversed (Cuthill and McKee 1969; George's reversal)
static std::vector<int> rcm_order(int n, const std::vector<int>& rp, const std::vector<int>& ci) {
  std::vector<int> deg(n), order;
  order.reserve(n);
  for (int i = 0; i < n; ++i) deg[i] = rp[i + 1] - rp[i];
  std::vector<char> seen(n, 0);
  std::vector<int> byd(n);
  for (int i = 0; i < n; ++i) byd[i] = i;
  std::stable_sort(byd.begin(), byd.end(), [&](int a, int b) { return deg[a] < deg[b]; });
  std::vector<int> nb;
  for (int start : byd) {
    if (seen[start]) continue;
    size_t head = order.size();
    order.push_back(start);
    seen[start] = 1;
    while (head < order.size()) {
      const int v = order[head++];
      nb.clear();
      for (int k = rp[v]; k < rp[v + 1]; ++k)
        if (!seen[ci[k]]) {
          seen[ci[k]] = 1;
          nb.push_back(ci[k]);
        }
      std::stable_sort(nb.begin(), nb.end(), [&](int a, int b) { return deg[a] < deg[b]; });
      order.insert(order.end(), nb.begin(), nb.end());
    }
  }
  std::reverse(order.begin(), order.end());
  return order;
}

void free_zsp(aim_ctx* c) {
  delete static_cast<Zsp*>(c->zsp);
  c->zsp = nullptr;
  c->zsp_ready = false;
  c->zsp_on = false;
  c->zsp64_dense = 0;
}

int zsp_prepare(aim_ctx* c, const double* d_verts, const int32_t* d_tris, const double* d_cen) {
  const int nobj = c->nobj;
  const double w = kTwoPi * c->freq;
  std::vector<double> rcut(nobj);
  int64_t dense = 0, nmax = 0;
  for (int i = 0; i < nobj; ++i) {
    const bem_material& mt = c->mat[i];
    std::complex<double> epsc(mt.eps_r, -mt.sigma / (w * kEps0));
    std::complex<double> ki = c->k0 * std::sqrt(epsc * mt.mu_r);
    if (ki.imag() > 0) ki = -ki;
    if (!(ki.imag() < 0)) return BEM_OK;  // lossless: no skin depth
    rcut[i] = kZspCut / -ki.imag();
    // extent of the object: no sparsity to find when R_cut spans it
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    for (int t = c->t0[i]; t < c->t1[i]; ++t)
      for (int a = 0; a < 3; ++a)
        for (int q = 0; q < 3; ++q) {
          const double v = c->verts[3 * (size_t)c->tris[3 * (size_t)t + a] + q];
          lo[q] = std::min(lo[q], v);
          hi[q] = std::max(hi[q], v);
        }
    const double ext = std::sqrt((hi[0] - lo[0]) * (hi[0] - lo[0]) + (hi[1] - lo[1]) * (hi[1] - lo[1]) +
                                 (hi[2] - lo[2]) * (hi[2] - lo[2]));
    if (rcut[i] >= 0.5 * ext) return BEM_OK;
    const int64_t n = c->e1[i] - c->e0[i];
    dense += n * n;
    nmax = std::max(nmax, n);
  }
  if (nmax * (int64_t)sizeof(double2) > 200 * 1024) return BEM_OK;  // vector beyond shared memory
  double* rad = nullptr;
  uint8_t* dmask = nullptr;
  BEM_CUDA(cudaMalloc(&rad, c->nt * sizeof(double)));
  std::unique_ptr<void, decltype(&cudaFree)> hold_rad(rad, &cudaFree);
  BEM_CUDA(cudaMalloc(&dmask, nmax * nmax));
  std::unique_ptr<void, decltype(&cudaFree)> hold_mask(dmask, &cudaFree);
  k_tri_radius<<<(c->nt + 255) / 256, 256>>>(d_verts, d_tris, d_cen, c->nt, rad);
  BEM_CUDA(cudaGetLastError());
  Zsp* z = new Zsp();
  std::unique_ptr<Zsp> hold(z);
  std::vector<int32_t> perm(c->ne), pos(c->ne), row(c->ne + 1, 0), col;
  std::vector<uint8_t> mask(nmax * nmax);
  std::vector<int> rp, ci;
  int64_t nband = 0, nband_true = 0, nwork = 0;
  for (int i = 0; i < nobj; ++i) {
    const int e0 = c->e0[i], n = c->e1[i] - e0;
    k_zsp_mask<<<(unsigned)(((int64_t)n * n + 255) / 256), 256>>>(d_cen, rad, c->d_et, e0, n,
                                                                   rcut[i], dmask);
    BEM_CUDA(cudaGetLastError());
    BEM_CUDA(cudaMemcpy(mask.data(), dmask, (size_t)n * n, cudaMemcpyDeviceToHost));
    rp.assign(n + 1, 0);
    ci.clear();
    for (int m = 0; m < n; ++m) {
      for (int k = 0; k < n; ++k)
        if (mask[(size_t)m * n + k] && k != m) ci.push_back(k);
      rp[m + 1] = (int)ci.size();
    }
    const std::vector<int> ord = rcm_order(n, rp, ci);
    std::vector<int> p(n);
    for (int r = 0; r < n; ++r) p[ord[r]] = r;
    int b = 0;
    for (int m = 0; m < n; ++m)
      for (int k = rp[m]; k < rp[m + 1]; ++k) b = std::max(b, std::abs(p[m] - p[ci[k]]));
    if (b > kZspBandMax) return BEM_OK;
    b = std::max(b, 1);
    z->bmax = std::max(z->bmax, b);
    nband_true += ((int64_t)n * b + 1) & ~(int64_t)1;
    b = std::max(b, kZspW32 - 1);  // a block's triangle lies in the stored band (k_zsp_invtri)
    ZspObj o;
    o.e0 = e0;
    o.n = n;
    o.b = b;
    o.pad = 0;
    o.loff = nband;
    o.woff = nwork;
    std::complex<double> epsc(c->mat[i].eps_r, -c->mat[i].sigma / (w * kEps0));
    const std::complex<double> al = -1.0 / (std::complex<double>(0.0, c->k0) * epsc);
    o.ar = al.real();
    o.ai = al.imag();
    z->obj.push_back(o);
    nband += ((int64_t)n * b + 1) & ~(int64_t)1;  // even: 16-byte aligned FP32 slabs
    nwork += (int64_t)n * (2 * b + 1);
    z->bstore = std::max(z->bstore, b);
    for (int r = 0; r < n; ++r) {
      perm[e0 + r] = e0 + ord[r];
      pos[e0 + ord[r]] = e0 + r;
      const int m = ord[r];
      col.push_back(e0 + m);  // the diagonal, then the other kept columns
      for (int k = rp[m]; k < rp[m + 1]; ++k) col.push_back(e0 + ci[k]);
      row[e0 + r + 1] = (int32_t)col.size();
    }
  }
  // room for the FP64 vector and two slabs of 8 columns
  if (16 + ((nmax * 16 + 15) & ~(int64_t)15) + 2 * kZspW64s * (int64_t)z->bmax * 16 > (int64_t)kZspSmemMax)
    return BEM_OK;
  // worth it only below half the dense bytes (FP32: band tables, diagonal, rows and columns)
  const int64_t sparse_b = 2 * nband_true * 8 + (int64_t)c->ne * 8 + (int64_t)col.size() * 12;
  if (sparse_b > 4 * dense) return BEM_OK;
  z->nnz = (int64_t)col.size();
  z->nband = nband;
  z->nwork = nwork;
  z->nmax = (int)nmax;
  z->w64 = zsp_smem_bytes<double2>(z, kZspW64, 2) <= kZspSmemCta ? kZspW64 : kZspW64s;
  BEM_TRY(upload(c, &z->d_obj, z->obj.data(), z->obj.size()));
  BEM_TRY(upload(c, &z->d_perm, perm.data(), perm.size()));
  BEM_TRY(upload(c, &z->d_pos, pos.data(), pos.size()));
  BEM_TRY(upload(c, &z->d_row, row.data(), row.size()));
  BEM_TRY(upload(c, &z->d_col, col.data(), col.size()));
  BEM_TRY(dalloc_t(c, &z->kv64, z->nnz));
  BEM_TRY(dalloc_t(c, &z->kv32, z->nnz));
  // two spare entries: a slab's copy is rounded up to 16 bytes
  BEM_TRY(dalloc_t(c, &z->L64, nband + 2));
  BEM_TRY(dalloc_t(c, &z->U64, nband + 2));
  BEM_TRY(dalloc_t(c, &z->D64, c->ne));
  BEM_TRY(dalloc_t(c, &z->L32, nband + 2));
  BEM_TRY(dalloc_t(c, &z->U32, nband + 2));
  BEM_TRY(dalloc_t(c, &z->D32, c->ne));
  BEM_TRY(dalloc_t(c, &z->d_fail, z->obj.size()));
  BEM_TRY(dalloc_t(c, &z->d_err, 1));
  BEM_CUDA(cudaMemset(z->d_err, 0, sizeof(int)));
  BEM_TRY(dalloc_t(c, &z->v32, (size_t)kMaxBatch * c->ne));
  BEM_TRY(dalloc_t(c, &z->v64, (size_t)kMaxBatch * c->ne));
  BEM_CUDA(cudaMemset(z->d_fail, 0, z->obj.size() * sizeof(int)));
  BEM_CUDA(cudaMalloc(&z->W, nwork * sizeof(double2)));
  BEM_CUDA(cudaMemset(z->W, 0, nwork * sizeof(double2)));
  c->zsp = hold.release();
  return BEM_OK;
}

int zsp_gather(aim_ctx* c, int obj, const double2* L, const double2* B) {
  Zsp* z = static_cast<Zsp*>(c->zsp);
  if (!z || !z->W) return BEM_OK;
  const ZspObj& o = z->obj[obj];
  k_zsp_gather<<<(o.n + 127) / 128, 128>>>(o, L, B, z->d_perm, z->d_pos, z->d_row, z->d_col, z->W,
                                           z->kv64);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

int zsp_factor(aim_ctx* c) {
  Zsp* z = static_cast<Zsp*>(c->zsp);
  if (!z || !z->W) return BEM_OK;
  const int nobj = (int)z->obj.size();
  k_zsp_lu<<<nobj, 256>>>(z->d_obj, z->W, z->d_fail);
  BEM_CUDA(cudaGetLastError());
  int64_t mx = 0;
  for (const ZspObj& o : z->obj) mx = std::max(mx, (int64_t)o.n * o.b);
  k_zsp_extract<<<dim3((unsigned)((mx + 255) / 256), nobj), 256>>>(z->d_obj, z->W, z->L64, z->U64,
                                                                   z->D64, z->L32, z->U32, z->D32);
  const auto blocks = [&](int w) { return dim3((unsigned)((z->nmax + w - 1) / w), nobj); };
  k_zsp_invtri<kZspW32, float2><<<blocks(kZspW32), 32>>>(z->d_obj, z->W, z->L32, z->U32);
  if (z->w64 == kZspW64)
    k_zsp_invtri<kZspW64, double2><<<blocks(kZspW64), 32>>>(z->d_obj, z->W, z->L64, z->U64);
  else
    k_zsp_invtri<kZspW64s, double2><<<blocks(kZspW64s), 32>>>(z->d_obj, z->W, z->L64, z->U64);
  k_round_kv<<<(unsigned)((z->nnz + 255) / 256), 256>>>(z->kv64, z->kv32, z->nnz);
  BEM_CUDA(cudaGetLastError());
  std::vector<int> fail(nobj);
  BEM_CUDA(cudaMemcpy(fail.data(), z->d_fail, nobj * sizeof(int), cudaMemcpyDeviceToHost));
  cudaFree(z->W);
  z->W = nullptr;
  for (int f : fail)
    if (f) {  // a vanishing pivot: the dense form stays
      free_zsp(c);
      return BEM_OK;
    }
  return BEM_OK;
}

__global__ void k_zsp_probe(double2* h, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint64_t v = (uint64_t)i * 0x9E3779B97F4A7C15ull + 0xD1B54A32D192ED03ull;
  v ^= v >> 31;
  v *= 0xBF58476D1CE4E5B9ull;
  v ^= v >> 29;
  h[i] = make_double2((double)(v >> 40) / 8388608.0 - 1.0, (double)((v >> 8) & 0xFFFFFF) / 8388608.0 - 1.0);
}

// largest over the objects of |a - d| / |d|
template <typename V> static double zsp_worst(const Zsp* z, const std::vector<V>& a, const std::vector<double2>& d) {
  double worst = 0;
  for (const ZspObj& o : z->obj) {
    double num = 0, den = 0;
    for (int r = o.e0; r < o.e0 + o.n; ++r) {
      const double dx = a[r].x - d[r].x, dy = a[r].y - d[r].y;
      num += dx * dx + dy * dy;
      den += d[r].x * d[r].x + d[r].y * d[r].y;
    }
    const double q = num == 0 ? 0.0 : std::sqrt(num / den);
    if (!(q <= worst) && worst == worst) worst = q;  // a NaN stays
  }
  return worst;
}

// Z_s h against the dense Z h (FP64) for one probe vector, whose entries FP32 holds exactly; the
// sparse form is kept when every object agrees to kZspCheck in FP64 and to kZspCheck32 in FP32,
// which has tables of its own (wider blocks, whose inverses are rounded)
int zsp_check(aim_ctx* c) {
  Zsp* z = static_cast<Zsp*>(c->zsp);
  if (!z) return BEM_OK;
  const int ne = c->ne;
  double2* h = nullptr;
  BEM_CUDA(cudaMalloc(&h, 4 * (size_t)ne * sizeof(double2)));
  std::unique_ptr<void, decltype(&cudaFree)> hold(h, &cudaFree);
  double2 *e1 = h + ne, *e2 = h + 2 * (size_t)ne;
  float2 *h32 = reinterpret_cast<float2*>(h + 3 * (size_t)ne), *e32 = h32 + ne;
  k_zsp_probe<<<(ne + 255) / 256, 256>>>(h, ne);
  k_round_kv<<<(ne + 255) / 256, 256>>>(h, h32, ne);
  c->zsp_ready = true;
  int rc = zsp_apply<double>(c, h, e1, 1, ne, ne, 0);
  if (rc == BEM_OK) rc = zsp_apply<float>(c, h32, e32, 1, ne, ne, 0);
  if (rc == BEM_OK) rc = run_gemv_plan<double>(c->gplan64, c->f64.Z, h, e2, 1, ne, nullptr, 0);
  if (rc != BEM_OK) {
    free_zsp(c);
    return rc;
  }
  std::vector<double2> a(ne), d(ne);
  std::vector<float2> f(ne);
  int err = 0;
  BEM_CUDA(cudaMemcpy(&err, z->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (err) {  // a bounded wait of the product timed out: keep the dense form
    free_zsp(c);
    return BEM_OK;
  }
  BEM_CUDA(cudaMemcpy(a.data(), e1, ne * sizeof(double2), cudaMemcpyDeviceToHost));
  BEM_CUDA(cudaMemcpy(f.data(), e32, ne * sizeof(float2), cudaMemcpyDeviceToHost));
  BEM_CUDA(cudaMemcpy(d.data(), e2, ne * sizeof(double2), cudaMemcpyDeviceToHost));
  z->check = zsp_worst(z, a, d);
  z->check32 = zsp_worst(z, f, d);
  if (!(z->check <= kZspCheck && z->check32 <= kZspCheck32)) {
    free_zsp(c);
    return BEM_OK;
  }
  c->zsp_on = true;
  return BEM_OK;
}

// FP64: an object's substitutions are bound by the FP64 rate of the one SM they run on, the dense
// product by the whole GPU's, so few objects are faster dense (4 rings of 912 edges 35 us against 413,
// 36 rings 282 / 453, 256 rings 2,000 / 979). For every number of vectors of the system products both
// forms are timed (best of three launches after a first one); the dense one is taken where it is the
// faster, both are the same product to rounding, and no caller chose the sparse form.
int zsp_time(aim_ctx* c) {
  Zsp* z = static_cast<Zsp*>(c->zsp);
  if (!z || !c->zsp_on || !(z->check <= kZspSame)) return BEM_OK;
  const int ne = c->ne;
  double2* h = nullptr;
  BEM_CUDA(cudaMalloc(&h, 2 * (size_t)kMaxBatch * ne * sizeof(double2)));
  std::unique_ptr<void, decltype(&cudaFree)> hold(h, &cudaFree);
  double2* e = h + (size_t)kMaxBatch * ne;
  k_zsp_probe<<<(kMaxBatch * ne + 255) / 256, 256>>>(h, kMaxBatch * ne);
  cudaEvent_t ev[2] = {nullptr, nullptr};
  int rc = BEM_OK;
  cudaError_t err = cudaEventCreate(&ev[0]);
  if (err == cudaSuccess) err = cudaEventCreate(&ev[1]);
  for (int r = 1; r <= kMaxBatch && rc == BEM_OK && err == cudaSuccess; ++r) {
    float best[2] = {1e30f, 1e30f};
    for (int k = 0; k < 8 && rc == BEM_OK && err == cudaSuccess; ++k) {  // in turn: sparse, dense
      cudaEventRecord(ev[0], 0);
      if (k % 2 == 0) rc = zsp_apply<double>(c, h, e, r, ne, ne, 0);
      else if (r > 1 && c->gmr.ntasks > 0) rc = run_gemv_mr<double>(c->gmr, c->f64.Z, h, e, r, ne, nullptr, 0);
      else rc = run_gemv_plan<double>(c->gplan64, c->f64.Z, h, e, r, ne, nullptr, 0);
      cudaEventRecord(ev[1], 0);
      err = cudaEventSynchronize(ev[1]);
      float ms = 1e30f;
      if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, ev[0], ev[1]);
      if (k >= 2) best[k % 2] = std::min(best[k % 2], ms);
    }
    if (best[1] < best[0]) c->zsp64_dense |= 1u << r;
  }
  for (cudaEvent_t q : ev)
    if (q) cudaEventDestroy(q);
  BEM_TRY(rc);
  BEM_CUDA(err);
  return BEM_OK;
}

void zsp_stats(const aim_ctx* c, int64_t* out) {
  const Zsp* z = static_cast<const Zsp*>(c->zsp);
  if (!z || !c->zsp_ready) {
    out[0] = 0;
    out[1] = 0;
    out[2] = 0;
    out[3] = 0;
    out[4] = -1;
    out[5] = 0;
    out[6] = -1;
    return;
  }
  out[0] = (int64_t)z->obj.size();
  out[1] = c->zsp_on ? 1 : 0;
  out[2] = z->bmax;
  out[3] = 2 * z->nband * 8 + (int64_t)c->ne * 8 + z->nnz * 12;
  out[4] = (int64_t)(z->check * 1e15);
  out[6] = (int64_t)(z->check32 * 1e12);
  int err = 0;  // set by a product whose bounded wait timed out
  if (cudaMemcpy(&err, z->d_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) err = -1;
  out[5] = err;
}

}  // namespace bem

extern "C" int bem_rcm_order(int n, const int32_t* rowptr, const int32_t* cols, int32_t* order) {
  if (n < 0 || (n > 0 && (!rowptr || !order || (rowptr[n] > 0 && !cols)))) {
    bem::set_error("bem_rcm_order: bad arguments");
    return BEM_EINVAL;
  }
  std::vector<int> rp(n + 1, 0), ci;  // the pattern without self loops
  for (int i = 0; i < n; ++i) {
    if (rowptr[i + 1] < rowptr[i]) {
      bem::set_error("bem_rcm_order: row pointers decrease at row %d", i);
      return BEM_EINVAL;
    }
    for (int k = rowptr[i]; k < rowptr[i + 1]; ++k) {
      if (cols[k] < 0 || cols[k] >= n) {
        bem::set_error("bem_rcm_order: column %d out of range at row %d", cols[k], i);
        return BEM_EINVAL;
      }
      if (cols[k] != i) ci.push_back(cols[k]);
    }
    rp[i + 1] = (int)ci.size();
  }
  const std::vector<int> ord = bem::rcm_order(n, rp, ci);
  for (int i = 0; i < n; ++i) order[i] = ord[i];
  return BEM_OK;
}
