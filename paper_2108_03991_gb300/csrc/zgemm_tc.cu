// Many right-hand sides through the internal blocks on the 5th-generation tensor cores: the
// products e_r = Z h_r and h_eq,r = C h_r (C = Y_eq Z, Eqs. MFIEinZin, EFIEeqYZ; block diagonal
// over the objects, Sec. II-C) for r = 1..R in one pass over each block, as the dense complex
// GEMM the internal problem becomes when many port excitations (Sec. IV) share the matrices.
//
// A complex product is one real GEMM. Row m of a block, stored as interleaved (re, im) FP32,
// is a real row of length 2n; right-hand side r contributes two real columns of B,
//   column 2r     = (Re x_0, -Im x_0, Re x_1, -Im x_1, ...)   (gives Re y_r),
//   column 2r + 1 = ( Im x_0,  Re x_0,  Im x_1,  Re x_1, ...)   (gives Im y_r),
// so D = A_real B (M = n, K = 2n, N = 2R) holds y_r as the (re, im) pair of columns 2r, 2r + 1.
//
// FP32 accuracy from BF16 tensor cores by a three-part split: a = a1 + a2 + a3, a1 the leading 8
// significant bits of the FP32 value (truncated), a2 the nearest BF16 value of the rest, a3 what is
// left, which BF16 holds exactly: all 24 bits, at every magnitude, since BF16 has FP32's exponents.
// D = A1 B1 + (A1 B2 + A2 B1 + A2 B2 + A1 B3 + A3 B1) in FP32; the dropped A2 B3 + A3 B2 is below 2^-22.
// (Two scaled FP16 parts, 22 bits, need half the MMAs, but entries far below the largest of their row
// or slice lose bits: 5 exponent bits. A column of Z falls by 2^-100 along a bar of 30 skin depths, and
// a unit vector's product has to return it.) Two TF32 parts take as many MMAs and more shared memory.
//
// Layout. B is packed once per call from x, stage by stage as shared memory holds it: [stage][3
// parts][NP rows][64 bytes, swizzled], every object's stages (32 values each, zeros past the object's 2 n)
// one after another, so that a stage is one contiguous bulk copy. (Rows of all objects' K values behind a
// tensor map put a stage's rows megabytes apart: C of 1,024 rings with 64 right-hand sides took
// 5.3 ms instead of 2.25.) A is read in place through one 2-D tensor map per object (inner extent 2n floats,
// rows n, row pitch 8 ld bytes): TMA fills the K tail and the rows past n with zeros; the landed FP32
// tile is turned in place into rows of 32 first parts and 32 second parts, its third parts go to a tile
// beside it. Shared-memory tiles are K-major; rows of 128 bytes (A) have the 128-byte swizzle, rows of 64
// bytes (A3, B) the 64-byte one. The parts of B follow each other, so that one MMA multiplies A1 by two
// or three of them.
//
// A product is bound by shared memory (a stage of 32 K values moves 168 KB through it at N = 128: the
// landing tiles, the conversion, the operands of 10 MMAs) and by the HBM reads of the blocks, so both
// matrices go in one launch of persistent CTAs and the K loops of the tiles are cut into units that
// load them evenly (tc_units). Z and C together, packing included (us, 64 right-hand sides): six bars of
// 240-1,920 edges 78, one bar of 2,016 45, 16 rings of 912 90 (257, 263, 144 with one launch per matrix
// and a CTA per tile in TF32; 69, 40, 72 with two FP16 parts); 16 right-hand sides 58, 33, 66; 128 of
// them 120, 63, 128 (539, 446, 262; 100, 56, 105). C alone of 576 rings 815 at 16 (HBM-bound), 1,299 at
// 64, 2,153 at 128 (786, 1,130, 2,242 with two FP16 parts behind a tensor map).
// Error against 64 bits on the bars 4.5e-7, on the rings 2.2e-6 (TF32 6.6e-6), the accumulator's.
// Every wait is bounded: on a timeout the CTA records an error (err[0], kept across products)
// and raises the launch's abort flag (err[1], cleared before each launch), waits (with a short
// limit) for its own MMAs and copies in flight, frees its TMEM and leaves; the other CTAs see
// the flag in their waits, or before they start, and leave too. The results are then invalid.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "bulk.cuh"
#include "common.cuh"

namespace bem {

constexpr int kTcM = 128;       // rows per tile (MMA M, TMEM lanes)
constexpr int kTcK = 32;        // floats of K per stage: one 128-byte swizzle row
// Per width NP of B: stages S, threads G that convert one stage. One group of threads per stage: a
// group waits on its loads and its proxy fence while the others work, and never waits for a phase
// of its stage that is two ahead.
template <int NP> struct TcShape;
template <> struct TcShape<32> { static constexpr int S = 7, G = 64; };
template <> struct TcShape<64> { static constexpr int S = 6, G = 64; };
template <> struct TcShape<128> { static constexpr int S = 4, G = 128; };
template <> struct TcShape<256> { static constexpr int S = 3, G = 128; };
constexpr int kTcEpi = 128;  // threads that read the accumulators, one row of a tile each
template <int NP> constexpr int tc_threads() { return kTcEpi + 64 + TcShape<NP>::S * TcShape<NP>::G; }
constexpr int kTcMaxRhs = 128;  // N = 2R <= 256 per launch
constexpr uint32_t kTcAtile = kTcM * kTcK * 4;  // 16 KB: FP32, then the first and second parts
constexpr uint32_t kTcA3 = kTcM * kTcK * 2;     // 8 KB: the third parts

struct TcUnit {  // stages [k0, k1) of one 128-row tile of one block of Z (mat 0) or C (mat 1)
  int32_t obj, row0, mat, k0, k1;
  int32_t parts;        // units of the tile; its partial sums are the slots slot0 .. slot0 + parts - 1
  int32_t slot, slot0;  // (parts > 1 only)
};
struct TcObj {   // per object: size, first unknown, first K column in the packed B
  int32_t n, xoff;
  int64_t koff;  // first stage in the packed B
};

// K-major operand in shared memory with the 128-byte swizzle: rows of 128 bytes, 8-row groups
// 1024 bytes apart (stride byte offset), leading byte offset unused (1), descriptor version 1,
// layout type 2 (128-byte swizzle). The tile base is 1024-byte aligned; the K steps inside the
// 128-byte row advance the start address by 32 bytes.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// the same with rows of 64 bytes, 8-row groups 512 bytes apart, layout type 4 (64-byte swizzle: the
// 16-byte vector v of row r at v ^ ((r >> 1) & 3))
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}
// instruction descriptor of kind::f16: D in FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9 and 10-12 =
// 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t bf16_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tc_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives on the mbarrier once every MMA this thread issued before it has completed
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
// 16 consecutive FP32 columns of this thread's TMEM lane (32x32b shape: lane = thread of the
// warp, from the warp's 32-lane quarter), waited for inside the same statement
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// the three BF16 parts of two values, packed
__device__ __forceinline__ void tc_split(float a, float b, uint32_t* p1, uint32_t* p2, uint32_t* p3) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  *p1 = __byte_perm(ua, ub, 0x7632);
  const float ra = a - __uint_as_float(ua & 0xFFFF0000u), rb = b - __uint_as_float(ub & 0xFFFF0000u);
  const __nv_bfloat162 m = __floats2bfloat162_rn(ra, rb);
  const uint32_t um = *reinterpret_cast<const uint32_t*>(&m);
  *p2 = um;
  const __nv_bfloat162 l =
      __floats2bfloat162_rn(ra - __uint_as_float(um << 16), rb - __uint_as_float(um & 0xFFFF0000u));
  *p3 = *reinterpret_cast<const uint32_t*>(&l);
}

// Bounded wait on an mbarrier phase that also gives up as soon as any CTA of the launch has
// recorded a failure in *err (polled every 8192 tries), so that one stuck CTA does not make
// every later CTA wait out its own limit.
constexpr uint32_t kTcSpin = 1u << 22;
constexpr uint32_t kTcSpinCleanup = 1u << 16;
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, const int* err, uint32_t spins) {
  for (uint32_t it = 0; it < spins; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 8191) == 8191 && *(const volatile int*)err) return false;
  }
  return false;
}

// B from x: rows 2r and 2r + 1 of right-hand side r < R (zero rows up to NP) of the three parts, one CTA
// per object and right-hand side: the slice's 2 n values, zeros up to the object's last stage. A word
// holds two values, 16 words are a row's part of a stage; the two rows of r share a 128-byte line
__global__ void __launch_bounds__(256) k_tc_pack(const float2* __restrict__ x, int64_t vstride, int R,
                                                 const TcObj* __restrict__ objs, int NP,
                                                 uint32_t* __restrict__ b) {
  const TcObj o = objs[blockIdx.x];
  const int r = blockIdx.y;
  const float2* xs = x + r * vstride + o.xoff;
  uint32_t* p0 = b + (o.koff * 3 * NP + 2 * r) * 16;
  for (int k = threadIdx.x; k < (o.n + 15 & ~15); k += 256) {
    const float2 v = r < R && k < o.n ? xs[k] : make_float2(0.f, 0.f);
    uint32_t* p = p0 + (int64_t)(k >> 4) * (48 * NP) + (((k >> 2 & 3) ^ (r & 3)) * 4 + (k & 3));
    tc_split(v.x, -v.y, p, p + 16 * NP, p + 32 * NP);
    tc_split(v.y, v.x, p + 16, p + 16 * NP + 16, p + 32 * NP + 16);
  }
}

// shared memory of one CTA: S stages of [A | A3 | B1 | B2 | B3], each tile 1024-byte aligned, then the
// barriers, the TMEM slot
template <int NP> struct TcSmem {
  static constexpr int S = TcShape<NP>::S;
  static constexpr uint32_t kB = kTcAtile + kTcA3, kBp = NP * kTcK * 2;  // kBp: bytes of one part of B
  static constexpr uint32_t kStage = kB + 3 * kBp;
  static constexpr uint32_t kTx = kStage - kTcA3;  // bytes landing per stage
  static constexpr uint32_t kBars = S * kStage;
  static constexpr uint32_t kBytes = kBars + 8 * (3 * S + 5) + 16 + 1024;  // + alignment slack
};

// one row of a landed FP32 tile (128 bytes, its 16-byte vectors swizzled by the row) turned in place
// into 32 first parts and 32 second parts, the third parts to the tile after it
__device__ __forceinline__ void tc_convert_row(uint8_t* tile, int row) {
  float4* a = reinterpret_cast<float4*>(tile + row * 128);
  uint4* a3 = reinterpret_cast<uint4*>(tile + kTcAtile + row * 64);
  const int x = row & 7, x3 = row >> 1 & 3;
  float4 v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = a[c ^ x];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 p = v[2 * j], q = v[2 * j + 1];
    uint4 h, m, l;
    tc_split(p.x, p.y, &h.x, &m.x, &l.x);
    tc_split(p.z, p.w, &h.y, &m.y, &l.y);
    tc_split(q.x, q.y, &h.z, &m.z, &l.z);
    tc_split(q.z, q.w, &h.w, &m.w, &l.w);
    reinterpret_cast<uint4*>(a)[j ^ x] = h;
    reinterpret_cast<uint4*>(a)[(4 + j) ^ x] = m;
    a3[j ^ x3] = l;
  }
}

// Persistent CTAs, one per SM; CTA b takes the units b, b + gridDim.x, ... (nst[b] stages in all): a unit
// is the stages [k0, k1) of the K loop of one 128-row tile of one block of one of the two matrices.
// Warps 0-3 read the accumulators, warp 4 issues the TMA loads, warp 5 the MMAs, the others convert the
// landed tiles; stages pass from one to the next through mbarriers and run on across units, and
// (NP <= 128) the accumulators are double, so a unit's start-up and its epilogue cost nothing. A1 B1
// is accumulated apart from the other five terms (NP columns, 2 NP where TMEM has them): the tensor core
// truncates every accumulation, and those terms, 2^-7 as large, would make the truncations of the large
// sum six times as many. The parts of a tile cut into several units go to a workspace, which k_tc_reduce sums (the
// unit that finishes last, four warps on one SM, took 50 us for it).
template <int NP>
__global__ void __launch_bounds__(tc_threads<NP>(), 1)
    k_zgemm_tc(const uint32_t* __restrict__ b, const CUtensorMap* __restrict__ mz,
               const CUtensorMap* __restrict__ mc, const TcUnit* __restrict__ units, int nunit,
               const int32_t* __restrict__ nst, const TcObj* __restrict__ objs,
               float2* __restrict__ yz, float2* __restrict__ yc, int64_t vstride, int R,
               float4* __restrict__ part, int* err) {
  typedef TcSmem<NP> L;
  constexpr int S = L::S, kG = TcShape<NP>::G;
  constexpr int NACC = NP <= 128 ? 2 : 1;          // sets of accumulators in TMEM
  constexpr uint32_t kAcc = (NP <= 64 ? 3 : 2) * NP;  // columns of one: A1 B1, then the other terms
  constexpr uint32_t kCols = NP == 32 ? 256 : 512;
  static_assert(NACC * kAcc <= kCols, "TMEM columns");
  constexpr uint32_t kIdesc = bf16_idesc(kTcM, NP), kIdesc2 = bf16_idesc(kTcM, NP <= 128 ? 2 * NP : NP),
                     kIdesc3 = bf16_idesc(kTcM, NP <= 64 ? 3 * NP : NP);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + L::kBars);  // [S] the stage's loads have landed
  uint64_t* conv = full + S;                                      // [S] its A tile is converted
  uint64_t* empty = conv + S;                                     // [S] its MMAs are done
  uint64_t* done = empty + S;                                     // [2] a unit's accumulators are final
  uint64_t* taken = done + 2;                                     // [2] ... and have been read
  uint64_t* fin = taken + 2;                                      // clean-up
  uint32_t* tslot = reinterpret_cast<uint32_t*>(fin + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int* const abort_flag = err + 1;  // set by any CTA of this launch that gave up

  // a CTA that starts after another one gave up leaves at once (one decision for the block)
  __shared__ int s_flag, s_fail;
  if (tid == 0) {
    s_flag = *(const volatile int*)abort_flag;
    s_fail = 0;
  }
  __syncthreads();
  if (s_flag) return;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&conv[s], kG / 32);
      mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&done[q], 1);
      mbar_init(&taken[q], kTcEpi / 32);
    }
    mbar_init(fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) tc_alloc(tslot, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;  // set q: columns kAcc q + [0, NP) A1 B1, then the other terms

  int issued = 0;  // producer: stages whose loads are issued
  bool ok = true;
  if (warp < 4) {
    // accumulators out: thread = row of the tile; warp 0 decides for the four (they share barriers)
    const int trow = tid;
    int n = 0;
    for (int ui = blockIdx.x; ui < nunit; ui += gridDim.x, ++n) {
      const TcUnit u = units[ui];
      const TcObj o = objs[u.obj];
      const int q = n % NACC;
      if (warp == 0) {
        ok = __all_sync(0xffffffffu, tc_wait(&done[q], (n / NACC) & 1, abort_flag, kTcSpin));
        if (lane == 0) s_flag = ok;
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (!*(volatile int*)&s_flag) break;
      tc_fence_after();
      const int row = u.row0 + trow, cend = min(NP, (2 * R + 15) & ~15);
      float2* y = u.mat ? yc : yz;
      const uint32_t tl = tmem + kAcc * q + ((uint32_t)(warp * 32) << 16);
      for (int c0 = 0; c0 < cend; c0 += 16) {
        float v[16], w[16];
        tc_ld16(tl + c0, v);
        tc_ld16(tl + NP + c0, w);
        if constexpr (kAcc > 2 * NP) {
          float w2[16];
          tc_ld16(tl + 2 * NP + c0, w2);
#pragma unroll
          for (int k = 0; k < 16; ++k) w[k] += w2[k];
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] += w[k];
        if (u.parts > 1) {
          float4* p = part + (int64_t)u.slot * (kTcM * NP / 4) + (c0 / 4) * kTcM + trow;
#pragma unroll
          for (int k = 0; k < 4; ++k) p[k * kTcM] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        } else if (row < o.n) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int r = c0 / 2 + k;
            if (r < R) y[r * vstride + o.xoff + row] = make_float2(v[2 * k], v[2 * k + 1]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&taken[q]);
      asm volatile("bar.sync 1, 128;" ::: "memory");  // s_flag is rewritten by the next unit
    }
  } else if (warp == 4) {
    if (lane == 0) {
      int slot = 0, ph = 1;  // ph: parity of the stage's previous MMAs (the first pass waits for none)
      for (int ui = blockIdx.x; ui < nunit && ok; ui += gridDim.x) {
        const TcUnit u = units[ui];
        const TcObj o = objs[u.obj];
        const CUtensorMap* mA = (u.mat ? mc : mz) + u.obj;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mA)) : "memory");
        for (int kc = u.k0; kc < u.k1; ++kc) {
          if (issued >= S && !tc_wait(&empty[slot], ph, abort_flag, kTcSpin)) {
            ok = false;
            break;
          }
          uint8_t* st = base + slot * L::kStage;
          mbar_arrive_tx(&full[slot], L::kTx);
          tma_load_2d(st, mA, kc * kTcK, u.row0, &full[slot]);
          bulk_g2s(st + L::kB, b + (o.koff + kc) * (48 * NP), 3 * L::kBp, &full[slot]);
          ++issued;
          if (++slot == S) {
            slot = 0;
            ph ^= 1;
          }
        }
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      int slot = 0, ph = 0, n = 0;
      for (int ui = blockIdx.x; ui < nunit && ok; ui += gridDim.x, ++n) {
        const int k0 = units[ui].k0, k1 = units[ui].k1, q = n % NACC;
        if (n >= NACC && !tc_wait(&taken[q], (n / NACC - 1) & 1, abort_flag, kTcSpin)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + kAcc * q;
        for (int kc = k0; kc < k1; ++kc) {
          if (!tc_wait(&full[slot], ph, abort_flag, kTcSpin) || !tc_wait(&conv[slot], ph, abort_flag, kTcSpin)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(base + slot * L::kStage), sb = sa + L::kB;
#pragma unroll
          for (int k = 0; k < kTcK / 16; ++k) {  // 16 BF16 = 32 bytes of K per instruction
            const uint64_t a1 = sw128_desc(sa + 32 * k), a2 = sw128_desc(sa + 64 + 32 * k);
            const uint64_t a3 = sw64_desc(sa + kTcAtile + 32 * k), b1 = sw64_desc(sb + 32 * k);
            const uint64_t b2 = sw64_desc(sb + L::kBp + 32 * k), b3 = sw64_desc(sb + 2 * L::kBp + 32 * k);
            const uint32_t acc = (kc > k0 || k > 0) ? 1u : 0u;
            if constexpr (NP <= 64) {
              tc_mma_bf16(d, a1, b1, kIdesc3, acc);        // A1 [B1 B2 B3]
              tc_mma_bf16(d + NP, a2, b1, kIdesc2, 1u);    // A2 [B1 B2], onto A1 B2 and A1 B3
            } else {
              if constexpr (NP == 128) {
                tc_mma_bf16(d, a1, b1, kIdesc2, acc);      // A1 [B1 B2]
              } else {
                tc_mma_bf16(d, a1, b1, kIdesc, acc);
                tc_mma_bf16(d + NP, a1, b2, kIdesc, acc);
              }
              tc_mma_bf16(d + NP, a2, b1, kIdesc, 1u);
              tc_mma_bf16(d + NP, a2, b2, kIdesc, 1u);
              tc_mma_bf16(d + NP, a1, b3, kIdesc, 1u);
            }
            tc_mma_bf16(d + NP, a3, b1, kIdesc, 1u);
          }
          tc_commit(&empty[slot]);
          if (++slot == S) {
            slot = 0;
            ph ^= 1;
          }
        }
        if (ok) tc_commit(&done[q]);
      }
    }
  } else {
    // a group converts the stages of its slot, a thread the rows t, t + kG, ... of each
    constexpr int kRows = kTcM / kG;
    const int t = (tid - 192) % kG, slot = (tid - 192) / kG, total = nst[blockIdx.x];
    int ph = 0;
    for (int i = slot; i < total; i += S, ph ^= 1) {
      ok = tc_wait(&full[slot], ph, abort_flag, kTcSpin);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      uint8_t* st = base + slot * L::kStage;
#pragma unroll
      for (int k = 0; k < kRows; ++k) tc_convert_row(st, t + k * kG);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&conv[slot]);
    }
  }
  if (!ok) {
    s_fail = 1;
    atomicExch(err, 1);
    atomicExch(abort_flag, 1);
  }
  __syncwarp();
  __syncthreads();
  if (s_fail) {  // leave cleanly: MMAs and copies in flight waited for (bounded)
    const int none = 0;  // these waits run their own short limit to the end
    if (warp == 5 && lane == 0) {
      tc_commit(fin);
      tc_wait(fin, 0, &none, kTcSpinCleanup);
    }
    if (warp == 4 && lane == 0)
      for (int c = max(issued - S, 0); c < issued; ++c) tc_wait(&full[c % S], (c / S) & 1, &none, kTcSpinCleanup);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 5) tc_dealloc(tmem, kCols);
}

// y of the tiles cut along K: the sum of their parts in order; one CTA per tile and 16 columns
template <int NP>
__global__ void __launch_bounds__(kTcM) k_tc_reduce(const TcUnit* __restrict__ tiles, const TcObj* __restrict__ objs,
                                                    const float4* __restrict__ part, float2* __restrict__ yz,
                                                    float2* __restrict__ yc, int64_t vstride, int R) {
  const TcUnit u = tiles[blockIdx.x];
  const TcObj o = objs[u.obj];
  const int row = u.row0 + threadIdx.x, c0 = 16 * blockIdx.y;
  if (row >= o.n) return;
  const float4* p = part + (int64_t)u.slot0 * (kTcM * NP / 4) + (c0 / 4) * kTcM + threadIdx.x;
  float4 a[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) a[c] = p[c * kTcM];
#pragma unroll 4
  for (int k = 1; k < u.parts; ++k) {
    p += kTcM * NP / 4;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 t = p[c * kTcM];
      a[c] = make_float4(a[c].x + t.x, a[c].y + t.y, a[c].z + t.z, a[c].w + t.w);
    }
  }
  float2* y = (u.mat ? yc : yz) + o.xoff + row;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int r = c0 / 2 + 2 * c;
    if (r < R) y[r * vstride] = make_float2(a[c].x, a[c].y);
    if (r + 1 < R) y[(r + 1) * vstride] = make_float2(a[c].z, a[c].w);
  }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
typedef PFN_cuTensorMapEncodeTiled_v12000 TcEncode;

struct TcState {
  CUtensorMap* mz = nullptr;  // per object, over the FP32 Z and C blocks (device)
  CUtensorMap* mc = nullptr;
  struct Units {
    TcUnit* d = nullptr;
    int32_t* nst = nullptr;   // [ctas] stages of each persistent CTA
    TcUnit* cut = nullptr;    // [ncut] first unit of every tile cut along K
    int n = 0, ncut = 0, slots = 0, ctas = 0;
  } units[3];                 // Z alone, C alone, both
  TcObj* objs = nullptr;
  int64_t ktot = 0;           // stages of the packed B
  uint32_t* b = nullptr;      // packed B, [ktot][3][NP][16]
  float4* part = nullptr;     // partial sums of tiles cut along K
  int np_cap = 0;
  int* err = nullptr;         // [2]: a wait timed out in some product (sticky); this launch gave up
  int64_t calls = 0;
  ~TcState() {
    for (Units& u : units)
      for (void* p : {(void*)u.d, (void*)u.nst, (void*)u.cut})
        if (p) cudaFree(p);
    for (void* p : {(void*)mz, (void*)mc, (void*)objs, (void*)b, (void*)part, (void*)err})
      if (p) cudaFree(p);
  }
};

static TcEncode tc_encoder() {
  static TcEncode fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<TcEncode>(p);
  }
  return fn;
}

// 2-D FP32 tensor map, inner extent `inner` floats, `rows` rows `pitch` bytes apart, box of
// 32 floats x box_rows, 128-byte swizzle, zero fill outside
static int tc_map(TcEncode enc, CUtensorMap* m, const void* base, int64_t inner, int64_t rows,
                  int64_t pitch, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch};
  const cuuint32_t box[2] = {(cuuint32_t)kTcK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (pitch & 15)) {
    set_error("tensor-core product: operand not 16-byte aligned");
    return BEM_EINVAL;
  }
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides,
                         box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("tensor-core product: cuTensorMapEncodeTiled failed (%d)", (int)r);
    return BEM_ECUDA;
  }
  return BEM_OK;
}

// The units of a product over the matrices in `mats` (bit 0 Z, bit 1 C): every tile's K loop is cut
// into equal parts of at most Lmax stages, Lmax the shortest for which there are at most w units per
// SM; w is the one with the least w Lmax, plus kTcOver where that cuts any tile (the trip through
// the workspace, in stages; 6 to 18 give the same times). Longest first, dealt to the CTAs in turn.
constexpr int kTcOver = 12, kTcMaxParts = 16;
static std::vector<TcUnit> tc_units(const std::vector<TcObj>& objs, int mats, int nsm, int* slots) {
  struct T { int obj, row0, mat, nk; };
  std::vector<T> ts;
  int longest = 0;
  for (int m = 0; m < 2; ++m)
    if (mats >> m & 1)
      for (int i = 0; i < (int)objs.size(); ++i)
        for (int r0 = 0; r0 < objs[i].n; r0 += kTcM) {
          ts.push_back({i, r0, m, (2 * objs[i].n + kTcK - 1) / kTcK});
          longest = std::max(longest, ts.back().nk);
        }
  auto count = [&](int L) {
    int64_t c = 0;
    for (const T& t : ts) c += (t.nk + L - 1) / L;
    return c;
  };
  const int shortest = std::max(1, (longest + kTcMaxParts - 1) / kTcMaxParts);
  int best = longest;
  int64_t cost = INT64_MAX;
  for (int w = 1; w <= 8; ++w) {
    int lo = shortest, hi = longest;  // smallest L with count(L) <= w nsm
    if (count(hi) > (int64_t)w * nsm) continue;
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (count(mid) <= (int64_t)w * nsm) hi = mid;
      else lo = mid + 1;
    }
    const int64_t c = (int64_t)w * lo + (lo < longest ? kTcOver : 0);
    if (c < cost) {
      cost = c;
      best = lo;
    }
  }
  std::vector<TcUnit> us;
  *slots = 0;
  for (int i = 0; i < (int)ts.size(); ++i) {
    const T& t = ts[i];
    const int p = (t.nk + best - 1) / best, s0 = *slots;
    for (int q = 0; q < p; ++q)
      us.push_back(TcUnit{t.obj, t.row0, t.mat, (int)((int64_t)t.nk * q / p), (int)((int64_t)t.nk * (q + 1) / p),
                          p, s0 + q, s0});
    if (p > 1) *slots += p;
  }
  std::stable_sort(us.begin(), us.end(), [](const TcUnit& a, const TcUnit& b) { return a.k1 - a.k0 > b.k1 - b.k0; });
  return us;
}

// units, object table, slot table and the per-object tensor maps of Z and C (first use)
static int tc_prepare(aim_ctx* c, TcState** out) {
  if (c->tc) {
    *out = static_cast<TcState*>(c->tc);
    return BEM_OK;
  }
  TcEncode enc = tc_encoder();
  if (!enc) {
    set_error("tensor-core product: cuTensorMapEncodeTiled is not available from the driver");
    return BEM_ECUDA;
  }
  if (!c->f32.Z || !c->f32.C) {
    set_error("tensor-core product: no FP32 internal blocks");
    return BEM_EINVAL;
  }
  TcState* t = new TcState();
  std::vector<TcObj> objs(c->nobj);
  int64_t ktot = 0;
  std::vector<CUtensorMap> mz(c->nobj), mc(c->nobj);
  int rc = BEM_OK;
  for (int i = 0, xo = 0; i < c->nobj && rc == BEM_OK; ++i) {
    const int n = c->e1[i] - c->e0[i], ld = c->zld[i];
    objs[i] = TcObj{n, xo, ktot};
    ktot += round_up(n, 16) / 16;
    rc = tc_map(enc, &mz[i], c->f32.Z + c->zoff[i], 2 * (int64_t)n, n, 8 * (int64_t)ld, kTcM);
    if (rc == BEM_OK) rc = tc_map(enc, &mc[i], c->f32.C + c->zoff[i], 2 * (int64_t)n, n, 8 * (int64_t)ld, kTcM);
    xo += n;
  }
  t->ktot = ktot;
  auto up = [&](void** p, const void* h, size_t bytes) {
    if (rc != BEM_OK) return;
    if (cudaMalloc(p, bytes) != cudaSuccess || cudaMemcpy(*p, h, bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
      set_error("tensor-core product: device allocation failed");
      rc = BEM_ENOMEM;
    }
  };
  up((void**)&t->mz, mz.data(), mz.size() * sizeof(CUtensorMap));
  up((void**)&t->mc, mc.data(), mc.size() * sizeof(CUtensorMap));
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  for (int m = 0; m < 3; ++m) {
    TcState::Units& q = t->units[m];
    const std::vector<TcUnit> us = tc_units(objs, m == 2 ? 3 : m + 1, std::max(nsm, 1), &q.slots);
    q.n = (int)us.size();
    q.ctas = std::min(q.n, std::max(nsm, 1));
    std::vector<int32_t> nst(q.ctas, 0);
    for (int i = 0; i < q.n; ++i) nst[i % q.ctas] += us[i].k1 - us[i].k0;
    up((void**)&q.nst, nst.data(), nst.size() * sizeof(int32_t));
    std::vector<TcUnit> cut;
    for (const TcUnit& v : us)
      if (v.parts > 1 && v.slot == v.slot0) cut.push_back(v);
    q.ncut = (int)cut.size();
    if (q.ncut > 0) up((void**)&q.cut, cut.data(), cut.size() * sizeof(TcUnit));
    up((void**)&q.d, us.data(), us.size() * sizeof(TcUnit));
  }
  up((void**)&t->objs, objs.data(), objs.size() * sizeof(TcObj));
  const int zero[2] = {0, 0};  // [0]: a wait timed out in some product; [1]: this launch gave up
  up((void**)&t->err, zero, sizeof(zero));
  if (rc != BEM_OK) {
    delete t;
    return rc;
  }
  c->tc = t;
  *out = t;
  return BEM_OK;
}

template <int NP>
static int tc_launch(TcState* t, float2* yz, float2* yc, int64_t vstride, int R, cudaStream_t s) {
  constexpr uint32_t kSmem = TcSmem<NP>::kBytes;
  static_assert(kSmem <= 227 * 1024, "shared memory per CTA");
  const TcState::Units& q = t->units[yz && yc ? 2 : yz ? 0 : 1];
  // per call: the attribute belongs to the current device (cheap next to the product)
  BEM_CUDA(cudaFuncSetAttribute(k_zgemm_tc<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
  BEM_CUDA(cudaMemsetAsync(t->err + 1, 0, sizeof(int), s));
  k_zgemm_tc<NP><<<q.ctas, tc_threads<NP>(), kSmem, s>>>(t->b, t->mz, t->mc, q.d, q.n, q.nst, t->objs, yz, yc,
                                                         vstride, R, t->part, t->err);
  if (q.ncut > 0)
    k_tc_reduce<NP><<<dim3(q.ncut, (2 * R + 15) / 16), kTcM, 0, s>>>(q.cut, t->objs, t->part, yz, yc, vstride, R);
  BEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// e_r = Z h_r and h_eq,r = C h_r for r < nrhs (FP32, vectors ne apart); either output may be null
int internal_tc(aim_ctx* c, const float2* h, float2* e, float2* heq, int nrhs, cudaStream_t s) {
  TcState* t = nullptr;
  BEM_TRY(tc_prepare(c, &t));
  if (t->units[0].n == 0) return BEM_OK;
  const int64_t ne = c->ne;
  for (int r0 = 0; r0 < nrhs; r0 += kTcMaxRhs) {
    const int R = std::min(kTcMaxRhs, nrhs - r0);
    const int NP = R <= 16 ? 32 : R <= 32 ? 64 : R <= 64 ? 128 : 256;
    if (NP > t->np_cap) {
      BEM_CUDA(cudaStreamSynchronize(s));  // the old workspace may be in use on s
      if (t->b) cudaFree(t->b);
      if (t->part) cudaFree(t->part);
      t->b = nullptr;
      t->part = nullptr;
      t->np_cap = 0;
      const size_t bytes = (size_t)3 * NP * 16 * t->ktot * sizeof(uint32_t);
      int slots = 0;
      for (const TcState::Units& q : t->units) slots = std::max(slots, q.slots);
      const size_t pbytes = (size_t)slots * kTcM * NP * sizeof(float) + 16;
      if (cudaMalloc((void**)&t->b, bytes) != cudaSuccess || cudaMalloc((void**)&t->part, pbytes) != cudaSuccess) {
        set_error("tensor-core product: no device memory for the packed right-hand sides");
        return BEM_ENOMEM;
      }
      t->np_cap = NP;
    }
    k_tc_pack<<<dim3(c->nobj, NP / 2), 256, 0, s>>>(h + r0 * ne, ne, R, t->objs, NP, t->b);
    BEM_CUDA(cudaGetLastError());
    float2* yz = e ? e + r0 * ne : nullptr;
    float2* yc = heq ? heq + r0 * ne : nullptr;
#define BEM_TC(NPV) BEM_TRY(tc_launch<NPV>(t, yz, yc, ne, R, s))
    switch (NP) {
      case 32: BEM_TC(32); break;
      case 64: BEM_TC(64); break;
      case 128: BEM_TC(128); break;
      default: BEM_TC(256); break;
    }
#undef BEM_TC
  }
  ++t->calls;
  return BEM_OK;
}

void free_tc(aim_ctx* c) {
  delete static_cast<TcState*>(c->tc);
  c->tc = nullptr;
}

// products made, a wait timed out (1) or not (0); -1 when the product was never used
void tc_stats(const aim_ctx* c, int64_t* out) {
  const TcState* t = static_cast<const TcState*>(c->tc);
  out[0] = t ? t->calls : 0;
  out[1] = -1;
  int v = 0;
  if (t && cudaMemcpy(&v, t->err, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess) out[1] = v;
}

}  // namespace bem
