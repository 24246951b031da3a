// Split-BF16 tensor-core sgemm without a packing pass: every CTA reads its
// FP32 operands itself, splits them in registers and feeds the tensor cores
// from shared memory.
//
// The packed path (split.cu) writes hi/lo panels to HBM and reads them back:
// three dependent stream items for a small call, and 12 bytes of traffic per
// operand element for a call whose operands are used by few tiles.  Here one
// launch does it all and an element is read from HBM once (and from L2 once
// per tile that uses it), at the price of splitting it once per tile.
// Measured against the packed path (us a call): 256^3 7.4 against 20.5,
// 1024^3 22.9 against 31.6, 512 x 512 x 65536 100 against 181, a batch of 64
// products 192 x 256 x 4096 111 against 283; at 2048^3 the two are equal
// (64), beyond that the packed path, whose MMAs find their operands ready,
// wins (4096^3: 534 against 340).
//
// Tile: 128 x BN per CTA, or with PAIR 256 x BN per cluster pair
// (tcgen05 cta_group::2, each CTA its own 128 rows of op(A) and half of the
// tile's columns of op(B)).  Every warp of a CTA loads its share of a step's
// k chunks of both operands into registers, two steps in flight, splits it
// into two or three BF16 parts and stores it in the 128-byte-swizzled K-major
// form the tensor cores read (three parts: the third in a 64-byte-swizzled
// block); one thread issues the MMAs, in the order of the packed path, when
// every warp has stored its share, and the warps split the next step
// meanwhile.  (A warp of its own for the MMAs would cost every thread a
// quarter of its registers.)  hi*hi accumulates in one accumulator and the
// smaller products in another, added at the end: the tensor cores truncate
// every addition, so the error of a sum grows with the number of additions
// to its large terms (k = 256: relative error 8e-8 against 1.8e-6 of the
// packed path; k = 4096: 5.3e-6 against 1.4e-5).
//
// What bounds a step (64 k, pair 256 x 256: 1.58 us, 1.0 of it MMAs at the
// packed kernel's rate): taking away the loads, or the splitting, saves 17%
// each.  It is a chain of loads, splitting and MMAs that two steps in
// registers and two in shared memory only partly overlap; registers (128 of
// 128) and the L1 left beside the ring keep it from more.
//
// k slices: `slices` CTAs (pairs) share a tile, each a contiguous range of k
// chunks.  Up to 16 CTAs they form one cluster and sum their accumulators in
// slice order through distributed shared memory, each finishing its share of
// the columns; more slices store raw tiles to the workspace for the split-K
// reduction.
//
// Scaling of badly scaled K-vectors (largest magnitude outside [2^-48,
// 2^48)): a vector's maximum is not known before its elements are loaded, so
// its exponent is taken from the first step (none if it is zero there), and
// the rest of the vector is watched: an element that comes out at 2^50 or
// more after scaling, or beyond FP32, or a vector that was zero in the first
// step and whose maximum then lies below 2^-48, makes the CTA (the pair's
// cluster) compute its slice again with exponents from the true maxima.  Three
// parts (at most 16 steps) take the exponent from the first step in which the
// vector is not zero, with barriers until then: 4% on a call with zero vectors,
// where the watch's code cost dense ones up to 5%.  With two parts the
// last watch costs only the threads that hold such vectors, and no barrier
// (512 x 512 x 65536 with every second row of op(A) zero, 129 -> 109 us
// against 98 of dense operands; both operands k contiguous at ld + 1, 267 ->
// 152 against 135; before, every step waited for the block's maxima while a
// vector was zero).  Within those limits the result is what exponents from
// the true maxima give: powers of two commute with FP32 rounding, and
// products stay within 2^100.  Every slice scales on its own; the sum of the
// slices brings their accumulators to the largest exponent of each row and
// column first, so that nothing is rounded to a subnormal before the end.
#pragma once

#include <atomic>

#include "direct.h"
#include "split_device.cuh"

namespace gbg {
namespace {

constexpr float kWatchLimit = 0x1p50f;
constexpr uint64_t kWaitNs = 2000000000ull;

// Shape of a kernel instance.  UK k chunks are split per step, each by eight
// warps of its own.  Two parts: two chunks (16 warps), so that the waits and
// arrivals of a step, which cost a warp as many instructions as splitting its
// values, are paid once per 64 k; three parts (k < 512): one chunk.
template <int BN, bool PAIR, int PARTS>
struct DirectShape {
  static constexpr int UK = PARTS == 3 ? 1 : 2;
  static constexpr int WARPS = 8 * UK, THREADS = 32 * WARPS;
  static constexpr int BS = PAIR ? BN / 2 : BN;       // B rows a CTA splits
  static constexpr int A2 = 128 * 128, B2 = BS * 128; // [hi | lo] or [hi | mid] bytes of a chunk
  static constexpr int A3 = PARTS == 3 ? 128 * 64 : 0, B3 = PARTS == 3 ? BS * 64 : 0;
  static constexpr int CHUNK = A2 + B2 + A3 + B3;
  static constexpr int STAGE = UK * CHUNK;
  // Two parts: one CTA per SM, for 128 registers with sixteen warps.  Two
  // stages, not as many as fit: the loads in flight live in what shared
  // memory leaves of the L1, and with 192 KiB of ring they were what a step
  // waited for (a batch of 64 products 192 x 256 x 4096: 126 against 112 us).
  static constexpr int CTAS = PARTS == 3 ? 2 : 1;
  static constexpr int STAGES = 2;
  static constexpr int RING = STAGES * STAGE;
  // alignment, barriers, exponents, maxima, every thread's late K-vectors
  static constexpr int SMEM = RING + 1024 + 256 + 1536 + 1024 + 4 * THREADS;
  static constexpr int DEPTH = 2;  // steps in flight in registers
  static constexpr int TMEM = 2 * BN;  // accumulators: hi*hi, and the smaller products
  static_assert(CTAS * TMEM <= 512 && CTAS * (SMEM + 1024) <= 228 * 1024, "resident CTAs");
  static_assert(BN > 128 || BN * 512 <= RING, "the cluster reduction puts the accumulator into the ring");
};

// Global loads that stay where they are written: as plain loads the compiler
// moved some prefetches down to their use (2.5 times slower at 512 x 512 x
// 65536).
__device__ __forceinline__ float ldg1(const char* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ldg4(const char* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
// max(|a|, |b|, |c|), NaN if any is.
__device__ __forceinline__ float amax3(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// One operand of a tile: ROWS K-vectors (128, or 64), split by 256 threads,
// N = ROWS / 8 values a thread and chunk:
//   kRows    X[r + p ld]: lane = row of a group of 32, a warp takes a run of
//            N consecutive k, so every load instruction reads 128 contiguous bytes;
//   kVec     X[p + r ld], 16-byte aligned rows: eight lanes a row, four k a
//            lane; the rows of a half warp differ by 4, so that its 8-byte
//            stores fall in different banks;
//   kScalar  X[p + r ld] at any alignment: lane = k, a row per load; lanes
//            trade halves of row pairs (r, r + 4) so that each stores two
//            consecutive k as one word.
// Rows past the operand repeat its last one (they only feed outputs that are
// never stored); k past its end reads as zero.  A thread's addresses are a
// base common to the CTA plus a 32-bit offset, set up once per tile; the
// variants are compiled for their modes: with a switch per chunk the loop
// waited for instructions more than for data (4.1 of 12 cycles each).
template <int ROWS, int MODE>
struct Operand {
  static constexpr int N = ROWS / 8;
  const char* x;       // k chunk 0 of the slice, tile row 0 (the same in every thread)
  uint32_t off;        // byte offset of value 0 (kVec, kScalar: of its k in row 0)
  uint32_t soff, soff3;  // where value 0 goes in a chunk's parts
  uint32_t ld4;        // bytes between rows (kRows: between k)
  int last;            // last valid row of the tile

  static __device__ __forceinline__ int row_of(int v) {  // tile row of value v
    const int warp = (threadIdx.x >> 5) & 7, lane = threadIdx.x & 31;
    if (MODE == kRows) return 32 * (warp % (ROWS / 32)) + lane;
    if (MODE == kVec) return warp * N + (v >> 3) * 8 + ((v >> 2) & 1) * 2 + ((lane >> 3) & 1) * 4 + (lane >> 4);
    return warp * N + v;
  }
  static __device__ __forceinline__ int k_of(int v) {  // k of value v within the chunk
    const int warp = (threadIdx.x >> 5) & 7, lane = threadIdx.x & 31;
    if (MODE == kRows) return (warp / (ROWS / 32)) * N + v;
    if (MODE == kVec) return 4 * (lane & 7) + (v & 3);
    return lane;
  }
  // The operand X's rows from row0 on (`rows` of them exist from there), k from p0 on.
  // sub: this warp's chunk of a step.
  __device__ __forceinline__ void init(const float* X, int64_t ld, int64_t row0, int64_t rows, int64_t p0, int sub) {
    x = reinterpret_cast<const char*>(X + (MODE == kRows ? row0 + p0 * ld : row0 * ld + p0));
    ld4 = (uint32_t)(ld * 4);
    const uint32_t first = sub * (MODE == kRows ? 32u * ld4 : 128u);
    last = (int)(rows < ROWS ? rows : ROWS) - 1;
    off = first + (MODE == kRows ? 4u * min(row_of(0), last) + (uint32_t)k_of(0) * ld4 : 4u * k_of(0));
    // where value 0 goes in a stage: row r at 128 r (64 r), 16-byte chunk c
    // at c ^ (r % 8) (c ^ (r / 2 % 4)); kScalar: lanes trade rows r, r + 4
    const int lane = threadIdx.x & 31;
    const int r = row_of(0) + (MODE == kScalar ? 4 * (lane & 1) : 0), k = k_of(0) & ~1;
    soff = 128u * r + 16u * ((k >> 3) ^ (r & 7)) + 2u * (k & 7);
    soff3 = 64u * r + 16u * ((k >> 3) ^ ((r >> 1) & 3)) + 2u * (k & 7);
  }
  // This warp's chunk of the step whose first chunk is chunk c of the slice
  // (kv of its 32 k exist) into registers.
  __device__ __forceinline__ void load(float (&v)[N], int c, int kv) const {
    const char* b = x + (MODE == kRows ? (size_t)c * 32 * ld4 : (size_t)c * 128);
    uint32_t ld4 = this->ld4;
    asm volatile("" : "+r"(ld4));  // offsets are formed here, not kept in registers from step to step
    auto at = [&](int j) {
      return MODE == kRows ? off + j * ld4
             : MODE == kVec ? off + (uint32_t)min(row_of(j), last) * ld4 + 4u * (j & 3)
                            : off + (uint32_t)min(row_of(j), last) * ld4;
    };
    if (kv >= 32) {
      if (MODE == kVec) {
#pragma unroll
        for (int u = 0; u < N / 4; ++u) {
          const float4 f = ldg4(b + at(4 * u));
          v[4 * u] = f.x; v[4 * u + 1] = f.y; v[4 * u + 2] = f.z; v[4 * u + 3] = f.w;
        }
      } else {
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = ldg1(b + at(j));
      }
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = k_of(j) < kv ? ldg1(b + at(j)) : 0.f;
    }
  }
  // Per-row maxima of a chunk into shared memory.
  __device__ __forceinline__ void row_max(const float (&v)[N], uint32_t* rowmax) const {
    if (MODE == kRows) {
      uint32_t b = 0u;
#pragma unroll
      for (int j = 0; j < N; ++j) b = max(b, __float_as_uint(v[j]) & 0x7FFFFFFFu);
      atomicMax(&rowmax[row_of(0)], b);
    } else if (MODE == kVec) {
#pragma unroll
      for (int u = 0; u < N / 4; ++u) {
        uint32_t b = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) b = max(b, __float_as_uint(v[4 * u + j]) & 0x7FFFFFFFu);
        atomicMax(&rowmax[row_of(4 * u)], b);
      }
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const uint32_t b = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v[j]) & 0x7FFFFFFFu);
        if ((threadIdx.x & 31) == 0) atomicMax(&rowmax[row_of(j)], b);
      }
    }
  }
  // The thread's rows: one (kRows), one of four values each (kVec), or one a
  // value (kScalar, the same rows in every lane).  Bits of those that rowmax
  // holds a zero for.
  static constexpr int R = MODE == kRows ? 1 : MODE == kVec ? N / 4 : N;
  static __device__ __forceinline__ uint16_t zero_rows(const uint32_t* rowmax) {
    uint32_t bits = 0u;
#pragma unroll
    for (int u = 0; u < R; ++u)
      if (rowmax[row_of(u * (N / R))] == 0u) bits |= 1u << u;
    return (uint16_t)bits;
  }
  // The chunk's part in the maxima of the rows in *late, which loses the rows
  // that turn out well scaled here.  Nobody waits for it: the maxima are read
  // after the last step.
  __device__ __forceinline__ void watch_rows(const float (&v)[N], uint16_t* late, uint32_t* rowmax) const {
    const uint32_t bits = *late;
    if (bits == 0u) return;
    uint32_t seen = 0u;
    if (MODE == kScalar) {  // a row's maximum is the warp's; mostly there is nothing but zeros
      uint32_t any = 0u;
#pragma unroll
      for (int u = 0; u < N; ++u) any |= (bits >> u) & 1u ? __float_as_uint(v[u]) : 0u;
      if (!__any_sync(0xFFFFFFFFu, (any & 0x7FFFFFFFu) != 0u)) return;
      const int lane = threadIdx.x & 31;
#pragma unroll
      for (int u = 0; u < N; ++u)
        if ((bits >> u) & 1u) {
          const uint32_t b = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v[u]) & 0x7FFFFFFFu);
          if (b != 0u && lane == 0) atomicMax(&rowmax[row_of(u)], b);
        }
      __syncwarp();
      seen = __ballot_sync(0xFFFFFFFFu, lane < N && rowmax[row_of(0) + min(lane, N - 1)] >= kWellScaledLo);
    } else {
#pragma unroll
      for (int u = 0; u < R; ++u) {
        if (!((bits >> u) & 1u)) continue;
        uint32_t b = 0u;
#pragma unroll
        for (int j = u * (N / R); j < (u + 1) * (N / R); ++j) b = max(b, __float_as_uint(v[j]) & 0x7FFFFFFFu);
        if (b == 0u) continue;
        atomicMax(&rowmax[row_of(u * (N / R))], b);
        if (b >= kWellScaledLo) seen |= 1u << u;
      }
    }
    if (bits & seen) *late = (uint16_t)(bits & ~seen);
  }
  // Whether a finite value left FP32's range (its vector's exponent, taken
  // from an earlier step, is far too small for it).
  __device__ __forceinline__ bool scale(float (&v)[N], const int* ex) const {
    bool left = false;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int e = ex[row_of(j)];
      if (e != 0 && isfinite(v[j])) {
        v[j] = scale_pow2(v[j], e);
        left |= !isfinite(v[j]);
      }
    }
    return left;
  }
  // Split the chunk and store it; returns the largest finite |v|.  One test
  // for Inf and NaN per chunk keeps the usual case one run of independent
  // instructions.
  template <int PARTS>
  __device__ __forceinline__ float store(const float (&v)[N], uint8_t* b2, uint8_t* b3) const {
    float m = amax3(v[0], v[1], v[2]);
#pragma unroll
    for (int j = 3; j + 1 < N; j += 2) m = amax3(m, v[j], v[j + 1]);
    m = amax3(m, v[N - 1], 0.f);
    if (m < INFINITY) {
      store_parts<PARTS, false>(v, b2, b3);
    } else {
      store_parts<PARTS, true>(v, b2, b3);
      m = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) m = fmaxf(m, isfinite(v[j]) ? fabsf(v[j]) : 0.f);
    }
    return m;
  }
  template <int PARTS, bool PATCH>
  __device__ __forceinline__ void store_parts(const float (&v)[N], uint8_t* b2, uint8_t* b3) const {
    uint32_t soff = this->soff, soff3 = this->soff3;
    asm volatile("" : "+r"(soff), "+r"(soff3));  // (as in load)
    if (MODE == kRows) {
      // 16-byte chunk c of a row at position c ^ (row % 8); the next chunk
      // and the lo half are one bit away
      const uint32_t o = soff, o3 = soff3;
#pragma unroll
      for (int c = 0; c < N / 8; ++c) {
        uint32_t h[4], l[4], t[4] = {};
#pragma unroll
        for (int q = 0; q < 4; ++q) split2<PARTS, PATCH>(v[8 * c + 2 * q], v[8 * c + 2 * q + 1], h[q], l[q], t[q]);
        *reinterpret_cast<uint4*>(b2 + (o ^ (16u * c))) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(b2 + (o ^ (16u * c + 64u))) = make_uint4(l[0], l[1], l[2], l[3]);
        if (PARTS == 3) *reinterpret_cast<uint4*>(b3 + (o3 ^ (16u * c))) = make_uint4(t[0], t[1], t[2], t[3]);
      }
    } else if (MODE == kVec) {
#pragma unroll
      for (int u = 0; u < N / 4; ++u) {
        uint32_t h[2], l[2], t[2] = {};
#pragma unroll
        for (int q = 0; q < 2; ++q) split2<PARTS, PATCH>(v[4 * u + 2 * q], v[4 * u + 2 * q + 1], h[q], l[q], t[q]);
        // rows 2 on (u odd) move two positions, rows 8 on none
        const uint32_t o = (soff ^ ((u & 1) * 32u)) + (u >> 1) * 1024u + (u & 1) * 256u;
        *reinterpret_cast<uint2*>(b2 + o) = make_uint2(h[0], h[1]);
        *reinterpret_cast<uint2*>(b2 + (o ^ 64u)) = make_uint2(l[0], l[1]);
        if (PARTS == 3)
          *reinterpret_cast<uint2*>(b3 + ((soff3 ^ ((u & 1) * 16u)) + (u >> 1) * 512u + (u & 1) * 128u)) = make_uint2(t[0], t[1]);
      }
    } else {
      const bool odd = threadIdx.x & 1;
#pragma unroll
      for (int g = 0; g < N / 8; ++g)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float lo = v[8 * g + j], hi = v[8 * g + j + 4];  // rows r and r + 4 at this lane's k
          const float got = __shfl_xor_sync(0xFFFFFFFFu, odd ? lo : hi, 1);
          uint32_t h, l, t = 0u;
          split2<PARTS, PATCH>(odd ? got : lo, odd ? hi : got, h, l, t);  // even lanes: row r, odd lanes: row r + 4
          const uint32_t o = (soff ^ (16u * j)) + g * 1024u + j * 128u;
          *reinterpret_cast<uint32_t*>(b2 + o) = h;
          *reinterpret_cast<uint32_t*>(b2 + (o ^ 64u)) = l;
          if (PARTS == 3) *reinterpret_cast<uint32_t*>(b3 + ((soff3 ^ (16u * (j >> 1))) + g * 512u + j * 64u)) = t;
        }
    }
  }
  // hi, lo (mid) and lo3 of two values, rounded to nearest even; x - hi and
  // x - hi - mid are exact.  PATCH: Inf and NaN are all hi.
  template <int PARTS, bool PATCH>
  static __device__ __forceinline__ void split2(float a, float b, uint32_t& h, uint32_t& l, uint32_t& t) {
    h = cvt_bf16x2(a, b);
    const float r0 = a - bf16_lo(h), r1 = b - bf16_hi(h);
    l = cvt_bf16x2(r0, r1);
    if (PARTS == 3) t = cvt_bf16x2(r0 - bf16_lo(l), r1 - bf16_hi(l));
    if (PATCH) {
      const uint32_t keep = (isfinite(a) ? 0xFFFFu : 0u) | (isfinite(b) ? 0xFFFF0000u : 0u);
      l &= keep;
      t &= keep;
    }
  }
};

__device__ __forceinline__ uint64_t make_desc_sw64(uint32_t saddr) {  // rows of 64 bytes, 8-row groups of 512
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__device__ __forceinline__ float ld_cluster(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ int ld_cluster_int(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Sixteen columns of the warp's 32 accumulator rows: both accumulators, added.
template <int BN>
__device__ __forceinline__ void tmem_sum16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[2][16];
#pragma unroll
  for (int a = 0; a < 2; ++a)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[a][0]), "=r"(r[a][1]), "=r"(r[a][2]), "=r"(r[a][3]), "=r"(r[a][4]), "=r"(r[a][5]), "=r"(r[a][6]),
          "=r"(r[a][7]), "=r"(r[a][8]), "=r"(r[a][9]), "=r"(r[a][10]), "=r"(r[a][11]), "=r"(r[a][12]), "=r"(r[a][13]),
          "=r"(r[a][14]), "=r"(r[a][15])
        : "r"(taddr + (uint32_t)(a * BN)));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[0][j]) + __uint_as_float(r[1][j]);
}

template <int BN, bool PAIR, int PARTS, int MA, int MB>
__global__ void __launch_bounds__(DirectShape<BN, PAIR, PARTS>::THREADS, DirectShape<BN, PAIR, PARTS>::CTAS)
    direct_gemm_kernel(const DirectArgs S) {
  using D = DirectShape<BN, PAIR, PARTS>;
  constexpr int BS = D::BS, UK = D::UK;
  // With two parts, steps with K-vectors to watch have a loop of their own: its
  // code in the one loop cost dense operands 1-6% of a call.  Not with two
  // kScalar operands (two loops spill), nor with three parts (few steps).
  constexpr bool OWN = PARTS == 2 && (MA != kScalar || MB != kScalar);
  static_assert(D::DEPTH == 2, "steps alternate between two sets of registers");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  uint8_t* const ring = smem_raw + (base - raw);
  uint8_t* const tail = ring + D::RING;
  const uint32_t bar0 = smem_u32(tail);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (D::STAGES + s); };
  const uint32_t accf = bar0 + 8u * (2 * D::STAGES);
  uint32_t* const tmem_holder = reinterpret_cast<uint32_t*>(tail + 128);
  volatile int* const redo_s = reinterpret_cast<volatile int*>(tail + 132);
  volatile int* const scaled_s = reinterpret_cast<volatile int*>(tail + 136);
  int* const exA = reinterpret_cast<int*>(tail + 256);          // exponents of the tile's 128 rows ...
  int* const exB = exA + 128;                                   // ... and BN columns
  uint32_t* const rowmax = reinterpret_cast<uint32_t*>(exB + 256);  // maxima: 128 rows, the BS columns split here
  uint16_t* const late = reinterpret_cast<uint16_t*>(rowmax + 256 + threadIdx.x);  // this thread's: rows, columns

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const bool clustered = PAIR || S.cluster_slices > 1;
  const uint32_t crank = clustered ? cluster_ctarank() : 0u;
  const uint32_t prank = PAIR ? (crank & 1u) : 0u, lead = crank & ~1u;
  // the block's tile and slice
  const int item = PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
  const int sl = item % S.slices;
  const int per = S.tiles_m * S.tiles_n;
  const int z = (item / S.slices) / per;
  int tm, tn;
  tile_coords(item / S.slices - z * per, S.tiles_m, S.tiles_n, 8, tm, tn);
  const int64_t m0 = (int64_t)tm * (PAIR ? 256 : 128) + 128 * prank, n0 = (int64_t)tn * BN;
  const int kc0 = sl * S.slice_chunks;
  const int nch = min(S.nkc - kc0, S.slice_chunks);
  float* const C = S.C + (size_t)z * S.sc;
  int* const exBo = exB + (PAIR ? BS * (int)prank : 0);

  if (tid == 0) {
    for (int s = 0; s < D::STAGES; ++s) {
      mbar_init(full_bar(s), (PAIR ? 2 : 1) * D::WARPS);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accf, 1);
    *redo_s = 0;
    *scaled_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < 128 + 256 + 256; i += D::THREADS) exA[i] = 0;  // exponents and maxima
  wait_prerequisite_grid();  // (the kernel before this one on the stream)
  launch_dependents();
  // op(A) rows of this CTA (an odd half past m repeats the last row), op(B) columns it splits
  const int sub = UK == 1 ? 0 : warp >> 3;  // this warp's chunk of step i: i UK + sub
  Operand<128, MA> OA;
  Operand<BS, MB> OB;
  {
    const int64_t ar = m0 < S.m ? m0 : S.m - 1;
    const int64_t br0 = n0 + (PAIR ? BS * (int64_t)prank : 0), br = br0 < S.n ? br0 : S.n - 1;
    OA.init(S.A + (size_t)z * S.sa, S.lda, ar, S.m - ar, (int64_t)kc0 * 32, sub);
    OB.init(S.B + (size_t)z * S.sb, S.ldb, br, S.n - br, (int64_t)kc0 * 32, sub);
  }
  const int kleft = (int)(S.k - (int64_t)kc0 * 32 < (int64_t)nch * 32 ? S.k - (int64_t)kc0 * 32 : (int64_t)nch * 32);
  const int steps = (nch + UK - 1) / UK;
  float va[D::DEPTH][16], vb[D::DEPTH][BS / 8];
  auto load_a = [&](float (&v)[16], int i) { OA.load(v, i * UK, kleft - 32 * (i * UK + sub)); };
  auto load_b = [&](float (&v)[BS / 8], int i) { OB.load(v, i * UK, kleft - 32 * (i * UK + sub)); };
  auto load_first = [&]() {
#pragma unroll
    for (int d = 0; d < D::DEPTH; ++d)
      if (d < steps) {
        load_a(va[d], d);
        load_b(vb[d], d);
      }
  };
  load_first();  // the first steps are on their way while the CTA sets itself up
  if (S.beta != 0.f && !S.partial && m0 < S.m) {  // ask L2 for the tile's C
    const int64_t rows = S.m - m0 < 128 ? S.m - m0 : 128, cols = S.n - n0 < BN ? S.n - n0 : BN;
    if (tid < cols) {
      const char* col = reinterpret_cast<const char*>(C + m0 + (n0 + tid) * S.ldc);
      for (int64_t off = 0; off < rows * 4; off += 128) prefetch_l2(col + off);
      prefetch_l2(col + rows * 4 - 4);
    }
  }
  if (warp == 0) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_holder)), "r"(D::TMEM) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_holder)), "r"(D::TMEM) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();  // the pair's barriers are initialised on both sides
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  bool dead = false;  // a wait ran out: go on without waiting, so that every barrier below is reached
  auto wait = [&](uint32_t bar, uint32_t parity) {  // (inline: a call would spill the values in flight)
    if (dead || mbar_try(bar, parity)) return;
    const uint64_t t0 = globaltimer();
    while (!mbar_try_hint(bar, parity, 20000u)) {
      if (globaltimer() - t0 > kWaitNs) {
        atomicCAS(S.status, 0, (int)GBGEMM_ERR_DEVICE_TIMEOUT);
        dead = true;
        break;
      }
    }
  };
  int stage = 0, passes = 0;
  uint32_t phase = 0;
  const bool issuer = tid == 0 && prank == 0u;
  const uint32_t idesc = make_idesc_bf16(PAIR ? 256 : 128, BN);
  auto multiply = [&](int i) {  // step i, once every warp (of the pair) has stored its share
    wait(full_bar(stage), phase);
    tc_fence_after();
    auto mma = [&](uint32_t d, uint64_t x, uint64_t y, uint32_t acc) {
      if constexpr (PAIR) mma_bf16_pair(d, x, y, idesc, acc);
      else mma_bf16(d, x, y, idesc, acc);
    };
    const int chunks = min(UK, nch - i * UK);
#pragma unroll
    for (int u = 0; u < UK; ++u) {
      if (u >= chunks) break;
      // descriptors of the chunk's parts: the start address is the low field
      const uint64_t at = (uint64_t)(uint32_t)((stage * D::STAGE + u * D::CHUNK) / 16);
      const uint64_t da = make_desc_sw128(base) + at, db = da + D::A2 / 16;
      const uint64_t ta = make_desc_sw64(base + D::A2 + D::B2) + at, tb = ta + D::A3 / 16;
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {  // 16 k: 32 bytes on; lo (mid) 64 bytes after hi
        const uint32_t acc = (i > 0 || u > 0 || kk > 0) ? 1u : 0u;
        mma(tmem, da + 2 * kk, db + 2 * kk, acc);
        mma(tmem + BN, da + 2 * kk, db + 2 * kk + 4, acc);
        mma(tmem + BN, da + 2 * kk + 4, db + 2 * kk, 1u);
        if constexpr (PARTS == 3) {  // hi*lo3 + mid*mid + lo3*hi
          mma(tmem + BN, da + 2 * kk, tb + 2 * kk, 1u);
          mma(tmem + BN, da + 2 * kk + 4, db + 2 * kk + 4, 1u);
          mma(tmem + BN, ta + 2 * kk, db + 2 * kk, 1u);
        }
      }
    }
    if constexpr (PAIR) mma_commit_pair(empty_bar(stage), (uint16_t)(3u << lead));
    else mma_commit(empty_bar(stage));
  };
  for (;;) {
    const bool again = passes > 0;
    bool scaled = false;         // some K-vector split here has an exponent
    // some K-vector split here was zero in the first step (three parts: so far), and
    // this thread's (row tid, or column tid - 128); at the end: throughout
    bool open = PARTS == 3 && !again, mine = open && tid < 128 + BS;
    if (again) {  // exponents from the true maxima of this slice
      __syncthreads();
      if (tid < 128 + BS) rowmax[tid] = 0u;
      __syncthreads();
      for (int i = 0; i < steps; ++i) {
        load_a(va[0], i);
        load_b(vb[0], i);
        OA.row_max(va[0], rowmax);
        OB.row_max(vb[0], rowmax + 128);
      }
      __syncthreads();
      int e = 0;
      if (tid < 128 + BS) e = scale_exp_from_bits(rowmax[tid]);
      mine = tid < 128 + BS && rowmax[tid] == 0u;
      if (tid < 128) exA[tid] = e;
      else if (tid < 128 + BS) exBo[tid - 128] = e;
      scaled = __syncthreads_or(e != 0);
      load_first();
    }
    float top = 0.f;
    auto step = [&](float (&a)[16], float (&b)[BS / 8], int i, bool watch) {
      if (PARTS == 2 && watch) {
        OA.watch_rows(a, late, rowmax);
        OB.watch_rows(b, late + 1, rowmax + 128);
      }
      if (PARTS == 3 && open) {  // exponents of the K-vectors whose first nonzero step this is
        OA.row_max(a, rowmax);
        OB.row_max(b, rowmax + 128);
        __syncthreads();
        int e = 0;
        if (mine && rowmax[tid] != 0u) {
          e = scale_exp_from_bits(rowmax[tid]);
          if (tid < 128) exA[tid] = e;
          else exBo[tid - 128] = e;
          mine = false;
        }
        if (tid < 128 + BS) rowmax[tid] = 0u;
        scaled |= __syncthreads_or(e != 0) != 0;
        open = __syncthreads_or(mine) != 0;
      }
      if (scaled) {
        const bool left_a = OA.scale(a, exA), left_b = OB.scale(b, exBo);
        if (left_a || left_b) top = INFINITY;
      }
      wait(empty_bar(stage), phase ^ 1u);
      uint8_t* const st = ring + stage * D::STAGE + sub * D::CHUNK;
      top = fmaxf(top, OA.template store<PARTS>(a, st, st + D::A2 + D::B2));
      if (i + D::DEPTH < steps) load_a(a, i + D::DEPTH);
      top = fmaxf(top, OB.template store<PARTS>(b, st + D::A2, st + D::A2 + D::B2 + D::A3));
      if (i + D::DEPTH < steps) load_b(b, i + D::DEPTH);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stores, before the MMAs' reads
      __syncwarp();
      if (lane == 0) {
        // The proxy fence has put the stores where the MMA reads them, each
        // CTA's own shared memory through its own async proxy.  Between the
        // odd CTA's warps and the issuer this relies on the hardware: the PTX
        // memory model orders them only by a release and an acquire at cluster
        // scope, and the release waits for every load this thread has in
        // flight (a batch of 64 products 192 x 256 x 4096 108 -> 143 us, with
        // one warp of the odd CTA passing the others' arrivals on 130).
        if (PAIR) mbar_arrive_remote(map_to_rank(full_bar(stage), lead));
        else mbar_arrive(full_bar(stage));
      }
      if (issuer) multiply(i);
      __syncwarp();
      if (++stage == D::STAGES) { stage = 0; phase ^= 1u; }
    };
    if (PARTS == 2 && !again) {  // exponents of the K-vectors that are not zero in the first step
      OA.row_max(va[0], rowmax);
      OB.row_max(vb[0], rowmax + 128);
      __syncthreads();
      int e = 0;
      if (tid < 128 + BS) {
        e = scale_exp_from_bits(rowmax[tid]);
        if (tid < 128) exA[tid] = e;
        else exBo[tid - 128] = e;
        mine = rowmax[tid] == 0u;
      }
      scaled = __syncthreads_or(e != 0) != 0;
      open = __syncthreads_or(mine) != 0;
      if (open) {
        late[0] = OA.zero_rows(rowmax);
        late[1] = OB.zero_rows(rowmax + 128);
        __syncthreads();  // every thread has its bits before the watch writes
      }
    }
    auto pass = [&](bool watch) {
      for (int i = 0; i < steps; i += D::DEPTH) {
#pragma unroll
        for (int d = 0; d < D::DEPTH; ++d)
          if (i + d < steps) step(va[d], vb[d], i + d, watch);
      }
    };
    if (!OWN) pass(open);
    else if (open) pass(true);
    else pass(false);
    if (issuer) {
      if constexpr (PAIR) mma_commit_pair(accf, (uint16_t)(3u << lead));
      else mma_commit(accf);
    }
    __syncwarp();
    bool low = false;  // a K-vector that was zero in the first step is badly scaled after it
    if (PARTS == 2 && open) {
      __syncthreads();  // the watched maxima are complete
      if (mine) {
        low = rowmax[tid] != 0u && rowmax[tid] < kWellScaledLo;
        mine = rowmax[tid] == 0u;
      }
    }
    const bool over = __syncthreads_or(!again && (top >= kWatchLimit || low)) != 0;
    if (tid == 0 && over) *redo_s = 1;
    if (tid == 0 && scaled) *scaled_s = 1;
    if (mine) (tid < 128 ? exA[tid] : exBo[tid - 128]) = kNoExp;
    if (PAIR) {  // the pair shares its columns' exponents; its cluster repeats together
      __syncthreads();
      if ((scaled || again || open) && tid < BS) st_cluster(map_to_rank(smem_u32(exBo + tid), crank ^ 1u), exBo[tid]);
      if (scaled && tid == 0) st_cluster(map_to_rank(smem_u32((const void*)scaled_s), crank ^ 1u), 1);
      if (over && tid < 2 * S.cluster_slices) st_cluster(map_to_rank(smem_u32((const void*)redo_s), (uint32_t)tid), 1);
      cluster_sync_all();
    } else {
      __syncthreads();
    }
    wait(accf, (uint32_t)(passes & 1));  // every MMA of this pass is done (in both CTAs of a pair)
    ++passes;
    if (again || !*redo_s) break;
  }
  tc_fence_after();

  // ---------------- epilogue ----------------
  const bool scaled = *scaled_s != 0;
  constexpr int WC = BN / (D::WARPS / 4);  // columns of a warp
  constexpr int EC = 16;                   // of which read at a time
  const int q = warp & 3, c_begin = (warp >> 2) * WC, c_end = c_begin + WC;
  const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
  const int row = q * 32 + lane;
  const int64_t i = m0 + row;
  if (S.cluster_slices > 1) {
    // Sum the slices' accumulators in slice order: each CTA puts its own in
    // its ring (column-major, 128 rows) and finishes a share of the columns.
    float* const red = reinterpret_cast<float*>(ring);
    for (int c0 = c_begin; c0 < c_end; c0 += EC) {
      float v[EC];
      tmem_sum16<BN>(taddr + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < EC; ++j) red[(c0 + j) * 128 + row] = v[j];
    }
    cluster_sync_all();
    constexpr int G = D::THREADS / 128;  // threads of a row
    const int ns = S.cluster_slices, share = BN / ns, r2 = tid & 127;
    const int64_t i2 = m0 + r2;
    auto rank_of = [&](int s) { return (uint32_t)(PAIR ? 2 * s + (int)prank : s); };
    bool any = false;
    for (int s = 0; s < ns; ++s) any |= ld_cluster_int(map_to_rank(smem_u32((const void*)scaled_s), rank_of(s))) != 0;
    for (int c0 = sl * share + (tid >> 7); c0 < (sl + 1) * share; c0 += 4 * G) {  // four columns at a time
      float v[4] = {0.f, 0.f, 0.f, 0.f}, cv[4];
      bool ok[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ok[u] = i2 < S.m && c0 + G * u < (sl + 1) * share && n0 + c0 + G * u < S.n;
        cv[u] = ok[u] && S.beta != 0.f ? __ldcs(C + i2 + (n0 + c0 + G * u) * S.ldc) : 0.f;
      }
      if (!any) {
        for (int s = 0; s < ns; ++s) {
          const uint32_t from = map_to_rank(smem_u32(red + c0 * 128 + r2), rank_of(s));
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (ok[u]) v[u] += ld_cluster(from + 512u * G * u);
        }
      } else {
        int er = kNoExp;
        for (int s = 0; s < ns; ++s) er = max(er, ld_cluster_int(map_to_rank(smem_u32(exA + r2), rank_of(s))));
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
          const int col = c0 + G * u;
          if (!ok[u]) continue;
          int ec = kNoExp;
          for (int s = 0; s < ns; ++s) ec = max(ec, ld_cluster_int(map_to_rank(smem_u32(exB + col), rank_of(s))));
          float sum = 0.f;
          for (int s = 0; s < ns; ++s) {
            const int e = ld_cluster_int(map_to_rank(smem_u32(exA + r2), rank_of(s))) - er +
                          ld_cluster_int(map_to_rank(smem_u32(exB + col), rank_of(s))) - ec;
            sum += scale_up(ld_cluster(map_to_rank(smem_u32(red + col * 128 + r2), rank_of(s))), e);
          }
          v[u] = scale_up(sum, er + ec);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (ok[u])
          __stcs(C + i2 + (n0 + c0 + G * u) * S.ldc, S.beta != 0.f ? fmaf(S.alpha, v[u], S.beta * cv[u]) : S.alpha * v[u]);
    }
  } else if (S.partial) {
    if (m0 < S.m) {
      const int tm128 = PAIR ? 2 * tm + (int)prank : tm, tiles128 = (int)((S.m + 127) / 128);
      const size_t tile = (size_t)(sl * tiles128 + tm128) * S.tiles_n + tn;
      float* pp = S.partial + tile * 128 * BN + row;
      for (int c0 = c_begin; c0 < c_end; c0 += EC) {
        float v[EC];
        tmem_sum16<BN>(taddr + (uint32_t)c0, v);
#pragma unroll
        for (int j = 0; j < EC; ++j) __stcg(pp + (size_t)(c0 + j) * 128, v[j]);
      }
      int* px = S.partial_exp + tile * kDirectExpInts;
      if (tid == 0) px[0] = scaled;
      if (tid < 128) px[1 + tid] = exA[tid];
      for (int j = tid; j < BN; j += D::THREADS) px[129 + j] = exB[j];
    }
  } else {
    const int ea = scaled ? exA[row] : 0;
    const bool row_ok = i < S.m;
    for (int c0 = c_begin; c0 < c_end; c0 += EC) {
      if (n0 + c0 >= S.n) break;  // warp-uniform
      const int jmax = S.n - (n0 + c0) < EC ? (int)(S.n - (n0 + c0)) : EC;
      float* cp = C + i + (n0 + c0) * S.ldc;
      float cv[EC];
      if (S.beta != 0.f) {
#pragma unroll
        for (int j = 0; j < EC; ++j) cv[j] = (row_ok && j < jmax) ? __ldcs(cp + j * S.ldc) : 0.f;
      }
      float v[EC];
      tmem_sum16<BN>(taddr + (uint32_t)c0, v);
      if (scaled) {
#pragma unroll
        for (int j = 0; j < EC; ++j) v[j] = scale_up(v[j], ea + exB[c0 + j]);
      }
#pragma unroll
      for (int j = 0; j < EC; ++j) {
        const float out = S.beta != 0.f ? fmaf(S.alpha, v[j], S.beta * cv[j]) : S.alpha * v[j];
        if (row_ok && j < jmax) __stcs(cp + j * S.ldc, out);
      }
    }
  }
  tc_fence_before();
  // no CTA leaves while another of its cluster may still read its shared memory
  if (clustered) cluster_sync_all();
  else __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(D::TMEM) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(D::TMEM) : "memory");
  }
}

// The launch of an instance with clusters of `cluster` CTAs: its attributes
// are set (once per device), cfg and attr filled in (attr outlives cfg's use).
template <int BN, bool PAIR, int PARTS, int MA, int MB>
cudaError_t prepare_direct_launch(int dev, int cluster, int64_t ctas, cudaLaunchConfig_t* cfg,
                                  cudaLaunchAttribute (&attr)[2]) {
  using D = DirectShape<BN, PAIR, PARTS>;
  static std::atomic<bool> attr_set[64] = {};
  auto* fn = direct_gemm_kernel<BN, PAIR, PARTS, MA, MB>;
  if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_relaxed)) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, D::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_relaxed);
  }
  cfg->gridDim = dim3((unsigned)ctas);
  cfg->blockDim = dim3(D::THREADS);
  cfg->dynamicSmemBytes = D::SMEM;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = cluster > 1 ? 2 : 1;
  return cudaSuccess;
}

template <int BN, bool PAIR, int PARTS, int MA, int MB>
cudaError_t launch_direct_kernel(const DirectArgs& S, int64_t items, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  const int per = PAIR ? 2 : 1;
  e = prepare_direct_launch<BN, PAIR, PARTS, MA, MB>(dev, S.cluster_slices * per, items * per, &cfg, attr);
  if (e != cudaSuccess) return e;
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, direct_gemm_kernel<BN, PAIR, PARTS, MA, MB>, S);
}

// Whether the device can hold a cluster of `cluster` (1, 2, 4, 8, 16) CTAs of
// an instance, asked once per device.
template <int BN, bool PAIR, int PARTS, int MA, int MB>
bool direct_kernel_fits(int cluster) {
  static std::atomic<signed char> known[64][5] = {};  // 1: fits, -1: does not
  int dev = 0, bit = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  while (1 << bit < cluster) ++bit;
  const bool keep = dev >= 0 && dev < 64 && bit < 5;
  if (keep)
    if (const signed char k = known[dev][bit].load(std::memory_order_relaxed)) return k > 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  cudaError_t e = prepare_direct_launch<BN, PAIR, PARTS, MA, MB>(dev, cluster, cluster, &cfg, attr);
  int n = 1;
  if (e == cudaSuccess && cluster > 1) {
    cfg.attrs = attr + 1;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&n, direct_gemm_kernel<BN, PAIR, PARTS, MA, MB>, &cfg);
  }
  if (e != cudaSuccess) (void)cudaGetLastError();  // no answer: not used this time, and not an error
  const bool fits = e == cudaSuccess && n > 0;
  if (keep && e == cudaSuccess) known[dev][bit].store(fits ? 1 : -1, std::memory_order_relaxed);
  return fits;
}

}  // namespace

// One of the six (parts, mode of op(A)) families of instances, a translation
// unit each.
#define GBG_DIRECT_CALL(FN, BN, PAIR, ...)                        \
  (mb == kRows  ? FN<BN, PAIR, PARTS, MA, kRows>(__VA_ARGS__)      \
   : mb == kVec ? FN<BN, PAIR, PARTS, MA, kVec>(__VA_ARGS__)       \
                : FN<BN, PAIR, PARTS, MA, kScalar>(__VA_ARGS__))
template <int PARTS, int MA>
cudaError_t launch_direct_mode(const DirectPlan& plan, int mb, const DirectArgs& S, int64_t items, cudaStream_t s) {
  if (plan.bn == 64 && !plan.pair) return GBG_DIRECT_CALL(launch_direct_kernel, 64, false, S, items, s);
  if (plan.bn == 128 && plan.pair) return GBG_DIRECT_CALL(launch_direct_kernel, 128, true, S, items, s);
  if constexpr (PARTS == 2)
    if (plan.bn == 256 && plan.pair) return GBG_DIRECT_CALL(launch_direct_kernel, 256, true, S, items, s);
  return cudaErrorInvalidValue;
}

template <int PARTS, int MA>
bool direct_mode_fits(const DirectPlan& plan, int mb) {
  const int cluster = direct_cluster_ctas(plan);
  if (plan.bn == 64 && !plan.pair) return GBG_DIRECT_CALL(direct_kernel_fits, 64, false, cluster);
  if (plan.bn == 128 && plan.pair) return GBG_DIRECT_CALL(direct_kernel_fits, 128, true, cluster);
  if constexpr (PARTS == 2)
    if (plan.bn == 256 && plan.pair) return GBG_DIRECT_CALL(direct_kernel_fits, 256, true, cluster);
  return false;
}
#undef GBG_DIRECT_CALL

}  // namespace gbg
