// Split-BF16 tensor-core sgemm for sm_103a: the scaling/packing kernels and
// the persistent tcgen05 GEMM.
//
// Method.  Every K-vector of the problem -- a row of op(A) or a column of
// op(B) -- is scaled by 2^-e, e being the frexp exponent of its largest
// magnitude, so its entries lie in (-1, 1).  Each scaled entry x' becomes
// hi = bf16_rn(x') and lo = bf16_rn(x' - hi) (x' - hi is exact in FP32).  The
// tensor cores accumulate hi_a*hi_b + hi_a*lo_b + lo_a*hi_b in FP32 and the
// epilogue multiplies by 2^(e_i + f_j), then applies alpha and beta once.
//
// Structure (after the paper's BLIS sgemm, Sections III-A and III-C):
//  * packing -- the BLIS packing of A and B panels becomes a pass that writes
//    hi/lo BF16 panels in exactly the byte order the tensor cores read from
//    shared memory (128-byte rows, 16-byte chunks XOR-swizzled by row mod 8);
//  * the micro-kernel's k loop -- the paper sends KSUB-deep blocks of a1 and
//    b1 into two alternating buffers with a `selector` while the coprocessor
//    works on the other (Section III-C).  Here a producer thread streams
//    32-deep blocks with bulk asynchronous copies into a ring of shared
//    memory stages guarded by full/empty mbarriers;
//  * the Accumulator -- the paper's `command` 0/1/2/3 protocol (clear on the
//    first block, accumulate, send the result on the last) becomes the
//    tcgen05.mma accumulate flag (off for the first MMA of a tile) and a
//    commit to an "accumulator full" barrier after the last block.  The
//    accumulator lives in tensor memory (TMEM), two buffers of 128 x BN FP32
//    so that the epilogue of one tile overlaps the main loop of the next;
//  * output ownership -- each CTA owns whole 128 x BN tiles of column-major
//    C, and the epilogue writes each column's 128 rows with one coalesced
//    warp store per 32 rows (Section III-D assigns each core whole column
//    blocks of the result for the same reason).
#include <algorithm>

#include "gemm_kernel.cuh"

namespace gbg {
namespace {

// The sum of the slices' accumulators of four rows and one column when some
// slice's tile has exponents: every slice's are first brought to the largest
// exponent of the row and of the column (a slice where either is zero
// throughout has kNoExp there and adds nothing).
__device__ __forceinline__ float4 rescaled_sum(const float4* p, size_t slice_elems, int splitk, const int* pexp,
                                               size_t pstride, int row, int col) {
  float out[4];
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    int er = kNoExp, ec = kNoExp;
#pragma unroll 1
    for (int s = 0; s < splitk; ++s) {
      er = max(er, pexp[s * pstride + 1 + row + q]);
      ec = max(ec, pexp[s * pstride + 129 + col]);
    }
    float sum = 0.f;
#pragma unroll 1
    for (int s = 0; s < splitk; ++s) {
      const float acc = reinterpret_cast<const float*>(p + s * (slice_elems / 4))[q];
      sum += scale_up(acc, pexp[s * pstride + 1 + row + q] - er + pexp[s * pstride + 129 + col] - ec);
    }
    out[q] = scale_up(sum, er + ec);
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}
__device__ __forceinline__ void rescale_slices(float4& acc, const float4* p, size_t slice_elems, int splitk,
                                               const int* pexp, size_t pstride, int row, int col) {
  int any = 0;
  for (int s = 0; s < splitk; ++s) any |= pexp[s * pstride];
  if (any) acc = rescaled_sum(p, slice_elems, splitk, pexp, pstride, row, col);
}

// Split-K reduction: a thread per four consecutive rows i .. i+3 of one
// column j of C (rows of a 128-row tile, so the partials are 16-byte
// vectors), the slices' raw accumulators summed in slice order
// (deterministic), then the epilogue of split_gemm_kernel: x 2^(e_i + f_j),
// alpha, and beta C with one rounding of beta C and one fused multiply-add.
// EXP: the slices have exponents of their own (pexp, direct.cu) instead of the
// operands' maxima.  Every load of a thread is independent, so one pass over
// the grid keeps them all in flight: the kernel is as fast as its blocks are
// many on an SM (1024^2 outputs of 4 slices, cold: 8.3 us; 13.2 with 128
// registers).  U slices' loads are in flight: eight, or sixteen where a small
// output gives no SM more than two blocks (300 x 300 x 5000, 31 slices: a call
// 33.2 -> 32.1 us).
template <bool EXP, int U>
__global__ void __launch_bounds__(256, U == 8 ? 4 : 2)
    splitk_reduce_kernel(int64_t m, int64_t n, int bn, int tiles_m, int tiles_n, int splitk,
                         const float* __restrict__ partial, const uint32_t* __restrict__ amaxA,
                         const uint32_t* __restrict__ amaxB, const int* __restrict__ pexp, float alpha, float beta,
                         float* __restrict__ C, int64_t ldc) {
  wait_prerequisite_grid();  // launched as a dependent of the GEMM
  const int64_t mq = (m + 3) / 4, total = mq * n;
  const size_t tile_elems = (size_t)128 * bn, slice_elems = (size_t)tiles_m * tiles_n * tile_elems;
  const bool c_vec = ((ldc & 3) == 0) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = (t % mq) * 4, j = t / mq;
    const int64_t tm = i0 >> 7, tn = j / bn;
    const float4* p = reinterpret_cast<const float4*>(
        partial + (size_t)(tm * tiles_n + tn) * tile_elems + (size_t)(j - tn * bn) * 128 + (i0 & 127));
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < splitk; s0 += U) {
      // U slices' loads in flight, then summed in slice order
      float4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (s0 + u < splitk) v[u] = __ldcs(p + (size_t)(s0 + u) * (slice_elems / 4));
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (s0 + u < splitk) { acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w; }
    }
    if (EXP) rescale_slices(acc, p, slice_elems, splitk, pexp + (tm * tiles_n + tn) * kDirectExpInts,
                            (size_t)tiles_m * tiles_n * kDirectExpInts, (int)(i0 & 127), (int)(j - tn * bn));
    const int fj = EXP ? 0 : scale_exp_from_bits(amaxB[j]);
    float* c = C + i0 + j * ldc;
    const float a4[4] = {acc.x, acc.y, acc.z, acc.w};
    float o[4];
    if (c_vec && i0 + 3 < m) {
      const float4 cv = beta != 0.f ? *reinterpret_cast<const float4*>(c) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float c4[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = EXP ? 0 : scale_exp_from_bits(amaxA[i0 + q]) + fj;
        const float v = (e >= -126 && e <= 127) ? a4[q] * __int_as_float((e + 127) << 23) : scalbnf(a4[q], e);
        o[q] = (beta != 0.f) ? fmaf(alpha, v, beta * c4[q]) : alpha * v;
      }
      *reinterpret_cast<float4*>(c) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (i0 + q >= m) break;
        const int e = EXP ? 0 : scale_exp_from_bits(amaxA[i0 + q]) + fj;
        const float v = (e >= -126 && e <= 127) ? a4[q] * __int_as_float((e + 127) << 23) : scalbnf(a4[q], e);
        c[q] = (beta != 0.f) ? fmaf(alpha, v, beta * c[q]) : alpha * v;
      }
    }
  }
}

// Failure-detection probe: one thread waits on an mbarrier that nothing
// arrives on and no copy is bound to, with the library's bounded wait; when
// the limit runs out it records GBGEMM_ERR_DEVICE_TIMEOUT in *status, as
// every kernel's waits do, and the CTA returns normally.
__global__ void __launch_bounds__(32) wait_probe_kernel(int* status, uint64_t timeout_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (threadIdx.x == 0 && !mbar_wait(smem_u32(&bar), 0u, &abort_flag, timeout_ns))
    raise_status(status, &abort_flag);
  __syncwarp();
}

}  // namespace

cudaError_t launch_wait_probe(int* status, uint64_t timeout_ns, cudaStream_t s) {
  wait_probe_kernel<<<1, 32, 0, s>>>(status, timeout_ns);
  return cudaGetLastError();
}

int choose_splitk(int64_t tiles, int64_t k, int num_sms) {
  if (split_parts(k) != 1 || tiles <= 0 || tiles * 2 > num_sms) return 1;
  int64_t s = num_sms / tiles;                    // about one item per SM
  const int64_t max_by_k = panel_k_chunks(k) / 4; // at least 4 k chunks (128 deep) per slice
  if (s > max_by_k) s = max_by_k;
  if (s > 32) s = 32;
  if (s < 2) return 1;
  // every slice gets at least one chunk: ceil(nkc / ceil(nkc / s)) slices
  const int64_t nkc = panel_k_chunks(k), per = (nkc + s - 1) / s;
  s = (nkc + per - 1) / per;
  return s >= 2 ? (int)s : 1;
}

SplitLayout split_layout(int64_t m, int64_t n, int64_t k, int64_t batch, int splitk, int bn) {
  SplitLayout L{};
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const int64_t ra = (m + 127) / 128, rb = (n + 127) / 128;
  L.bands = (size_t)(ra + rb) * (size_t)batch;
  L.band_off = kSplitCtlBytes;
  L.amax_off = L.band_off + up(L.bands * 4);
  L.amax_stride = m + n;
  L.head = L.amax_off + up((size_t)batch * (size_t)(m + n) * 4);
  L.pa = up(panel_bytes(m, k));
  L.pb = up(panel_bytes(n, k));
  L.block = (size_t)split_parts(k) * (L.pa + L.pb);
  L.panel_off = L.head;
  L.partial_off = L.panel_off + L.block * (size_t)batch;
  const size_t tiles = (size_t)((m + 127) / 128) * (size_t)((n + bn - 1) / bn);
  L.total = L.partial_off + (splitk > 1 ? (size_t)splitk * tiles * 128 * (size_t)bn * 4 : 0);
  return L;
}

namespace {

// The scheduler of one call (or strided batch) over the workspace `ws`.
// pack_only: no tiles, only the packing of op(A)'s rows (panel inspection).
SingleSched make_single_sched(const SplitCall& c, const SplitLayout& L) {
  uint8_t* ws = static_cast<uint8_t*>(c.ws);
  SingleSched S;
  S.ctl = reinterpret_cast<WorkCtl*>(ws);
  S.band_cnt = reinterpret_cast<int*>(ws + L.band_off);
  S.A = c.A; S.B = c.B; S.lda = c.lda; S.ldb = c.ldb; S.sa = c.sa; S.sb = c.sb;
  S.ta = c.ta; S.tb = c.tb;
  S.panelA = ws + L.panel_off;
  S.panelB = ws + L.panel_off + L.pa;
  S.amaxA = reinterpret_cast<uint32_t*>(ws + L.amax_off);
  S.amaxB = S.amaxA + c.m;
  S.m = c.m; S.n = c.n; S.k = c.k;
  S.alpha = c.alpha; S.beta = c.beta;
  S.C = c.C; S.ldc = c.ldc;
  S.tiles_m = (int)((c.m + 127) / 128);
  S.tiles_n = (int)((c.n + c.bn - 1) / c.bn);
  S.nkc = (int)panel_k_chunks(c.k);
  S.raster = c.raster > 0 ? c.raster : 16;
  S.bn = c.bn;
  S.parts = split_parts(c.k);
  S.rbA = panel_row_blocks(c.m);
  S.rbB = panel_row_blocks(c.n);
  S.ra = (int)((c.m + 127) / 128);
  S.rb = (int)((c.n + 127) / 128);
  // Chunks per packing task: kPackChunks, halved (down to 1) while the
  // tasks would not give every SM three of them, so that small operands are
  // packed in one round of loads.
  const int64_t sms = c.num_sms > 0 ? c.num_sms : 148;
  S.pchunks = kPackChunks;
  while (S.pchunks > 1 && c.batch * (S.ra + S.rb) * ((S.nkc + S.pchunks - 1) / S.pchunks) < 3 * sms) S.pchunks >>= 1;
  S.ngroups = (S.nkc + S.pchunks - 1) / S.pchunks;
  // per problem [A | B | A2 | B2]: A2 - A = B2 - B = pa + pb
  S.a_part = S.parts == 2 ? (int64_t)(L.pa + L.pb) : 0;
  S.b_part = S.a_part;
  S.batch = (int)c.batch;
  S.ps = (int64_t)L.block;
  S.as = L.amax_stride;
  S.cs = c.sc;
  S.splitk = c.splitk > 1 ? c.splitk : 1;
  S.slice_chunks = (S.nkc + S.splitk - 1) / S.splitk;
  S.partial = c.splitk > 1 ? reinterpret_cast<float*>(ws + L.partial_off) : nullptr;
  S.pair = 0;
  S.tail_start = 0;
  return S;
}

}  // namespace

// Estimated time of a tile of `w` columns: the MMAs of its k chunks (0.5 us a
// chunk of 256 columns, twice that with three parts), or below about 205
// columns the copies that feed them (a chunk's op(A) block is as large for
// every width), and the fill and the way out.
static double pair_tile_us(int w, int64_t chunks, bool three) {
  const double wide = std::max((double)w, (16384.0 + 64.0 * w) / 144.0) / 256.0;
  return (double)chunks * (three ? 1.0 : 0.5) * wide + 1.0 + 3.0 * w / 256.0;
}

// With 256 columns throughout, the last round of tiles is often nearly empty
// (4096^2: 256 tiles on 76 pairs, 3.37 rounds; 1931 x 1207: 40 tiles) while a
// narrower tile, or halves of the last ones, fills it.  Measured against 256
// throughout: 1931 x 1207 x 877 35.6 -> 34.0 us (160 columns, 64 tiles),
// 4096^3 298.7 -> 293.4 us (224 columns, exactly four rounds), 8192^3 the same
// within 0.1% (halves for the last 36 tiles; bound by power).
PairTiles choose_pair_tiles(int64_t m, int64_t n, int64_t batch, int64_t chunks, bool three, int pairs) {
  PairTiles best;
  const int64_t rows = (m + 255) / 256 * batch;
  for (int w = 256; w >= 64; w -= 32) {
    const int64_t tiles = rows * ((n + w - 1) / w), tail = tiles % pairs;
    const double whole = (double)(tiles - tail) / pairs * pair_tile_us(w, chunks, three);
    auto offer = [&](int64_t tail_start, double us) {
      if (best.tiles != 0 && us >= 0.99 * best.us) return;
      best.bn = w; best.tiles = tiles; best.tail_start = tail_start; best.us = us;
    };
    offer(tiles, whole + (tail ? pair_tile_us(w, chunks, three) : 0.0));
    if (tail && w % 64 == 0)
      offer(tiles - tail, whole + (double)((2 * tail + pairs - 1) / pairs) * pair_tile_us(w / 2, chunks, three));
  }
  return best;
}

extern "C" void gbgemm_internal_pair_tiles(int64_t m, int64_t n, int64_t batch, int64_t chunks, int three, int pairs,
                                           int64_t* tiles) {
  const PairTiles t = choose_pair_tiles(m, n, batch, chunks, three != 0, pairs);
  tiles[0] = t.bn; tiles[1] = t.tiles; tiles[2] = t.tail_start;
}

namespace {

// The head of the workspace (control words, band counters, row maxima) set to
// zero.  A kernel and not a memset, so that the packing can be launched ahead
// of its end: a packing task needs the zeros only once it has its maxima.
// 1931 x 1207 x 877 33.9 -> 31.3 us, 8192^2 x 128 120.6 -> 118.3 us.
__global__ void __launch_bounds__(256) clear_head_kernel(uint4* __restrict__ p, int64_t n16) {
  launch_dependents();
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n16; i += (int64_t)gridDim.x * 256)
    p[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

cudaError_t launch_split_call(const SplitCall& c, cudaStream_t s) {
  if (c.m <= 0 || c.k <= 0 || c.batch <= 0) return cudaSuccess;
  if (c.n < 0 || (c.n == 0 && !c.pack_only)) return cudaSuccess;
  if (c.bn != 64 && c.bn != 128 && c.bn != 256) return cudaErrorInvalidValue;
  if (c.batch > 65535 || !c.ws) return cudaErrorInvalidValue;
  const int splitk = c.splitk > 1 ? c.splitk : 1;
  if (splitk > 1 && (c.batch != 1 || split_parts(c.k) != 1)) return cudaErrorInvalidValue;
  const int64_t tm = (c.m + 127) / 128, tn = (c.n + c.bn - 1) / c.bn;
  const int64_t nkc = panel_k_chunks(c.k);
  const int64_t tasks = c.batch * (tm + (c.n + 127) / 128) * ((nkc + kPackChunks - 1) / kPackChunks);
  if (tm * tn * c.batch * splitk > (int64_t)0x7FFFFFFF || tasks > (int64_t)0x7FFFFFFF) return cudaErrorInvalidValue;
  const SplitLayout L = split_layout(c.m, c.n, c.k, c.batch, splitk, c.bn);
  SingleSched S = make_single_sched(c, L);
  // fewer chunks per task only below 3 tasks per SM: still far below 2^31
  const int64_t ptasks = c.batch * (int64_t)(S.ra + S.rb) * S.ngroups;
  if (c.pack_only) {
    S.tiles_n = 0;  // no tiles: the packers only
    if (c.panel_out) {
      S.panelA = static_cast<const uint8_t*>(c.panel_out);
      S.a_part = c.panel2_out ? static_cast<const uint8_t*>(c.panel2_out) - S.panelA : 0;
    }
    if (c.amax_out) S.amaxA = c.amax_out;
  }
  // no empty slice (an empty slice would store a stale accumulator)
  if ((int64_t)(S.splitk - 1) * S.slice_chunks >= S.nkc) return cudaErrorInvalidValue;
  const int64_t head16 = (int64_t)(L.head / 16);
  const bool ahead = !c.pack_only && ptasks > 0 && L.head % 16 == 0;
  cudaError_t e = cudaSuccess;
  if (ahead) {
    clear_head_kernel<<<(unsigned)std::min<int64_t>((head16 + 255) / 256, 64), 256, 0, s>>>(
        static_cast<uint4*>(c.ws), head16);
    e = cudaGetLastError();
  } else {
    e = cudaMemsetAsync(c.ws, 0, L.head, s);
  }
  if (e != cudaSuccess) return e;
  if (c.pack_only && c.amax_out) {
    e = cudaMemsetAsync(c.amax_out, 0, (size_t)c.m * 4, s);
    if (e != cudaSuccess) return e;
  }
  const int64_t items = tm * tn * c.batch * splitk;
  const int64_t sms = c.num_sms > 0 ? c.num_sms : 148;
  // packing tasks first, each its own CTA, then the GEMM
  if (ptasks > 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ptasks);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ahead ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, pack_tasks_kernel<SingleSched>, S);
  }
  if (e != cudaSuccess || items == 0) return e;
  const int grid = (int)(items < sms ? items : sms);
  const bool timed = c.gemm_begin && c.gemm_end;
  // Pair tiles (clusters of two CTAs, tiles of 256 rows) for the widest tiles
  // of calls with at least two tile rows; with three-part panels (k < 512)
  // only from 8 k chunks: below that a tile's MMAs take less time than its
  // epilogue, and pairing two CTAs' epilogues (and the fixed tile order) cost
  // more than the halved operand loads gain (k = 128: 21% slower at 16384^2).
  const bool pair_ok = !c.pack_only && c.bn == 256 && tm >= 2 && (S.parts == 1 || S.nkc >= 8);
  const int pair_cap = !pair_ok ? 0
                       : S.parts == 2 ? gemm_pair_capacity<SingleSched, true>() : gemm_pair_capacity<SingleSched>();
  if (timed && (e = cudaEventRecord(c.gemm_begin, s)) != cudaSuccess) return e;
  if (pair_cap > 0) {
    S.pair = 1;
    int64_t pair_items = (tm + 1) / 2 * tn * c.batch * splitk;
    S.tail_start = (int)pair_items;
    if (splitk == 1) {
      const PairTiles T = choose_pair_tiles(c.m, c.n, c.batch, nkc, S.parts == 2, pair_cap);
      // what job_pair and the epilogue's column split rest on
      const int narrow = T.tail_start < T.tiles ? T.bn / 2 : T.bn;
      if (T.bn < 64 || T.bn > kMaxBN || narrow % 32 != 0) return cudaErrorInvalidValue;
      if (2 * T.tiles <= (int64_t)0x7FFFFFFF) {
        S.bn = T.bn;
        S.tiles_n = (int)((c.n + T.bn - 1) / T.bn);
        S.tail_start = (int)T.tail_start;
        pair_items = 2 * T.tiles - T.tail_start;
      }
    }
    const int pairs = (int)(pair_items < pair_cap ? pair_items : pair_cap);
    e = S.parts == 2 ? launch_gemm_kernel_pair<SingleSched, true>(S, pairs, c.status, s, ptasks > 0 && !timed)
                     : launch_gemm_kernel_pair<SingleSched>(S, pairs, c.status, s, ptasks > 0 && !timed);
  } else {
    e = launch_gemm_kernel<SingleSched>(S, grid, c.status, s, ptasks > 0 && !timed);
  }
  if (e != cudaSuccess) return e;
  if (timed && (e = cudaEventRecord(c.gemm_end, s)) != cudaSuccess) return e;
  e = cudaGetLastError();
  if (e != cudaSuccess || splitk == 1 || c.pack_only) return e;
  SplitGemmArgs a;
  a.m = c.m; a.n = c.n; a.k = c.k; a.alpha = c.alpha; a.beta = c.beta; a.C = c.C; a.ldc = c.ldc;
  a.amaxA = S.amaxA; a.amaxB = S.amaxB; a.num_sms = c.num_sms; a.bn = c.bn; a.splitk = splitk;
  a.partial = S.partial;
  return launch_splitk_reduce(a, s);
}

cudaError_t launch_splitk_reduce(const SplitGemmArgs& a, cudaStream_t s) {
  if (a.m <= 0 || a.n <= 0 || a.splitk <= 1) return cudaSuccess;
  const int tm = (int)((a.m + 127) / 128), tn = (int)((a.n + a.bn - 1) / a.bn);
  const int64_t total = (a.m + 3) / 4 * a.n;  // a thread per four rows of a column
  int64_t blocks = (total + 255) / 256;
  const int64_t sms = a.num_sms > 0 ? a.num_sms : 148, cap = sms * 16;
  if (blocks > cap) blocks = cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool deep = a.splitk > 8 && blocks <= 2 * sms;
  auto* kernel = a.partial_exp ? (deep ? splitk_reduce_kernel<true, 16> : splitk_reduce_kernel<true, 8>)
                               : (deep ? splitk_reduce_kernel<false, 16> : splitk_reduce_kernel<false, 8>);
  return cudaLaunchKernelEx(&cfg, kernel, a.m, a.n, a.bn, tm, tn, a.splitk, (const float*)a.partial,
                            a.amaxA, a.amaxB, a.partial_exp, a.alpha, a.beta, a.C, a.ldc);
}

}  // namespace gbg
